// The record scan of a partitioned many-group aggregation (records.cu),
// specialised on a plan shape JS (fields: jit_common.cuh) and compiled at run
// time.
//
// A thread takes four consecutive rows, loads every column of them at once
// with vector loads, and its warp appends their records.  Rows in flight hide
// the chain of column load, table probe and cursor atomic, so what counts is
// registers: the ahead-of-time scan, which reads the column types as it goes,
// spilled at 64 of them and took 744 us for 60M rows of the orders query where
// this one took 566 (at one list per partition).  Each lane also prefetches a line of the warp's next
// rows into L2.
#pragma once
#include "jit_common.cuh"
#include "records.cuh"

namespace tpj {

static_assert(ST_RPL == REC_RPT, "the probes take a thread's rows");

// TPJ_SELECTED: the rows are four entries of a selection vector, whose filter
// has been evaluated, and their columns are gathered: 600k of 60M rows in 56 us
// (66 with column types read as it goes), bound by 2.4M scattered sectors.
#ifdef TPJ_SELECTED
constexpr bool SELECTED = true;
#else
constexpr bool SELECTED = false;
#endif

// A thread's rows: r .. r + 3, those below n; selected: row[i], all loadable.
struct Rows {
    uint64_t r, n;
    uint32_t row[4];
};

template <int T>
struct Quad {
    typename ColT<T>::type v[4];
    __device__ __forceinline__ void load(const DevCol& c, const Rows& rows) {
        typedef typename ColT<T>::type E;
        if constexpr (SELECTED) {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = __ldcs((const E*)c.ptr + rows.row[i]);
            return;
        }
        const uint64_t r = rows.r, n = rows.n;
        const E* p = (const E*)c.ptr + r;
        if (r + 4 <= n) {
            if constexpr (T == T_I32) {
                const int4 a = __ldcs((const int4*)p);
                v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
            } else if constexpr (T == T_I64) {
                const longlong2 a = __ldcs((const longlong2*)p), b = __ldcs((const longlong2*)p + 1);
                v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
            } else {
                const uchar4 a = __ldcs((const uchar4*)p);
                v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = r + i < n ? p[i] : (E)0;
        }
    }
    // this lane's line of the 128 rows from r on
    __device__ static __forceinline__ void prefetch(const DevCol& c, uint64_t r, uint64_t n, uint32_t lane) {
        constexpr uint32_t lines = 128 * sizeof(typename ColT<T>::type) / 128;
        if (r + 128 <= n && lane < lines)
            asm volatile("prefetch.global.L2 [%0];" ::"l"((const typename ColT<T>::type*)c.ptr + r +
                                                         lane * (128 / sizeof(typename ColT<T>::type))));
    }
};

template <class S, int F>
__device__ __forceinline__ void key_fields(const QueryDev& q, const Rows& rows, uint64_t key[4], uint32_t& bad) {
    if constexpr (F < S::ng) {
        constexpr int bits = S::gbits[F];
        Quad<S::gtype[F]> v;
        v.load(q.gcol[F], rows);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint64_t f = (uint64_t)(int64_t)v.v[i];
            if constexpr (bits < 64) {
                bad |= (uint32_t)((f >> bits) != 0) << i;
                key[i] = (key[i] << bits) | f;
            } else {
                key[i] = f;
            }
        }
        key_fields<S, F + 1>(q, rows, key, bad);
    }
}

template <class S, int I>
__device__ __forceinline__ void terms(const QueryDev& q, const Rows& rows, int64_t (&t)[S::ns > 0 ? S::ns : 1][4]) {
    if constexpr (I < S::ns) {
        Quad<S::atype[I]> a;
        a.load(q.sa[I], rows);
        if constexpr (S::skind[I] == S_MUL_SUB) {
            Quad<S::btype[I]> b;
            b.load(q.sb[I], rows);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                t[I][i] = (int64_t)((uint64_t)(int64_t)a.v[i] * ((uint64_t)q.sk[I] - (uint64_t)(int64_t)b.v[i]));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) t[I][i] = (int64_t)a.v[i];
        }
        terms<S, I + 1>(q, rows, t);
    }
}

template <class S, int F, int I>
__device__ __forceinline__ void prefetch_rest(const QueryDev& q, uint64_t r, uint64_t n, uint32_t lane) {
    if constexpr (F < S::ng) {
        Quad<S::gtype[F]>::prefetch(q.gcol[F], r, n, lane);
        prefetch_rest<S, F + 1, I>(q, r, n, lane);
    } else if constexpr (I < S::ns) {
        Quad<S::atype[I]>::prefetch(q.sa[I], r, n, lane);
        if constexpr (S::skind[I] == S_MUL_SUB) Quad<S::btype[I]>::prefetch(q.sb[I], r, n, lane);
        prefetch_rest<S, F, I + 1>(q, r, n, lane);
    }
}

}  // namespace tpj

extern "C" __global__ void __launch_bounds__(tpk::REC_THREADS, JS::ns > 2 ? 3 : 5)
    tpj_records(const __grid_constant__ tpk::QueryDev q, uint64_t n, const uint32_t* __restrict__ sel,
                const unsigned long long* count, const __grid_constant__ tpk::RecDev rec) {
    using namespace tpk;
    using namespace tpj;
    const Flt flt = make_flt(q);
    const uint32_t lane = threadIdx.x & 31u;
    if constexpr (SELECTED) n = *count;
    // a warp's rows: 128 in a row, then on by the grid's
    const uint64_t step = (uint64_t)gridDim.x * REC_TILE;
    for (uint64_t w0 = (uint64_t)blockIdx.x * REC_TILE + (threadIdx.x >> 5) * 128; w0 < n; w0 += step) {
        const uint64_t r = w0 + 4 * lane;
        Rows rows;
        rows.r = r;
        rows.n = n;
        if constexpr (SELECTED) {   // past the end: the first entry's row, left out below
#pragma unroll
            for (int i = 0; i < 4; ++i) rows.row[i] = __ldcs(sel + (r + i < n ? r + i : 0));
        }
        bool pass[4];
        uint64_t key[4] = {0, 0, 0, 0};
        uint32_t bad = 0;
        int64_t t[JS::ns > 0 ? JS::ns : 1][4] = {};
        Quad<JS::filter ? JS::ftype : T_U8> f;
        Quad<JS::join != J_NONE ? JS::ktype : T_U8> k;
        if constexpr (JS::filter && !SELECTED) f.load(q.fcol, rows);
        if constexpr (JS::join != J_NONE) k.load(q.fk, rows);
        key_fields<JS, 0>(q, rows, key, bad);
        terms<JS, 0>(q, rows, t);
        if constexpr (!SELECTED) {
            if constexpr (JS::filter) Quad<JS::ftype>::prefetch(q.fcol, w0 + step, n, lane);
            if constexpr (JS::join != J_NONE) Quad<JS::ktype>::prefetch(q.fk, w0 + step, n, lane);
            prefetch_rest<JS, 0, 0>(q, w0 + step, n, lane);
        }
        uint32_t pm = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            bool in = r + i < n;
            if constexpr (JS::filter && !SELECTED) {
                if constexpr (JS::ftype == T_I64) in = in && f.v[i] >= flt.lo && f.v[i] <= flt.hi;
                else in = in && (int32_t)f.v[i] >= flt.lo32 && (int32_t)f.v[i] <= flt.hi32;
            }
            pm |= (uint32_t)in << i;
        }
        if constexpr (JS::join != J_NONE) {
            uint32_t pay[4];
            int64_t fk[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) fk[i] = (int64_t)k.v[i];
            if constexpr (JS::lip) lip_mask<4>(q.jt, fk, pm);
            if constexpr (JS::join == J_DIRECT) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint64_t idx = (uint64_t)(fk[i] - q.jt.kmin);
                    pay[i] = (pm >> i & 1u) && idx < q.jt.range ? __ldg((const unsigned int*)q.jt.slots + idx) : EMPTY32;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (pay[i] == EMPTY32) pm &= ~(1u << i);
            } else if constexpr (JS::join == J_PACKED64) {
                probe_rows_packed(q.jt, fk, pm, pay);
            } else if constexpr (JS::join == J_HASH32) {
                probe_rows_k32(q.jt, fk, pm, pay, q.err);
            } else {
                probe_rows_k64(q.jt, fk, pm, pay, q.err);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) bad |= (uint32_t)((pay[i] & PAYLOAD_BAD) != 0) << i;
        }
        if (bad & pm) {
            atomicOr(q.err, ERR_RANGE);
            pm &= ~bad;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) pass[i] = pm >> i & 1u;
        fold_append<(JS::ns > 0 ? JS::ns : 1)>(q, rec, pass, key, t);
    }
}
