// Many-group aggregation through partitioned records.
//
// Paper basis: Section 3.1 (operators run GPU kernels over batches of
// equal-length columns), Section 3.2 (join), Section 4 (exact decimal sums).
// The split is this library's design.  Updating a table of millions of groups
// in place costs a random read-modify-write of device memory per row; here
//
//  * the scan (k_rec_scan, or k_rec_selected over a selection vector) filters,
//    joins and keys the rows, folds a thread's consecutive rows of one key into
//    one record {key within its partition, count, sums}, and appends the
//    records to key-range partitions: the lanes of a warp whose records go to
//    one partition reserve their places with one atomic (sorted keys would
//    queue on one cursor otherwise), and a partition's tail stays in L2 until
//    its sectors are full.  Counting a CTA's tile per partition in shared
//    memory first, to reserve once per tile, was slower (1.09 ms against 0.96
//    for 60M rows): the reservations of a tile waited on one another and on
//    two barriers while no loads were in flight.  The chunked layout took that
//    to 0.74 ms, the run-time compiled scan to 0.57, four lists per partition
//    to 0.47;
//  * k_rec_direct / k_rec_hash aggregate one partition per CTA in shared memory
//    (32-bit atomics; sums as two words with carries), a dense range of keys
//    directly addressed or a sparse one hashed and then put in key order, and
//    write the groups over the partition's records;
//  * partitions are key ranges, so an exclusive scan of their group counts gives
//    every group its place in the ordered result and k_rec_emit copies them
//    there: no sort.
//
// A partition that outgrows its region or its table sets ERR_RECORDS and the
// caller aggregates through the global table instead.
#include <algorithm>

#include "records.cuh"

namespace tpk {

constexpr int RAGG_THREADS = 512;

// Rows r .. r + 3 of a column (r a multiple of 4, all of them in range): one
// or two vector loads; 16-byte aligned columns.
__device__ __forceinline__ void ld_quad(const DevCol& c, uint64_t r, int64_t v[4]) {
    switch (c.type) {
    case T_I32: {
        const int4 a = __ldcs(reinterpret_cast<const int4*>((const int32_t*)c.ptr + r));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        break;
    }
    case T_I64: {
        const longlong2* p = reinterpret_cast<const longlong2*>((const int64_t*)c.ptr + r);
        const longlong2 a = __ldcs(p), b = __ldcs(p + 1);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
        break;
    }
    default: {
        const uchar4 a = __ldcs(reinterpret_cast<const uchar4*>((const uint8_t*)c.ptr + r));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        break;
    }
    }
}

// The same for the last rows of a table: those at or past n read as 0.
__device__ __forceinline__ void ld_quad_n(const DevCol& c, uint64_t r, uint64_t n, int64_t v[4]) {
    if (r + 4 <= n) {
        ld_quad(c, r, v);
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = r + i < n ? ld1(c, r + i) : 0;
}

// Packs one more group field (values f of `bits` bits) into the keys; bad
// collects the rows whose value does not fit.
__device__ __forceinline__ void pack_field(const int64_t f[4], int bits, uint64_t key[4], uint32_t& bad) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (bits < 64) {
            bad |= (uint32_t)(((uint64_t)f[i] >> bits) != 0) << i;
            key[i] = (key[i] << bits) | (uint64_t)f[i];
        } else {
            key[i] = (uint64_t)f[i];
        }
    }
}

// probe4 as a call of its own: the hashed walks need more registers than the
// scans have to spare, and inside them they spilled on the direct tables' path
// too.
__device__ __noinline__ uint32_t probe4_call(const JoinTable& jt, int64_t k0, int64_t k1, int64_t k2, int64_t k3,
                                             uint32_t pm, uint32_t* out, uint32_t* err) {
    const int64_t key[4] = {k0, k1, k2, k3};
    bool pass[4];
    uint32_t pay[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) pass[i] = pm >> i & 1u;
    probe4<true>(jt, key, pass, pay, err);
    pm = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        out[i] = pay[i];
        pm |= (uint32_t)pass[i] << i;
    }
    return pm;
}

// Join of four rows whose foreign keys are fk, then the check of their group
// fields (bad): out-of-range values matter only in rows that survive.
__device__ __forceinline__ void join_rows(const QueryDev& q, const int64_t fk[4], uint32_t bad, bool pass[4]) {
    if (q.has_join) {
        uint32_t pay[4];
        if (q.jt.direct && q.jt.lip == nullptr) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint64_t idx = (uint64_t)fk[i] - (uint64_t)q.jt.kmin;
                pay[i] = pass[i] && idx < q.jt.range ? __ldg((const unsigned int*)q.jt.slots + idx) : EMPTY32;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) pass[i] = pass[i] && pay[i] != EMPTY32;
        } else {
            const uint32_t pm = probe4_call(q.jt, fk[0], fk[1], fk[2], fk[3],
                                            pass[0] | pass[1] << 1 | pass[2] << 2 | pass[3] << 3, pay, q.err);
#pragma unroll
            for (int i = 0; i < 4; ++i) pass[i] = pm >> i & 1u;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (pass[i] && (pay[i] & PAYLOAD_BAD)) {
                atomicOr(q.err, ERR_RANGE);
                pass[i] = false;
            }
        }
    }
    if (bad == 0) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (pass[i] && (bad >> i & 1u)) {
            atomicOr(q.err, ERR_RANGE);
            pass[i] = false;
        }
    }
}

// The whole scan, every column of a row loaded up front.  Bound by HBM: the
// columns once and the records written and read again.
template <int NS>
__global__ void __launch_bounds__(REC_THREADS, NS > 2 ? 2 : 4)
    k_rec_scan(const __grid_constant__ QueryDev q, uint64_t n, const __grid_constant__ RecDev rec) {
    for (uint64_t t0 = (uint64_t)blockIdx.x * REC_TILE; t0 < n; t0 += (uint64_t)gridDim.x * REC_TILE) {
        const uint64_t r = t0 + (uint64_t)threadIdx.x * REC_RPT;
        bool pass[4];
        int64_t fv[4], fk[4], a[NS][4], b[NS][4];
        uint64_t key[4] = {0, 0, 0, 0};
        uint32_t bad = 0;
        if (q.has_filter) ld_quad_n(q.fcol, r, n, fv);
        if (q.has_join) ld_quad_n(q.fk, r, n, fk);
        for (int g = 0; g < q.n_group; ++g) {
            int64_t v[4];
            ld_quad_n(q.gcol[g], r, n, v);
            pack_field(v, q.gbits[g], key, bad);
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if (s >= q.n_sum) continue;
            ld_quad_n(q.sa[s], r, n, a[s]);
            if (q.skind[s] == S_MUL_SUB) ld_quad_n(q.sb[s], r, n, b[s]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            pass[i] = r + i < n && (!q.has_filter || (fv[i] >= q.flo && fv[i] <= q.fhi));
        join_rows(q, fk, bad, pass);
        int64_t t[NS][4];
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                t[s][i] = 0;
                if (s < q.n_sum)
                    t[s][i] = q.skind[s] == S_MUL_SUB
                                  ? (int64_t)((uint64_t)a[s][i] * ((uint64_t)q.sk[s] - (uint64_t)b[s][i]))
                                  : a[s][i];
            }
        fold_append<NS>(q, rec, pass, key, t);
    }
}

// The selected rows (four consecutive entries of the selection vector per
// thread), their columns gathered; the filter is not evaluated again.
template <int NS>
__global__ void __launch_bounds__(REC_THREADS, NS > 2 ? 2 : 4)
    k_rec_selected(const __grid_constant__ QueryDev q, const uint32_t* __restrict__ sel,
                   const unsigned long long* count, const __grid_constant__ RecDev rec) {
    const uint64_t n = *count;
    for (uint64_t t0 = (uint64_t)blockIdx.x * REC_TILE; t0 < n; t0 += (uint64_t)gridDim.x * REC_TILE) {
        const uint64_t e = t0 + (uint64_t)threadIdx.x * REC_RPT;
        bool pass[4];
        uint64_t row[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            pass[i] = e + i < n;
            row[i] = pass[i] ? (uint64_t)__ldcs(sel + e + i) : 0;
        }
        int64_t fk[4], a[NS][4], b[NS][4];
        uint64_t key[4] = {0, 0, 0, 0};
        uint32_t bad = 0;
        for (int g = 0; g < q.n_group; ++g) {
            int64_t v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = pass[i] ? ld1(q.gcol[g], row[i]) : 0;
            pack_field(v, q.gbits[g], key, bad);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            fk[i] = q.has_join && pass[i] ? ld1(q.fk, row[i]) : 0;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const bool on = s < q.n_sum && pass[i];
                a[s][i] = on ? ld1(q.sa[s], row[i]) : 0;
                b[s][i] = on && q.skind[s] == S_MUL_SUB ? ld1(q.sb[s], row[i]) : 0;
            }
        }
        join_rows(q, fk, bad, pass);
        int64_t t[NS][4];
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                t[s][i] = s < q.n_sum && q.skind[s] == S_MUL_SUB
                              ? (int64_t)((uint64_t)a[s][i] * ((uint64_t)q.sk[s] - (uint64_t)b[s][i]))
                              : a[s][i];
        fold_append<NS>(q, rec, pass, key, t);
    }
}

// 32-bit atomics and loads at shared-memory addresses: through generic pointers
// the hashed partitions took 400 us for 30M records, this way 336.
__device__ __forceinline__ uint32_t sm_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void sm_red(uint32_t a, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t sm_add(uint32_t a, uint32_t v) {
    uint32_t old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ uint32_t sm_cas(uint32_t a, uint32_t was, uint32_t v) {
    uint32_t old;
    asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(old) : "r"(a), "r"(was), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ uint32_t sm_ld(uint32_t a) {
    uint32_t v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

// Adds a record's count and sums to slot k of a table of K slots in shared
// memory at cnt: count[K], then low[K], high[K] per sum.
template <int NS>
__device__ __forceinline__ void add_record(uint32_t cnt, uint32_t K, uint32_t k, int n_sum, uint32_t c,
                                           const uint64_t v[NS]) {
    uint32_t a = cnt + 4 * k;
    sm_red(a, c);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        if (s >= n_sum) break;
        a += 4 * K;
        const uint32_t old = sm_add(a, (uint32_t)v[s]);
        a += 4 * K;
        const uint32_t h = (uint32_t)(v[s] >> 32) + (old + (uint32_t)v[s] < old ? 1u : 0u);
        if (h) sm_red(a, h);
    }
}

// Calls fn(on, key, rows, sums) for every record of partition p (on: this lane
// has one; all lanes of a warp make the same calls), each way's list by the
// warps of its own share of the CTA, RAGG_UNROLL records' loads per thread
// ahead of their use.
constexpr int RAGG_UNROLL = 4;
template <int NS, class F>
__device__ __forceinline__ void for_each_record(const RecDev& rec, uint32_t p, int n_sum, F&& fn) {
    constexpr uint32_t SHARE = RAGG_THREADS / REC_WAYS;
    static_assert(SHARE % 32 == 0, "a warp reads one list");
    const uint32_t list = p * REC_WAYS + threadIdx.x / SHARE;
    const uint32_t n = min(rec.cursor[(uint64_t)list * REC_CURSOR_STRIDE], rec.cap);
    for (uint32_t i0 = 0; i0 < n; i0 += SHARE * RAGG_UNROLL) {
        uint4 r[RAGG_UNROLL];
        uint64_t v[RAGG_UNROLL][NS];
#pragma unroll
        for (int u = 0; u < RAGG_UNROLL; ++u) {
            const uint32_t i = i0 + u * SHARE + threadIdx.x % SHARE;
            r[u] = make_uint4(0, 0, 0, 0);
            if (i >= n) continue;
            const uint64_t w = rec_at(rec, list, i);
            r[u] = __ldcs(rec.r0 + w);
#pragma unroll
            for (int s = 1; s < NS; ++s)
                if (s < n_sum) v[u][s] = __ldcs((const unsigned long long*)rec.sum[s] + w);
        }
#pragma unroll
        for (int u = 0; u < RAGG_UNROLL; ++u) {
            v[u][0] = (uint64_t)r[u].w << 32 | r[u].z;
            fn(i0 + u * SHARE + threadIdx.x % SHARE < n, r[u].x, r[u].y, v[u]);
        }
    }
}

// One partition per CTA: keys [0, 2^shift) of its range directly addressed.
// The table is cleared once; a partition's groups clear their own slots as
// they leave.  A warp takes a contiguous share of the keys, counts its groups,
// and after one barrier writes them at its place.
template <int NS>
__global__ void __launch_bounds__(RAGG_THREADS)
    k_rec_direct(const __grid_constant__ RecDev rec, int n_sum, uint32_t* __restrict__ groups) {
    extern __shared__ __align__(16) uint32_t rsm[];
    __shared__ uint32_t warp_tot[RAGG_THREADS / 32];
    constexpr uint32_t WARPS = RAGG_THREADS / 32;
    const uint32_t K = 1u << rec.shift, words = K * (1 + 2 * (uint32_t)n_sum);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t per = (K / 4 + 32 * WARPS - 1) / (32 * WARPS) * 128;   // keys per warp: whole 128-key steps
    for (uint32_t i = threadIdx.x; i < words; i += RAGG_THREADS) rsm[i] = 0;
    __syncthreads();
    for (uint32_t p = blockIdx.x; p < rec.n_part; p += gridDim.x) {
        for_each_record<NS>(rec, p, n_sum, [&](bool on, uint32_t k, uint32_t c, const uint64_t (&v)[NS]) {
            if (on) add_record<NS>(sm_addr(rsm), K, k, n_sum, c, v);
        });
        __syncthreads();   // every record is read: the groups go over them
        const uint32_t kb = min(warp * per, K), ke = min(kb + per, K);
        uint32_t mine = 0;
        for (uint32_t k = kb + 4 * lane; k < ke; k += 128) {
            const uint4 c = *(const uint4*)(rsm + k);
            mine += (c.x != 0) + (c.y != 0) + (c.z != 0) + (c.w != 0);
        }
        mine = __reduce_add_sync(0xffffffffu, mine);
        if (lane == 0) warp_tot[warp] = mine;
        __syncthreads();
        uint32_t at = 0, all = 0;
#pragma unroll
        for (uint32_t w = 0; w < WARPS; ++w) {
            at += w < warp ? warp_tot[w] : 0u;
            all += warp_tot[w];
        }
        if (mine != 0)
            for (uint32_t k0 = kb; k0 < ke; k0 += 32) {
                const uint32_t k = k0 + lane;
                const uint32_t c = k < ke ? rsm[k] : 0u;
                const unsigned m = __ballot_sync(0xffffffffu, c != 0);
                if (c != 0) {
                    uint64_t v[NS];
                    rsm[k] = 0;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        if (s >= n_sum) break;
                        uint32_t* lo = rsm + (uint64_t)K * (1 + 2 * s) + k;
                        v[s] = (uint64_t)lo[K] << 32 | lo[0];
                        lo[0] = lo[K] = 0;
                    }
                    put_record<NS>(rec, group_at(rec, p, at + __popc(m & ((1u << lane) - 1u))), n_sum, k, c, v);
                }
                at += __popc(m);
            }
        if (threadIdx.x == 0) groups[p] = all;
        __syncthreads();
    }
}

// One partition per CTA, its keys hashed into REC_HASH slots; the groups are
// then ordered by their key's top REC_ORDER_BITS bits (a counting sort) and,
// among equal ones, by comparison.
constexpr int REC_ORDER_BITS = 11;
constexpr uint32_t REC_ORDER = 1u << REC_ORDER_BITS;
constexpr uint32_t REC_NO_KEY = 0xFFFFFFFFu;

template <int NS>
__global__ void __launch_bounds__(RAGG_THREADS)
    k_rec_hash(const __grid_constant__ RecDev rec, int n_sum, uint32_t* __restrict__ groups, uint32_t* err) {
    extern __shared__ uint32_t rsm[];
    __shared__ uint32_t warp_tot[RAGG_THREADS / 32];
    uint32_t* keys = rsm;
    uint32_t* cnt = keys + REC_HASH;                                      // count, then low and high words per sum
    uint32_t* first = cnt + REC_HASH * (1 + 2 * (uint32_t)n_sum);        // per bucket: its first place, then fill
    uint32_t* order = first + REC_ORDER + 1;                              // slots by bucket
    const int bshift = rec.shift > REC_ORDER_BITS ? rec.shift - REC_ORDER_BITS : 0;
    for (uint32_t p = blockIdx.x; p < rec.n_part; p += gridDim.x) {
        for (uint32_t i = threadIdx.x; i < REC_HASH * (1 + 2 * (uint32_t)n_sum); i += RAGG_THREADS) cnt[i] = 0;
        for (uint32_t i = threadIdx.x; i < REC_HASH; i += RAGG_THREADS) keys[i] = REC_NO_KEY;
        for (uint32_t i = threadIdx.x; i <= REC_ORDER; i += RAGG_THREADS) first[i] = 0;
        __syncthreads();
        // most records meet a key that is there: find it with plain loads, claim
        // only at an empty slot.  The walk goes on for the whole warp until its
        // last lane is done: left to themselves the lanes came out of it one by
        // one and did the rest apart (8 of 32 lanes busy on average, 336 us for
        // 30M records; 290 now, 20 lanes).
        for_each_record<NS>(rec, p, n_sum, [&](bool on, uint32_t key, uint32_t c, const uint64_t (&v)[NS]) {
            uint32_t s = (key * 0x9E3779B1u) >> (32 - REC_HASH_BITS), left = on ? REC_HASH : 0;
            while (__any_sync(0xffffffffu, left != 0)) {
                if (left == 0) continue;
                uint32_t k = sm_ld(sm_addr(keys) + 4 * s);
                if (k == REC_NO_KEY) {
                    k = sm_cas(sm_addr(keys) + 4 * s, REC_NO_KEY, key);
                    if (k == REC_NO_KEY) {
                        sm_red(sm_addr(first + 1) + 4 * (key >> bshift), 1u);
                        k = key;
                    }
                }
                if (k == key) {
                    left = 0;
                    continue;
                }
                s = (s + 1) & (REC_HASH - 1u);
                // a full table; one that is full in another partition means this one need not go on
                if (--left == 0 || ((left & 127u) == 0 && (*(volatile uint32_t*)err & ERR_RECORDS))) {
                    atomicOr(err, ERR_RECORDS);
                    left = 0;
                    on = false;
                }
            }
            if (on) add_record<NS>(sm_addr(cnt), REC_HASH, s, n_sum, c, v);
        });
        __syncthreads();
        // bucket starts: an inclusive scan of first[1 ..]
        {
            constexpr uint32_t PER = REC_ORDER / RAGG_THREADS;
            static_assert(PER * RAGG_THREADS == REC_ORDER, "whole buckets per thread");
            uint32_t v[PER], sum = 0;
#pragma unroll
            for (uint32_t j = 0; j < PER; ++j) {
                sum += first[1 + threadIdx.x * PER + j];
                v[j] = sum;
            }
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            uint32_t x = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) warp_tot[warp] = x;
            __syncthreads();
            uint32_t before = x - sum;
            for (int w = 0; w < warp; ++w) before += warp_tot[w];
#pragma unroll
            for (uint32_t j = 0; j < PER; ++j) first[1 + threadIdx.x * PER + j] = before + v[j];
            __syncthreads();
        }
        const uint32_t g = first[REC_ORDER];
        __syncthreads();   // everyone has g before the fill moves it
        // slots into their buckets, filled from the back: first[b + 1] - 1 down
        for (uint32_t s = threadIdx.x; s < REC_HASH; s += RAGG_THREADS) {
            const uint32_t k = keys[s];
            if (k != REC_NO_KEY) order[atomicSub(first + 1 + (k >> bshift), 1u) - 1u] = s;
        }
        __syncthreads();
        // first[b + 1] is now the bucket's start; its end is the next one's start
        for (uint32_t i = threadIdx.x; i < g; i += RAGG_THREADS) {
            const uint32_t s = order[i], k = keys[s], b = k >> bshift;
            const uint32_t lo = first[1 + b], hi = b + 1 < REC_ORDER ? first[2 + b] : g;
            uint32_t at = lo;
            for (uint32_t j = lo; j < hi; ++j) at += keys[order[j]] < k ? 1u : 0u;
            uint64_t v[NS];
#pragma unroll
            for (int u = 0; u < NS; ++u)
                if (u < n_sum)
                    v[u] = (uint64_t)cnt[(uint64_t)REC_HASH * (2 + 2 * u) + s] << 32 |
                           cnt[(uint64_t)REC_HASH * (1 + 2 * u) + s];
            put_record<NS>(rec, group_at(rec, p, at), n_sum, k, cnt[s], v);
        }
        if (threadIdx.x == 0) groups[p] = g;
        __syncthreads();
    }
}

// Groups of every partition to their places in the result, one CTA per
// partition at a time.
__global__ void __launch_bounds__(256) k_rec_emit(const __grid_constant__ RecDev rec, int n_sum,
                                                  const uint32_t* __restrict__ groups,
                                                  const unsigned long long* __restrict__ offsets,
                                                  const __grid_constant__ OutDev o) {
    for (uint32_t p = blockIdx.x; p < rec.n_part; p += gridDim.x) {
        const uint32_t n = groups[p];
        const uint64_t out = offsets[p];
        const uint64_t k0 = rec.kmin + ((uint64_t)p << rec.shift);
        for (uint32_t i = threadIdx.x; i < n; i += 256) {
            const uint64_t w = group_at(rec, p, i);
            const uint4 r = __ldcs(rec.r0 + w);
            __stcs((unsigned long long*)o.keys + out + i, (unsigned long long)(k0 + r.x));
            __stcs((long long*)o.counts + out + i, (long long)r.y);
            for (int s = 0; s < n_sum; ++s) {
                const uint64_t lo =
                    s == 0 ? (uint64_t)r.w << 32 | r.z : __ldcs((const unsigned long long*)rec.sum[s] + w);
                const uint64_t hi = (uint64_t)((int64_t)lo >> 63);
                __stcs((ulonglong2*)o.sums[s] + out + i, make_ulonglong2(lo, hi));
                if (o.has_avg[s])
                    o.avgs[s][out + i] = __ddiv_rn(i128_to_double(lo, hi), __ll2double_rn((long long)r.y));
            }
        }
    }
}

// How evenly samples of the passing rows spread over the partitions: hist
// (n_part + 1 zeroed words) counts them, and the CTA that ends last writes
// out[0] = samples passing the filter, out[1] = most in one partition.
constexpr int RSAMPLE_THREADS = 256;
__global__ void __launch_bounds__(RSAMPLE_THREADS)
    k_rec_sample(const __grid_constant__ QueryDev q, uint64_t n, uint32_t samples, const __grid_constant__ RecDev rec,
                 uint32_t* hist, unsigned long long* out) {
    __shared__ uint32_t most, passed;
    __shared__ bool last;
    if (threadIdx.x == 0) most = passed = 0;
    for (uint32_t j = blockIdx.x * RSAMPLE_THREADS + threadIdx.x; j < samples; j += gridDim.x * RSAMPLE_THREADS) {
        const uint64_t r = (uint64_t)(((unsigned __int128)j * n) / samples);
        if (q.has_filter) {
            const int64_t v = ld1(q.fcol, r);
            if (v < q.flo || v > q.fhi) continue;
        }
        uint64_t key = 0;
        for (int g = 0; g < q.n_group; ++g) {
            const uint64_t f = (uint64_t)ld1(q.gcol[g], r);
            key = q.gbits[g] < 64 ? key << q.gbits[g] | f : f;
        }
        key -= rec.kmin;
        if (key < rec.span) atomicAdd(&hist[key >> rec.shift], 1u);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&hist[rec.n_part], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    uint32_t mine = 0, top = 0;
    for (uint32_t p = threadIdx.x; p < rec.n_part; p += RSAMPLE_THREADS) {
        const uint32_t c = __ldcg(hist + p);
        mine += c;
        top = max(top, c);
    }
    atomicAdd(&passed, mine);
    atomicMax(&most, top);
    __syncthreads();
    if (threadIdx.x == 0) {
        out[0] = passed;
        out[1] = most;
    }
}

// Distinct group keys of the rows that pass the filter, by HyperLogLog (Flajolet et al. 2007) over 2^12
// registers: the top bits of a key's hash pick a register, which keeps the
// longest run of leading zeros of the rest, plus one.
__global__ void __launch_bounds__(REC_THREADS)
    k_rec_distinct(const __grid_constant__ QueryDev q, uint64_t n, uint32_t* __restrict__ regs) {
    __shared__ uint32_t sm[HLL_REGS];
    for (uint32_t i = threadIdx.x; i < HLL_REGS; i += REC_THREADS) sm[i] = 0;
    __syncthreads();
    for (uint64_t r = ((uint64_t)blockIdx.x * REC_THREADS + threadIdx.x) * 4; r < n;
         r += (uint64_t)gridDim.x * REC_THREADS * 4) {
        uint64_t key[4] = {0, 0, 0, 0};
        uint32_t pm = 15u;
        if (q.has_filter) {
            int64_t f[4];
            ld_quad_n(q.fcol, r, n, f);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (f[i] < q.flo || f[i] > q.fhi) pm &= ~(1u << i);
            if (pm == 0) continue;
        }
        for (int g = 0; g < q.n_group; ++g) {
            int64_t v[4];
            ld_quad_n(q.gcol[g], r, n, v);
#pragma unroll
            for (int i = 0; i < 4; ++i) key[i] = q.gbits[g] < 64 ? key[i] << q.gbits[g] | (uint64_t)v[i] : (uint64_t)v[i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (r + i >= n || !(pm >> i & 1u) || (i > 0 && (pm >> (i - 1) & 1u) && key[i] == key[i - 1])) continue;
            const uint64_t h = fmix64(key[i]);
            const uint32_t z = (uint32_t)__clzll((long long)(h << HLL_BITS | 1ull << (HLL_BITS - 1))) + 1u;
            uint32_t* w = sm + (h >> (64 - HLL_BITS));
            if (*(volatile uint32_t*)w < z) atomicMax(w, z);
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < HLL_REGS; i += REC_THREADS)
        if (sm[i]) atomicMax(regs + i, sm[i]);
}

// ------------------------------------------------------------------- host

cudaError_t launch_rec_distinct(const QueryDev& q, uint64_t n, uint32_t* regs, int num_sms, cudaStream_t st) {
    const uint64_t blocks = (n + REC_TILE - 1) / REC_TILE;
    k_rec_distinct<<<(unsigned)std::min<uint64_t>(blocks, (uint64_t)num_sms * 4), REC_THREADS, 0, st>>>(q, n, regs);
    return cudaGetLastError();
}

uint32_t rec_hash_smem(int n_sum) { return 4 * (REC_HASH * (3 + 2 * (uint32_t)n_sum) + REC_ORDER + 1); }
uint32_t rec_direct_smem(int shift, int n_sum) { return (4u << shift) * (1 + 2 * (uint32_t)n_sum); }

template <class K>
static cudaError_t rec_grid(K fn, int threads, uint32_t smem, uint64_t blocks, int num_sms, unsigned* grid) {
    cudaError_t e = ensure_smem_limit((const void*)fn, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    if (e != cudaSuccess) return e;
    *grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(blocks, (uint64_t)num_sms * std::max(per_sm, 1)));
    return cudaSuccess;
}

template <int NS>
static cudaError_t rec_scan_t(const QueryDev& q, uint64_t n, const RecDev& rec, int num_sms, cudaStream_t st) {
    unsigned grid;
    const uint32_t smem = 0;
    cudaError_t e = rec_grid(k_rec_scan<NS>, REC_THREADS, smem, (n + REC_TILE - 1) / REC_TILE, num_sms, &grid);
    if (e != cudaSuccess) return e;
    k_rec_scan<NS><<<grid, REC_THREADS, smem, st>>>(q, n, rec);
    return cudaGetLastError();
}

cudaError_t launch_rec_scan(const QueryDev& q, uint64_t n, const RecDev& rec, int num_sms, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (q.n_sum <= 1) return rec_scan_t<1>(q, n, rec, num_sms, st);
    if (q.n_sum <= 2) return rec_scan_t<2>(q, n, rec, num_sms, st);
    return rec_scan_t<REC_MAX_SUM>(q, n, rec, num_sms, st);
}

cudaError_t launch_rec_scan_jit(const void* kernel, const QueryDev& q, uint64_t n, const uint32_t* sel,
                                const unsigned long long* count, const RecDev& rec, int num_sms, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, REC_THREADS, 0);
    if (e != cudaSuccess) return e;
    const uint64_t blocks = (n + REC_TILE - 1) / REC_TILE;
    const unsigned grid = (unsigned)std::min<uint64_t>(blocks, (uint64_t)num_sms * std::max(per_sm, 1));
    QueryDev qa = q;
    RecDev ra = rec;
    void* args[] = {&qa, &n, &sel, &count, &ra};
    return cudaLaunchKernel(kernel, dim3(grid), dim3(REC_THREADS), args, 0, st);
}

template <int NS>
static cudaError_t rec_selected_t(const QueryDev& q, const uint32_t* sel, const unsigned long long* count,
                                  uint64_t max_rows, const RecDev& rec, int num_sms, cudaStream_t st) {
    unsigned grid;
    const uint32_t smem = 0;
    cudaError_t e = rec_grid(k_rec_selected<NS>, REC_THREADS, smem, (max_rows + REC_TILE - 1) / REC_TILE, num_sms, &grid);
    if (e != cudaSuccess) return e;
    k_rec_selected<NS><<<grid, REC_THREADS, smem, st>>>(q, sel, count, rec);
    return cudaGetLastError();
}

cudaError_t launch_rec_selected(const QueryDev& q, const uint32_t* sel, const unsigned long long* count,
                                uint64_t max_rows, const RecDev& rec, int num_sms, cudaStream_t st) {
    if (max_rows == 0) return cudaSuccess;
    if (q.n_sum <= 1) return rec_selected_t<1>(q, sel, count, max_rows, rec, num_sms, st);
    if (q.n_sum <= 2) return rec_selected_t<2>(q, sel, count, max_rows, rec, num_sms, st);
    return rec_selected_t<REC_MAX_SUM>(q, sel, count, max_rows, rec, num_sms, st);
}

template <int NS>
static cudaError_t rec_aggregate_t(const RecDev& rec, int n_sum, bool hashed, uint32_t* groups, uint32_t* err,
                                   int num_sms, cudaStream_t st) {
    unsigned grid;
    cudaError_t e;
    if (hashed) {
        const uint32_t smem = rec_hash_smem(n_sum);
        if ((e = rec_grid(k_rec_hash<NS>, RAGG_THREADS, smem, rec.n_part, num_sms, &grid)) != cudaSuccess) return e;
        k_rec_hash<NS><<<grid, RAGG_THREADS, smem, st>>>(rec, n_sum, groups, err);
    } else {
        const uint32_t smem = rec_direct_smem(rec.shift, n_sum);
        if ((e = rec_grid(k_rec_direct<NS>, RAGG_THREADS, smem, rec.n_part, num_sms, &grid)) != cudaSuccess) return e;
        k_rec_direct<NS><<<grid, RAGG_THREADS, smem, st>>>(rec, n_sum, groups);
    }
    return cudaGetLastError();
}

cudaError_t launch_rec_aggregate(const RecDev& rec, int n_sum, bool hashed, uint32_t* groups, uint32_t* err,
                                 int num_sms, cudaStream_t st) {
    if (n_sum <= 1) return rec_aggregate_t<1>(rec, n_sum, hashed, groups, err, num_sms, st);
    if (n_sum <= 2) return rec_aggregate_t<2>(rec, n_sum, hashed, groups, err, num_sms, st);
    return rec_aggregate_t<REC_MAX_SUM>(rec, n_sum, hashed, groups, err, num_sms, st);
}

cudaError_t launch_rec_emit(const RecDev& rec, int n_sum, const uint32_t* groups, const unsigned long long* offsets,
                            const OutDev& o, int num_sms, cudaStream_t st) {
    const unsigned grid = std::min<uint32_t>(rec.n_part, (uint32_t)num_sms * 8);
    k_rec_emit<<<grid, 256, 0, st>>>(rec, n_sum, groups, offsets, o);
    return cudaGetLastError();
}

cudaError_t launch_rec_sample(const QueryDev& q, uint64_t n, uint32_t samples, const RecDev& rec,
                              uint32_t* hist, unsigned long long* out, cudaStream_t st) {
    const unsigned grid = (samples + RSAMPLE_THREADS - 1) / RSAMPLE_THREADS;
    k_rec_sample<<<std::min(grid, 256u), RSAMPLE_THREADS, 0, st>>>(q, n, samples, rec, hist, out);
    return cudaGetLastError();
}

}  // namespace tpk
