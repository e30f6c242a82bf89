// Records of the partitioned many-group aggregation (records.cu): their places
// and the appends of the scans.
#pragma once
#include "device.cuh"

namespace tpk {

constexpr int REC_THREADS = 256;
constexpr int REC_RPT = 4;                            // rows per thread per tile
constexpr int REC_TILE = REC_THREADS * REC_RPT;

__device__ __forceinline__ uint64_t rec_at(const RecDev& rec, uint32_t l, uint32_t i) {
    return ((uint64_t)(i / REC_CHUNK) * (rec.n_part * REC_WAYS) + l) * REC_CHUNK + i % REC_CHUNK;
}

// Place of the i-th group of partition p: its lists' places one after another.
__device__ __forceinline__ uint64_t group_at(const RecDev& rec, uint32_t p, uint32_t i) {
    return rec_at(rec, p * REC_WAYS + i / rec.cap, i % rec.cap);
}

// Writes / reads record w.
template <int NS>
__device__ __forceinline__ void put_record(const RecDev& rec, uint64_t w, int n_sum, uint32_t key, uint32_t rows,
                                           const uint64_t v[NS]) {
    const uint64_t v0 = n_sum > 0 ? v[0] : 0;
    rec.r0[w] = make_uint4(key, rows, (uint32_t)v0, (uint32_t)(v0 >> 32));
#pragma unroll
    for (int s = 1; s < NS; ++s)
        if (s < n_sum) rec.sum[s][w] = v[s];
}

// Appends the warp's records (valid[i]) to their partitions; all 32 lanes call
// it.
template <int NS>
__device__ __forceinline__ void append_records(const RecDev& rec, int n_sum, uint32_t* err, const bool valid[REC_RPT],
                                               const uint64_t local[REC_RPT], const uint32_t cnt[REC_RPT],
                                               const int64_t t[NS][REC_RPT]) {
    const uint32_t lane = threadIdx.x & 31u, way = (threadIdx.x >> 5) % REC_WAYS;
    uint32_t list[REC_RPT], at[REC_RPT], peers[REC_RPT];
#pragma unroll
    for (int i = 0; i < REC_RPT; ++i) {   // the atomics of all four records in flight together
        peers[i] = 0;
        at[i] = 0;
        list[i] = valid[i] ? (uint32_t)(local[i] >> rec.shift) * REC_WAYS + way : 0xFFFFFFFFu;
        if (__ballot_sync(0xffffffffu, valid[i]) == 0) continue;
        peers[i] = __match_any_sync(0xffffffffu, list[i]);
        if (valid[i] && lane == (uint32_t)__ffs(peers[i]) - 1u)
            at[i] = atomicAdd(&rec.cursor[(uint64_t)list[i] * REC_CURSOR_STRIDE], (uint32_t)__popc(peers[i]));
    }
    const uint32_t mask = (uint32_t)((1ull << rec.shift) - 1ull);
#pragma unroll
    for (int i = 0; i < REC_RPT; ++i) {
        if (__ballot_sync(0xffffffffu, valid[i]) == 0) continue;
        const uint32_t base = __shfl_sync(0xffffffffu, at[i], __ffs(peers[i]) - 1);
        if (!valid[i]) continue;
        const uint32_t pos = base + __popc(peers[i] & ((1u << lane) - 1u));
        if (pos >= rec.cap) {
            atomicOr(err, ERR_RECORDS);
            continue;
        }
        uint64_t v[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) v[s] = (uint64_t)t[s][i];
        put_record<NS>(rec, rec_at(rec, list[i], pos), n_sum, (uint32_t)local[i] & mask, cnt[i], v);
    }
}

// Folds a thread's rows of equal keys into the first of them, then appends.
template <int NS>
__device__ __forceinline__ void fold_append(const QueryDev& q, const RecDev& rec, bool pass[REC_RPT],
                                            const uint64_t key[REC_RPT], int64_t t[NS][REC_RPT]) {
    uint64_t local[REC_RPT];
    uint32_t cnt[REC_RPT];
#pragma unroll
    for (int i = 0; i < REC_RPT; ++i) {
        local[i] = key[i] - rec.kmin;
        cnt[i] = 1;
        if (pass[i] && local[i] >= rec.span) {   // a caller's column changed since its bounds were taken
            atomicOr(q.err, ERR_RECORDS);
            pass[i] = false;
        }
    }
#pragma unroll
    for (int i = 1; i < REC_RPT; ++i) {
        bool done = !pass[i];
#pragma unroll
        for (int j = 0; j < i; ++j) {
            if (done || !pass[j] || local[j] != local[i]) continue;
            cnt[j] += 1;
#pragma unroll
            for (int s = 0; s < NS; ++s) t[s][j] = (int64_t)((uint64_t)t[s][j] + (uint64_t)t[s][i]);
            pass[i] = false;
            done = true;
        }
    }
    append_records<NS>(rec, q.n_sum, q.err, pass, local, cnt, t);
}

}  // namespace tpk
