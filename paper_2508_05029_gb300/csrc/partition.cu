// Radix partitioning for the out-of-core (hybrid) hash join.
//
// Paper basis: Section 3.1 (Batch Holders move data to a larger memory tier
// when the GPU's is scarce), Section 3.3.2 (the Memory Executor spills data
// that is not needed soon), Section 3.2 (the exchange hash-partitions both
// join sides).  On one GPU both sides of the join are split into P = 2^k
// partitions by the top k bits of fmix64(key).  Partitions whose hash table
// fits the device budget stay resident and are probed while the fact table
// streams; the build and fact rows of the other partitions are written out
// (these kernels) and spilled to pinned host pages, then joined one partition
// at a time.
#include "device.cuh"

namespace tpk {

__device__ __forceinline__ uint32_t part_of(int64_t key, int shift) {
    return (uint32_t)(fmix64((uint64_t)key) >> shift);
}

// Per-block shared histogram of the admitted build rows, merged into counts.
__global__ void k_part_hist(const __grid_constant__ BuildDev b, uint64_t n, int shift, unsigned long long* counts) {
    __shared__ unsigned h[256];
    const uint32_t P = 1u << (64 - shift);
    for (uint32_t i = threadIdx.x; i < P; i += blockDim.x) h[i] = 0;
    __syncthreads();
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        if (dim_row_admitted(b, i)) atomicAdd(&h[part_of(ld1(b.key, i), shift)], 1u);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < P; i += blockDim.x)
        if (h[i]) atomicAdd(&counts[i], (unsigned long long)h[i]);
}

cudaError_t launch_part_hist(const BuildDev& b, uint64_t n, int shift, unsigned long long* counts, int num_sms,
                             cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (shift < 56 || shift > 63) return cudaErrorInvalidValue;   // 2..256 partitions
    uint64_t blocks = (n + 255) / 256;
    if (blocks > (uint64_t)num_sms * 4) blocks = (uint64_t)num_sms * 4;
    k_part_hist<<<(unsigned)blocks, 256, 0, st>>>(b, n, shift, counts);
    return cudaGetLastError();
}

__device__ __forceinline__ bool fact_row_passes(const QueryDev& q, uint64_t i) {
    if (!q.has_filter) return true;
    const int64_t v = ld1(q.fcol, i);
    return v >= q.flo && v <= q.fhi;
}

// Fact rows that pass the filter and the lookahead filter and fall in a
// spilled partition, per partition.
__global__ void k_part_hist_fact(const __grid_constant__ QueryDev q, uint64_t n, int shift, uint64_t spill_mask,
                                 unsigned long long* counts) {
    __shared__ unsigned h[256];
    const uint32_t P = 1u << (64 - shift);
    for (uint32_t i = threadIdx.x; i < P; i += blockDim.x) h[i] = 0;
    __syncthreads();
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        if (!fact_row_passes(q, i)) continue;
        const int64_t key = ld1(q.fk, i);
        const uint32_t p = part_of(key, shift);
        if (((spill_mask >> p) & 1ull) && (q.jt.lip == nullptr || lip_test(q.jt, key))) atomicAdd(&h[p], 1u);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < P; i += blockDim.x)
        if (h[i]) atomicAdd(&counts[i], (unsigned long long)h[i]);
}

cudaError_t launch_part_hist_fact(const QueryDev& q, uint64_t n, int shift, uint64_t spill_mask,
                                  unsigned long long* counts, int num_sms, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (shift < 58 || shift > 63) return cudaErrorInvalidValue;   // masks cover at most 64 partitions
    uint64_t blocks = (n + 255) / 256;
    if (blocks > (uint64_t)num_sms * 4) blocks = (uint64_t)num_sms * 4;
    k_part_hist_fact<<<(unsigned)blocks, 256, 0, st>>>(q, n, shift, spill_mask, counts);
    return cudaGetLastError();
}

// Scatter kernels place rows of spilled partitions with one global cursor
// atomic per (tile, partition): a tile of SP_TILE rows counts its rows per
// partition in shared memory, reserves each partition's range at once, and
// every row takes its rank inside its partition's range, so the rows of a
// partition from one tile land next to each other.
constexpr int SP_THREADS = 512;
constexpr int SP_RPT = 4;                          // rows per thread per tile
constexpr int SP_TILE = SP_THREADS * SP_RPT;

// Admitted build rows: insert the resident partitions, spill the others as
// pairs; every admitted key enters the lookahead filter.
__global__ void __launch_bounds__(SP_THREADS)
    k_build_part(const __grid_constant__ BuildDev b, uint64_t n, const unsigned long long* base,
                 unsigned long long* cursor, int64_t* keys, uint32_t* pays) {
    __shared__ unsigned cnt[64];
    __shared__ unsigned long long at0[64];
    const JoinTable& jt = b.jt;
    for (uint64_t t0 = (uint64_t)blockIdx.x * SP_TILE; t0 < n; t0 += (uint64_t)gridDim.x * SP_TILE) {
        if (threadIdx.x < 64) cnt[threadIdx.x] = 0;
        __syncthreads();
        uint32_t part[SP_RPT], rank[SP_RPT];
        bool spill[SP_RPT];
#pragma unroll
        for (int k = 0; k < SP_RPT; ++k) {
            const uint64_t i = t0 + (uint64_t)k * SP_THREADS + threadIdx.x;
            spill[k] = false;
            if (i >= n || !dim_row_admitted(b, i)) continue;
            const int64_t key = ld1(b.key, i);
            part[k] = part_of(key, jt.part_shift);
            if ((jt.part_mask >> part[k]) & 1ull) {
                build_insert(b, i);
            } else {
                if (jt.lip != nullptr) lip_insert(jt, key);
                spill[k] = true;
                rank[k] = atomicAdd(&cnt[part[k]], 1u);
            }
        }
        __syncthreads();
        if (threadIdx.x < 64 && cnt[threadIdx.x])
            at0[threadIdx.x] = base[threadIdx.x] + atomicAdd(&cursor[threadIdx.x], (unsigned long long)cnt[threadIdx.x]);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < SP_RPT; ++k) {
            if (!spill[k]) continue;
            const uint64_t i = t0 + (uint64_t)k * SP_THREADS + threadIdx.x;
            uint32_t payload = 0;
            for (int f = 0; f < b.n_dfield; ++f) {
                const int64_t v = ld1(b.dcol[f], i);
                if (v < 0 || ((uint64_t)v >> b.dbits[f]) != 0) payload |= PAYLOAD_BAD;
                else payload |= (uint32_t)((uint64_t)v << b.dpos[f]);
            }
            const uint64_t at = at0[part[k]] + rank[k];
            keys[at] = ld1(b.key, i);
            pays[at] = payload;
        }
        __syncthreads();
    }
}

cudaError_t launch_build_part(const BuildDev& b, uint64_t n, const unsigned long long* base,
                              unsigned long long* cursor, int64_t* keys, uint32_t* pays, int num_sms,
                              cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    uint64_t blocks = (n + SP_TILE - 1) / SP_TILE;
    if (blocks > (uint64_t)num_sms * 4) blocks = (uint64_t)num_sms * 4;
    k_build_part<<<(unsigned)blocks, SP_THREADS, 0, st>>>(b, n, base, cursor, keys, pays);
    return cudaGetLastError();
}

// Insert spilled (key, payload) pairs: the same table layout build_insert makes.
__global__ void k_build_pairs(const __grid_constant__ JoinTable jt, const int64_t* keys, const uint32_t* pays,
                              uint64_t n, uint32_t* err) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        // the payload is already packed: the same table logic as build_insert
        const int64_t key = keys[i];
        const uint32_t payload = pays[i];
        if (jt.direct) {
            const uint32_t v = (payload & PAYLOAD_BAD) ? PAYLOAD_BAD : payload;
            const uint64_t idx = (uint64_t)key - (uint64_t)jt.kmin;
            if (idx >= jt.range) { atomicOr(err, ERR_INTERNAL); continue; }
            if (atomicCAS((unsigned int*)jt.slots + idx, EMPTY32, v) != EMPTY32) atomicOr(err, ERR_DUP);
            continue;
        }
        const bool special = jt.key64 ? (uint64_t)key == EMPTY64 : (uint32_t)key == EMPTY32;
        if (special) {
            if (atomicCAS(jt.side, 0u, 1u) != 0u) atomicOr(err, ERR_DUP);
            else jt.side[1] = payload;
            continue;
        }
        uint64_t s = join_hash(jt, key) & jt.mask;
        bool placed = false;
        for (uint64_t it = 0; it <= jt.mask; ++it) {
            if (!jt.key64) {
                const unsigned long long want = ((unsigned long long)payload << 32) | (uint32_t)key;
                const unsigned long long prev =
                    atomicCAS((unsigned long long*)jt.slots + s, (unsigned long long)EMPTY64, want);
                if (prev == EMPTY64) { placed = true; break; }
                if ((uint32_t)prev == (uint32_t)key) { atomicOr(err, ERR_DUP); placed = true; break; }
            } else {
                const unsigned long long prev = atomicCAS((unsigned long long*)jt.slots + 2 * s,
                                                          (unsigned long long)EMPTY64, (unsigned long long)key);
                if (prev == EMPTY64) {
                    jt.slots[2 * s + 1] = payload;
                    placed = true;
                    break;
                }
                if (prev == (unsigned long long)key) { atomicOr(err, ERR_DUP); placed = true; break; }
            }
            s = (s + 1) & jt.mask;
        }
        if (!placed) atomicOr(err, ERR_INTERNAL);
    }
}

cudaError_t launch_build_pairs(const JoinTable& jt, const int64_t* keys, const uint32_t* pays, uint64_t n,
                               uint32_t* err, int num_sms, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > (uint64_t)num_sms * 8) blocks = (uint64_t)num_sms * 8;
    k_build_pairs<<<(unsigned)blocks, 256, 0, st>>>(jt, keys, pays, n, err);
    return cudaGetLastError();
}

// Fact rows of spilled partitions: copy every requested column to its
// partition's run in the staging columns, narrow where cols says so
// (tile-aggregated cursors, as above).
__global__ void __launch_bounds__(SP_THREADS)
    k_fact_spill(const __grid_constant__ QueryDev q, uint64_t n, uint64_t spill_mask,
                 const __grid_constant__ SpillCols cols, const unsigned long long* base, unsigned long long* cursor) {
    __shared__ unsigned cnt[64];
    __shared__ unsigned long long at0[64];
    const int shift = q.jt.part_shift;
    for (uint64_t t0 = (uint64_t)blockIdx.x * SP_TILE; t0 < n; t0 += (uint64_t)gridDim.x * SP_TILE) {
        if (threadIdx.x < 64) cnt[threadIdx.x] = 0;
        __syncthreads();
        uint32_t part[SP_RPT], rank[SP_RPT];
        bool spill[SP_RPT];
#pragma unroll
        for (int k = 0; k < SP_RPT; ++k) {
            const uint64_t i = t0 + (uint64_t)k * SP_THREADS + threadIdx.x;
            spill[k] = false;
            if (i >= n || !fact_row_passes(q, i)) continue;
            const int64_t key = ld1(q.fk, i);
            part[k] = part_of(key, shift);
            if (!((spill_mask >> part[k]) & 1ull)) continue;
            if (q.jt.lip != nullptr && !lip_test(q.jt, key)) continue;   // cannot join: not spilled
            spill[k] = true;
            rank[k] = atomicAdd(&cnt[part[k]], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 64 && cnt[threadIdx.x])
            at0[threadIdx.x] = base[threadIdx.x] + atomicAdd(&cursor[threadIdx.x], (unsigned long long)cnt[threadIdx.x]);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < SP_RPT; ++k) {
            if (!spill[k]) continue;
            const uint64_t i = t0 + (uint64_t)k * SP_THREADS + threadIdx.x;
            const uint64_t at = at0[part[k]] + rank[k];
            for (int c = 0; c < cols.n; ++c) {
                int64_t v;
                switch (cols.esize[c]) {
                case 8: v = ((const int64_t*)cols.src[c])[i]; break;
                case 4: v = ((const int32_t*)cols.src[c])[i]; break;
                default: v = ((const uint8_t*)cols.src[c])[i]; break;
                }
                const uint64_t d = cols.w[c] < cols.esize[c] ? (uint64_t)v - (uint64_t)cols.base[c] : (uint64_t)v;
                switch (cols.w[c]) {
                case 8: ((uint64_t*)cols.dst[c])[at] = d; break;
                case 4: ((uint32_t*)cols.dst[c])[at] = (uint32_t)d; break;
                case 2: ((uint16_t*)cols.dst[c])[at] = (uint16_t)d; break;
                default: ((uint8_t*)cols.dst[c])[at] = (uint8_t)d; break;
                }
            }
        }
        __syncthreads();
    }
}

cudaError_t launch_fact_spill(const QueryDev& q, uint64_t n, uint64_t spill_mask, const SpillCols& cols,
                              const unsigned long long* base, unsigned long long* cursor, int num_sms,
                              cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    uint64_t blocks = (n + SP_TILE - 1) / SP_TILE;
    if (blocks > (uint64_t)num_sms * 4) blocks = (uint64_t)num_sms * 4;
    k_fact_spill<<<(unsigned)blocks, SP_THREADS, 0, st>>>(q, n, spill_mask, cols, base, cursor);
    return cudaGetLastError();
}

// ------------------------------------------------------- fan-out build
//
// Groups the admitted build rows by key without sorting them: the join table
// itself counts a key's rows, the counts become run starts, and every row is
// written at its run's start plus its rank.  Runs come in slot order and rows
// in no order inside a run, which an inner join's sums do not see.  Three
// passes over rows or slots, bound by the table's random accesses.  Build and
// query of 20M fact rows over 1.5M build rows: 1.34 ms per pass when the
// (key, payload) pairs were sorted by 64 key bits (29 launches, 0.42 ms of
// kernels and two synchronisations), 0.97 ms grouped this way.

// The 32-bit word of table slot s that counts, then holds the start of, its
// key's run (the slot's payload).
__device__ __forceinline__ uint32_t* many_word(const JoinTable& jt, uint64_t s) {
    uint32_t* w = (uint32_t*)jt.slots;
    return jt.direct ? w + s : (jt.key64 ? w + 4 * s + 2 : w + 2 * s + 1);
}

// One row's key takes or finds its slot; the row's rank among the key's rows
// is what the slot's word counted before it.  The words start at all ones
// (the empty pattern), so a count of c rows reads c - 1.  The key equal to
// the empty pattern counts in the side cell, from zero.
__device__ __forceinline__ uint64_t many_insert(const JoinTable& jt, int64_t key, uint32_t* err, uint32_t* rank) {
    if (jt.direct) {
        const uint64_t idx = (uint64_t)key - (uint64_t)jt.kmin;
        if (idx >= jt.range) { atomicOr(err, ERR_INTERNAL); return MANY_NONE; }
        *rank = atomicAdd(many_word(jt, idx), 1u) + 1u;
        return idx;
    }
    if (jt.key64 ? (uint64_t)key == EMPTY64 : (uint32_t)key == EMPTY32) {
        jt.side[0] = 1;
        *rank = atomicAdd(jt.side + 1, 1u);
        return MANY_SIDE;
    }
    uint64_t s = join_hash(jt, key) & jt.mask;
    for (uint64_t it = 0; it <= jt.mask; ++it) {
        unsigned long long* p = (unsigned long long*)jt.slots + (jt.key64 ? 2 * s : s);
        bool mine;
        if (jt.key64) {
            const unsigned long long prev = atomicCAS(p, (unsigned long long)EMPTY64, (unsigned long long)key);
            mine = prev == EMPTY64 || prev == (unsigned long long)key;
        } else {
            const unsigned long long prev =
                atomicCAS(p, (unsigned long long)EMPTY64, ((unsigned long long)EMPTY32 << 32) | (uint32_t)key);
            mine = (uint32_t)prev == EMPTY32 || (uint32_t)prev == (uint32_t)key;
        }
        if (mine) {
            *rank = atomicAdd(many_word(jt, s), 1u) + 1u;
            return s;
        }
        s = (s + 1) & jt.mask;
    }
    atomicOr(err, ERR_INTERNAL);
    return MANY_NONE;
}

__global__ void k_many_count(const __grid_constant__ BuildDev b, uint64_t n, uint32_t* __restrict__ pays,
                             uint64_t* __restrict__ place) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        if (!dim_row_admitted(b, i)) {
            place[i] = MANY_NONE;
            continue;
        }
        const int64_t key = ld1(b.key, i);
        if (b.jt.lip != nullptr) lip_insert(b.jt, key);
        uint32_t rank = 0;
        const uint64_t s = many_insert(b.jt, key, b.err, &rank);
        pays[i] = build_payload(b, i);
        place[i] = s == MANY_NONE ? MANY_NONE : (s << MANY_RANK_BITS) | rank;
    }
}

cudaError_t launch_many_count(const BuildDev& b, uint64_t n, uint32_t* pays, uint64_t* place, int num_sms,
                              cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > (uint64_t)num_sms * 8) blocks = (uint64_t)num_sms * 8;
    k_many_count<<<(unsigned)blocks, 256, 0, st>>>(b, n, pays, place);
    return cudaGetLastError();
}

// Turns the counts of the table's slots into run starts; total[0] ends as the
// number of rows, total[1] as the longest run.  One reservation on *total per
// tile of MS_TILE slots: one per warp would queue on that word.
constexpr int MS_THREADS = 256;
constexpr int MS_ITEMS = 16;
constexpr int MS_TILE = MS_THREADS * MS_ITEMS;

__global__ void __launch_bounds__(MS_THREADS)
    k_many_starts(const __grid_constant__ JoinTable jt, uint64_t n_slots, uint2* __restrict__ rows,
                  unsigned long long* total, uint32_t limit, uint32_t* err) {
    __shared__ uint32_t warp_sum[MS_THREADS / 32];
    __shared__ unsigned long long base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t longest = 0;
    for (uint64_t t0 = (uint64_t)blockIdx.x * MS_TILE; t0 < n_slots; t0 += (uint64_t)gridDim.x * MS_TILE) {
        uint32_t cnt[MS_ITEMS], sum = 0;
#pragma unroll
        for (int j = 0; j < MS_ITEMS; ++j) {
            const uint64_t s = t0 + (uint64_t)j * MS_THREADS + threadIdx.x;
            cnt[j] = s < n_slots ? *many_word(jt, s) + 1u : 0u;
            sum += cnt[j];
            longest = max(longest, cnt[j]);
        }
        uint32_t x = sum;
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        uint32_t before = 0, all = 0;
        for (int w = 0; w < MS_THREADS / 32; ++w) {
            if (w < warp) before += warp_sum[w];
            all += warp_sum[w];
        }
        if (threadIdx.x == 0) base = atomicAdd(total, (unsigned long long)all);
        __syncthreads();
        uint32_t at = (uint32_t)base + before + x - sum;
#pragma unroll
        for (int j = 0; j < MS_ITEMS; ++j) {
            const uint64_t s = t0 + (uint64_t)j * MS_THREADS + threadIdx.x;
            if (cnt[j]) {
                *many_word(jt, s) = at;
                rows[at].y = cnt[j] - 1u;
            }
            at += cnt[j];
        }
        __syncthreads();
    }
    // the key equal to the empty pattern
    if (!jt.direct && blockIdx.x == 0 && threadIdx.x == 0 && jt.side[0] != 0) {
        const uint32_t n = jt.side[1], at = (uint32_t)atomicAdd(total, (unsigned long long)n);
        rows[at].y = n - 1u;
        jt.side[1] = at;
        longest = max(longest, n);
    }
    longest = __reduce_max_sync(0xffffffffu, longest);
    if (lane != 0 || longest == 0) return;
    if (longest > limit) atomicOr(err, ERR_FANOUT);
    atomicMax(total + 1, (unsigned long long)longest);
}

cudaError_t launch_many_starts(const JoinTable& jt, uint2* rows, unsigned long long* total, uint32_t limit,
                               uint32_t* err, int num_sms, cudaStream_t st) {
    const uint64_t n_slots = jt.direct ? jt.range : jt.mask + 1;
    uint64_t blocks = (n_slots + MS_TILE - 1) / MS_TILE;
    if (blocks > (uint64_t)num_sms * 8) blocks = (uint64_t)num_sms * 8;
    k_many_starts<<<(unsigned)blocks, MS_THREADS, 0, st>>>(jt, n_slots, rows, total, limit, err);
    return cudaGetLastError();
}

__global__ void k_many_place(const __grid_constant__ JoinTable jt, const uint32_t* __restrict__ pays,
                             const uint64_t* __restrict__ place, uint64_t n, uint2* __restrict__ rows) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t p = place[i];
        if (p == MANY_NONE) continue;
        const uint64_t s = p >> MANY_RANK_BITS;
        const uint32_t start = s == MANY_SIDE ? jt.side[1] : *many_word(jt, s);
        rows[(uint64_t)start + (p & ((1ull << MANY_RANK_BITS) - 1ull))].x = pays[i];
    }
}

cudaError_t launch_many_place(const JoinTable& jt, const uint32_t* pays, const uint64_t* place, uint64_t n,
                              uint2* rows, int num_sms, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > (uint64_t)num_sms * 8) blocks = (uint64_t)num_sms * 8;
    k_many_place<<<(unsigned)blocks, 256, 0, st>>>(jt, pays, place, n, rows);
    return cudaGetLastError();
}

}  // namespace tpk
