// Map-size updates between mapping iterations (RMGS-SLAM §III-C): low-opacity pruning under a
// bounded removal ratio, the 3-D proximity test that filters redundant new Gaussians before
// insertion, and the compaction that applies both to the parameter planes, the Adam moments
// and an optional per-row tag (e.g. the segment id that decides which rows are frozen).
//
// Pruning picks, among the rows with opacity below opacity_min (decided on the FP32 logit),
// at most floor(max_ratio * n) rows with the smallest (logit, row index): the candidates' keys
// (ordered logit bits, row index) are listed once, the k-th smallest is found by a radix select
// over that list (11 bits a round), and the rows at or below it are marked.  No sort.
//
// The proximity test hashes the map means into cubic cells of side 1.001 * radius; a new mean
// looks at the 27 cells around its own and is redundant if any map mean there lies strictly
// within radius (squared distance summed in FP32 in x, y, z order).
#include <cstddef>
#include <math_constants.h>

#include "gs_kernels.cuh"

namespace gs {

constexpr int kMuThreads = 256;

// True in every thread of the block that finishes last of the grid; what the other blocks wrote
// before their call is then visible to it (read it past L1).
__device__ __forceinline__ bool last_block(uint32_t* done) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// Exclusive scan over the block's threads (a whole number of warps).
template <typename U>
__device__ __forceinline__ U block_scan_excl(U x, U& total) {
    __shared__ U s_w[33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    U inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const U y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_w[w] = inc;
    __syncthreads();
    if (w == 0) {
        const U t = lane < (int)(blockDim.x >> 5) ? s_w[lane] : U(0);
        U ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const U y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        s_w[lane] = ti - t;
        if (lane == 31) s_w[32] = ti;
    }
    __syncthreads();
    total = s_w[32];
    const U r = s_w[w] + inc - x;
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------------------------------
// Prune plan.  One pass over the logits lists the candidates and counts their first digit; the
// later rounds and the marking read that list (2% of the rows, in L2) and not the map, and the
// block that finishes a histogram last picks its digit, so a round is one launch: at 2M rows, 2%
// of them candidates, 6 kernels of 43 us together instead of 19 of 205.  The pass over the
// logits (10 MB) is 13 of it, the rest chains of a few memory latencies each.  (An 11-bit digit
// takes 8 KB of counters; 8 bits would take 7 rounds for a 53-bit key instead of 5.)
// ---------------------------------------------------------------------------------------
constexpr int kDigitBits = 11, kDigits = 1 << kDigitBits, kMaxRounds = 6;
constexpr int kCollectRows = 8;   // rows per thread of the listing pass

struct alignas(32) SelectState {
    unsigned long long prefix;   // key bits decided so far
    unsigned long long rank;     // rank (1-based) of the threshold key inside the current prefix group
    unsigned long long kept;     // rows kept / new rows accepted
    uint32_t k;                  // rows to remove
    uint32_t count;              // candidates
    uint32_t done;               // blocks finished
    uint32_t hist[kMaxRounds][kDigits];
};

__device__ __forceinline__ unsigned long long prune_key(float logit, uint32_t i, int idx_bits) {
    const uint32_t b = __float_as_uint(logit);
    const uint32_t ord = (b >> 31) ? ~b : (b | 0x80000000u);   // monotone in the float value
    return ((unsigned long long)ord << idx_bits) | i;
}

// The last block: the digit holding the rank-th key of the prefix group.
__device__ __forceinline__ void prune_pick(const uint32_t* hist, int shift, SelectState* s) {
    constexpr int kPer = kDigits / kMuThreads;
    uint32_t h[kPer], sum = 0, tot;
#pragma unroll
    for (int j = 0; j < kPer; j++) sum += h[j] = __ldcg(&hist[threadIdx.x * kPer + j]);
    const unsigned long long rank = s->rank;
    uint32_t below = block_scan_excl(sum, tot);
    if (rank > below && rank <= (unsigned long long)below + sum) {   // one thread (rank 0: none)
        int j = 0;
        while (rank > (unsigned long long)below + h[j]) below += h[j++];
        s->prefix |= (unsigned long long)(threadIdx.x * kPer + j) << shift;
        s->rank = rank - below;
    }
    if (threadIdx.x == 0) s->done = 0;
}

__device__ __forceinline__ void hist_flush(const uint32_t* h, uint32_t* hist) {
    for (int t = threadIdx.x; t < kDigits; t += kMuThreads)
        if (h[t]) atomicAdd(&hist[t], h[t]);
}

__global__ void __launch_bounds__(kMuThreads) prune_collect_kernel(const float* lg, int64_t n, float thr,
                                                                   unsigned long long k_max, int idx_bits, int shift,
                                                                   unsigned long long* list, uint8_t* keep,
                                                                   SelectState* s) {
    __shared__ uint32_t h[kDigits];
    __shared__ uint32_t s_base;
    for (int t = threadIdx.x; t < kDigits; t += kMuThreads) h[t] = 0;
    const int64_t i0 = (int64_t)blockIdx.x * (kMuThreads * kCollectRows) + threadIdx.x;
    float x[kCollectRows];
    uint32_t mine = 0, tot;
#pragma unroll
    for (int j = 0; j < kCollectRows; j++) {
        const int64_t i = i0 + j * kMuThreads;
        x[j] = i < n ? lg[i] : CUDART_INF_F;
    }
#pragma unroll
    for (int j = 0; j < kCollectRows; j++) {
        const int64_t i = i0 + j * kMuThreads;
        if (i < n) keep[i] = 1;
        mine += i < n && x[j] < thr;
    }
    const uint32_t at = block_scan_excl(mine, tot);
    if (tot) {
        if (threadIdx.x == 0) s_base = atomicAdd(&s->count, tot);
        __syncthreads();
        uint32_t o = s_base + at;
#pragma unroll
        for (int j = 0; j < kCollectRows; j++) {
            const int64_t i = i0 + j * kMuThreads;
            if (i < n && x[j] < thr) {
                const unsigned long long key = prune_key(x[j], (uint32_t)i, idx_bits);
                list[o++] = key;
                atomicAdd(&h[key >> shift], 1u);
            }
        }
        __syncthreads();
        hist_flush(h, s->hist[0]);
    }
    if (!last_block(&s->done)) return;
    if (threadIdx.x == 0) {
        const uint32_t c = __ldcg(&s->count);
        s->k = c < k_max ? c : (uint32_t)k_max;
        s->rank = s->k;
        s->kept = (unsigned long long)n - s->k;
    }
    __syncthreads();
    prune_pick(s->hist[0], shift, s);
}

// Round r: histogram of the digit at `shift` of the listed keys whose higher digits equal the
// prefix.
__global__ void __launch_bounds__(kMuThreads) prune_round_kernel(const unsigned long long* list, int round, int shift,
                                                                 SelectState* s) {
    __shared__ uint32_t h[kDigits];
    pdl_begin();
    const uint32_t c = s->count;
    if (s->k == 0) return;
    for (int t = threadIdx.x; t < kDigits; t += kMuThreads) h[t] = 0;
    __syncthreads();
    const unsigned long long group = s->prefix >> (shift + kDigitBits);
    for (uint64_t i = (uint64_t)blockIdx.x * kMuThreads + threadIdx.x; i < c; i += (uint64_t)gridDim.x * kMuThreads) {
        const unsigned long long key = list[i];
        if (key >> (shift + kDigitBits) == group) atomicAdd(&h[(key >> shift) & (kDigits - 1)], 1u);
    }
    __syncthreads();
    hist_flush(h, s->hist[round]);
    if (last_block(&s->done)) prune_pick(s->hist[round], shift, s);
}

__global__ void __launch_bounds__(kMuThreads) prune_mark_kernel(const unsigned long long* list, int idx_bits,
                                                                const SelectState* s, uint8_t* keep) {
    pdl_begin();
    if (s->k == 0) return;
    const unsigned long long t = s->prefix, mask = (1ull << idx_bits) - 1;
    const uint32_t c = s->count;
    for (uint64_t i = (uint64_t)blockIdx.x * kMuThreads + threadIdx.x; i < c; i += (uint64_t)gridDim.x * kMuThreads) {
        const unsigned long long key = list[i];
        if (key <= t) keep[key & mask] = 0;
    }
}

// ---------------------------------------------------------------------------------------
// Proximity test.  The table holds a linked list per slot: the build is one pass over the means
// with one atomic exchange a row, and a row's coordinates and link are one 16-byte record, so a
// step along a list is one sector.  (A counting sort of the rows by slot took two passes with
// two atomics a row and a scan of the table, and each visit then read four sectors: 200 us for
// 2M means and 200k new ones, now 63.  Where very many map rows share a cell and none of them is
// near, a list is a long chain of reads: 200k rows in dense cells and 50k new ones beside them take
// 105, 115, 167, 542 and 3682 us at 1, 8, 64, 512 and 4096 rows a cell, the runs of the counting sort
// took 146, 165, 275, 713 and 2180.  With the same rows spread evenly most new ones are near: 73 to
// 86 us against 136 to 11137.)  Eight cells along x share a 32-byte sector of slots, so
// the 27 cells are 9 reads of mostly one sector; 9 lanes take a new mean, each a row of three
// cells whose lists it walks side by side, and all stop when one has found a near mean.  What
// bounds both kernels is the rate of scattered sector reads and atomics at L2.
// ---------------------------------------------------------------------------------------
constexpr int kBuildRows = 4;      // rows per thread of the build, all exchanges in flight together
constexpr int kQueryLanes = 9, kQueriesPerWarp = 3;

// 1 / cell side as a sum of two floats.
struct CellScale { float hi, lo; };

// floor(p / side).  The product is carried in two floats: FP64 here, at 1/64 of the FP32 rate,
// was half of the table's build.  Its error is below 1e-4 cells where two different floats p can
// be less than a side apart at all (beyond 2^30 cells they cannot, and only p itself counts), and
// a cell is 0.1% wider than the radius, so two means closer than the radius never end up two
// cells apart.
__device__ __forceinline__ int cell_of(float p, CellScale c) {
    const float h = __fmul_rn(p, c.hi);
    if (!(fabsf(h) < 1073741824.f)) return (int)h;
    const float l = __fmaf_rn(p, c.lo, __fmaf_rn(p, c.hi, -h)), f = floorf(h);
    return (int)f + (int)floorf(__fadd_rn(__fsub_rn(h, f), l));
}

__device__ __forceinline__ uint32_t cell_slot(int cx, int cy, int cz, uint32_t mask) {
    // large odd multipliers, XOR-combined; the low 3 bits of x stay so that neighbours share a sector
    const uint32_t h = (uint32_t)(cx >> 3) * 73856093u ^ (uint32_t)cy * 19349663u ^ (uint32_t)cz * 83492791u;
    return (h << 3 | ((uint32_t)cx & 7u)) & mask;
}

__device__ __forceinline__ int cell_add(int c, int d) { return (int)((uint32_t)c + (uint32_t)d); }

__global__ void __launch_bounds__(kMuThreads) hash_build_kernel(const float* mm, int64_t n, CellScale cs, uint32_t mask,
                                                                uint32_t* head, uint4* node) {
    const int64_t i0 = (int64_t)blockIdx.x * (kMuThreads * kBuildRows) + threadIdx.x;
    float x[kBuildRows], y[kBuildRows], z[kBuildRows];
#pragma unroll
    for (int j = 0; j < kBuildRows; j++) {
        const int64_t i = i0 + j * kMuThreads;
        x[j] = i < n ? mm[i] : 0.f;
        y[j] = i < n ? mm[n + i] : 0.f;
        z[j] = i < n ? mm[2 * n + i] : 0.f;
    }
    uint32_t next[kBuildRows];
#pragma unroll
    for (int j = 0; j < kBuildRows; j++) {
        const int64_t i = i0 + j * kMuThreads;
        if (i < n) next[j] = atomicExch(&head[cell_slot(cell_of(x[j], cs), cell_of(y[j], cs), cell_of(z[j], cs), mask)], (uint32_t)i + 1u);
    }
#pragma unroll
    for (int j = 0; j < kBuildRows; j++) {
        const int64_t i = i0 + j * kMuThreads;
        if (i < n) node[i] = make_uint4(__float_as_uint(x[j]), __float_as_uint(y[j]), __float_as_uint(z[j]), next[j]);
    }
}

__global__ void __launch_bounds__(kMuThreads) dedup_query_kernel(const float* qm, int64_t nq, CellScale cs, float r2,
                                                                 uint32_t mask, const uint32_t* __restrict__ head,
                                                                 const uint4* __restrict__ node, uint8_t* accept,
                                                                 SelectState* s) {
    __shared__ uint32_t s_acc;
    if (threadIdx.x == 0) s_acc = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, q = lane / kQueryLanes, row = lane - q * kQueryLanes;
    const int64_t j = ((int64_t)blockIdx.x * (kMuThreads / 32) + (threadIdx.x >> 5)) * kQueriesPerWarp + q;
    const bool on = q < kQueriesPerWarp && j < nq;
    const uint32_t group = q < kQueriesPerWarp ? ((1u << kQueryLanes) - 1u) << (q * kQueryLanes) : 0u;
    float qx = 0.f, qy = 0.f, qz = 0.f;
    uint32_t at[3] = {0u, 0u, 0u};   // 1 + the next record of each list, 0 at its end
    if (on) {
        qx = qm[j]; qy = qm[nq + j]; qz = qm[2 * nq + j];
        const int cx = cell_of(qx, cs), cy = cell_add(cell_of(qy, cs), row % 3 - 1), cz = cell_add(cell_of(qz, cs), row / 3 - 1);
#pragma unroll
        for (int k = 0; k < 3; k++) at[k] = head[cell_slot(cell_add(cx, k - 1), cy, cz, mask)];
    }
    bool near = false;
    while (__any_sync(0xffffffffu, (at[0] | at[1] | at[2]) != 0u)) {
        uint4 v[3];
#pragma unroll
        for (int k = 0; k < 3; k++)
            if (at[k]) v[k] = node[at[k] - 1u];
#pragma unroll
        for (int k = 0; k < 3; k++)
            if (at[k]) {
                const float ex = __fsub_rn(qx, __uint_as_float(v[k].x)), ey = __fsub_rn(qy, __uint_as_float(v[k].y)),
                            ez = __fsub_rn(qz, __uint_as_float(v[k].z));
                near |= __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez)) < r2;
                at[k] = v[k].w;
            }
        if (__ballot_sync(0xffffffffu, near) & group) at[0] = at[1] = at[2] = 0u;
    }
    const uint32_t found = __ballot_sync(0xffffffffu, near) & group;   // (every lane votes)
    const bool taken = on && !found;
    if (on && row == 0) accept[j] = taken ? 1 : 0;
    const uint32_t c = __popc(__ballot_sync(0xffffffffu, taken && row == 0));
    if (lane == 0 && c) atomicAdd(&s_acc, c);
    __syncthreads();
    if (threadIdx.x == 0 && s_acc) atomicAdd(&s->kept, (unsigned long long)s_acc);
}

// ---------------------------------------------------------------------------------------
// Exclusive scan of uint32 over up to 2^31 items: per-block totals, a scan of the totals in one
// block, then the per-item offsets.
// ---------------------------------------------------------------------------------------
constexpr int kScanT = 1024;

__global__ void __launch_bounds__(kScanT) scan_totals_kernel(const uint32_t* x, int64_t n, uint32_t* bsum) {
    const int64_t i = (int64_t)blockIdx.x * kScanT + threadIdx.x;
    uint32_t tot;
    block_scan_excl(i < n ? x[i] : 0u, tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanT) scan_bsum_kernel(uint32_t* bsum, int nb, uint32_t* total) {
    uint32_t carry = 0;
    for (int b0 = 0; b0 < nb; b0 += kScanT) {
        const int b = b0 + threadIdx.x;
        uint32_t tot;
        const uint32_t ex = block_scan_excl(b < nb ? bsum[b] : 0u, tot);
        if (b < nb) bsum[b] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void __launch_bounds__(kScanT) scan_apply_kernel(const uint32_t* x, int64_t n, const uint32_t* bsum,
                                                            uint32_t* out) {
    const int64_t i = (int64_t)blockIdx.x * kScanT + threadIdx.x;
    uint32_t tot;
    const uint32_t ex = block_scan_excl(i < n ? x[i] : 0u, tot);
    if (i < n) out[i] = bsum[blockIdx.x] + ex;
}

cudaError_t exclusive_scan_u32(const uint32_t* x, int64_t n, uint32_t* out, uint32_t* bsum, uint32_t* total,
                               cudaStream_t st) {
    const int nb = (int)((n + kScanT - 1) / kScanT);
    if (nb > 0) scan_totals_kernel<<<nb, kScanT, 0, st>>>(x, n, bsum);
    scan_bsum_kernel<<<1, kScanT, 0, st>>>(bsum, nb, total);
    if (nb > 0) scan_apply_kernel<<<nb, kScanT, 0, st>>>(x, n, bsum, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Positions of the update: the rows of each chunk of 1024 whose flag is not 0 are counted by a
// warp, and the block that finishes last scans the counts,
// first those of the map, then those of the new rows.  The compaction ranks the rows inside their
// chunk itself, so that no position per row is written (9 us for 2M + 200k flags; the scans of
// all rows took 37).
// ---------------------------------------------------------------------------------------
constexpr int kRowsPerThread = 4, kChunkRows = kMuThreads * kRowsPerThread;   // rows of a chunk: one block of the compaction

struct ScanState { uint32_t totals[2], done, pad; };

__device__ void scan_chunks(uint32_t* sum, int64_t nc, uint32_t* total) {
    constexpr int kPer = 8;
    uint32_t carry = 0;
    for (int64_t c0 = 0; c0 < nc; c0 += kMuThreads * kPer) {
        const int64_t c = c0 + threadIdx.x * kPer;
        uint32_t x[kPer], t = 0, tot;
#pragma unroll
        for (int j = 0; j < kPer; j++) x[j] = c + j < nc ? __ldcg(&sum[c + j]) : 0u;
#pragma unroll
        for (int j = 0; j < kPer; j++) t += x[j];
        uint32_t o = carry + block_scan_excl(t, tot);
#pragma unroll
        for (int j = 0; j < kPer; j++) {
            if (c + j < nc) sum[c + j] = o;
            o += x[j];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(kMuThreads) chunk_sum_kernel(const uint8_t* keep, int64_t n, const uint8_t* accept,
                                                               int64_t n_new, int64_t nc, int64_t nc_new,
                                                               uint32_t* sum, ScanState* s) {
    const int lane = threadIdx.x & 31;
    const int64_t c = (int64_t)blockIdx.x * (kMuThreads / 32) + (threadIdx.x >> 5);
    if (c < nc + nc_new) {
        const uint8_t* f = c < nc ? keep : accept;
        const int64_t m = c < nc ? n : n_new, i0 = (c < nc ? c : c - nc) * kChunkRows + lane * 8;
        uint32_t x = 0;
#pragma unroll
        for (int k = 0; k < kChunkRows / 256; k++) {
            const int64_t i = i0 + k * 256;
            if (((uintptr_t)f & 7) == 0 && i + 8 <= m) {
                const uint2 w = *reinterpret_cast<const uint2*>(f + i);
                x = __dp4a(__vsetne4(w.x, 0u), 0x01010101u, __dp4a(__vsetne4(w.y, 0u), 0x01010101u, x));
            } else {
                for (int j = 0; j < 8; j++)
                    if (i + j < m) x += f[i + j] != 0;
            }
        }
        x = warp_sum(x);
        if (lane == 0) sum[c] = x;
    }
    if (!last_block(&s->done)) return;
    scan_chunks(sum, nc, &s->totals[0]);
    scan_chunks(sum + nc, nc_new, &s->totals[1]);
}

// ---------------------------------------------------------------------------------------
// Compaction: kept rows to their positions, accepted new rows after them (with zero moments).
// Every plane is passed by its own base pointer (input stride n, new rows n_new, output n_out).
// A block takes 1024 rows of a group of 8 planes, blocks of neighbouring rows run together, and
// a thread has the 4 rows of 2 planes and their moments, 24 loads, in flight before their
// stores (which may alias later loads as far as the compiler knows, so it cannot reorder them
// itself).  Bound by DRAM: 2.9 GB of 2M rows of degree 3 and
// 200k new ones in 482 us (545 with one row of all planes to a thread, 177 streams a block).
// ---------------------------------------------------------------------------------------
constexpr int kCompactPlanes = 8, kCompactPair = 2;

__global__ void __launch_bounds__(kMuThreads) compact_kernel(MapUpdateArgs a) {
    const bool old = blockIdx.x < a.n_chunks;
    const int64_t c = old ? (int64_t)blockIdx.x : (int64_t)blockIdx.x - a.n_chunks;
    const int64_t i0 = c * kChunkRows + threadIdx.x, n = old ? a.n : a.n_new;
    const uint8_t* flag = old ? a.keep : a.accept;
    // the flags of the 4 rows in 16-bit fields (a field's sum over the block is at most 256)
    unsigned long long f = 0, tot;
#pragma unroll
    for (int k = 0; k < kRowsPerThread; k++) {
        const int64_t i = i0 + k * kMuThreads;
        if (i < n) f |= (unsigned long long)(!flag || flag[i]) << (16 * k);
    }
    const unsigned long long rank = block_scan_excl(f, tot);
    int64_t o[kRowsPerThread], base = (old ? 0 : a.n_keep) + (flag ? (int64_t)a.chunk_pos[blockIdx.x] : c * kChunkRows);
    bool on[kRowsPerThread];
#pragma unroll
    for (int k = 0; k < kRowsPerThread; k++) {
        on[k] = (f >> (16 * k)) & 0xffffu;
        o[k] = base + (int64_t)((rank >> (16 * k)) & 0xffffu);
        base += (int64_t)((tot >> (16 * k)) & 0xffffu);
    }
    const int pe = min((int)(blockIdx.y + 1) * kCompactPlanes, a.n_planes);
    for (int p0 = blockIdx.y * kCompactPlanes; p0 < pe; p0 += kCompactPair) {
        float x[kCompactPair][kRowsPerThread], m[kCompactPair][kRowsPerThread], v[kCompactPair][kRowsPerThread];
#pragma unroll
        for (int q = 0; q < kCompactPair; q++) {
            const int p = p0 + q;
            if (p >= pe) continue;
#pragma unroll
            for (int k = 0; k < kRowsPerThread; k++) {
                if (!on[k]) continue;
                const int64_t i = i0 + k * kMuThreads;
                x[q][k] = old ? a.in[p][i] : a.nw[p][i];
                m[q][k] = old ? a.m_in[p][i] : 0.f;
                v[q][k] = old ? a.v_in[p][i] : 0.f;
            }
        }
#pragma unroll
        for (int q = 0; q < kCompactPair; q++) {
            const int p = p0 + q;
            if (p >= pe) continue;
#pragma unroll
            for (int k = 0; k < kRowsPerThread; k++) {
                if (!on[k]) continue;
                a.out[p][o[k]] = x[q][k];
                a.m_out[p][o[k]] = m[q][k];
                a.v_out[p][o[k]] = v[q][k];
            }
        }
    }
    if (blockIdx.y || !a.tags_out) return;
#pragma unroll
    for (int k = 0; k < kRowsPerThread; k++) {
        const int64_t i = i0 + k * kMuThreads;
        if (on[k]) a.tags_out[o[k]] = old ? (a.tags_in ? a.tags_in[i] : 0u) : (a.new_tags ? a.new_tags[i] : 0u);
    }
}

static int64_t chunks_of(int64_t n) { return (n + kChunkRows - 1) / kChunkRows; }

static uint64_t table_slots(int64_t n) {
    uint64_t T = 8;
    while (T < (uint64_t)(2 * (n > 0 ? n : 1))) T <<= 1;
    return T;
}

size_t map_update_scratch_bytes(int64_t n_map, int64_t n_new) {
    const size_t prune = sizeof(SelectState) + sizeof(unsigned long long) * (size_t)n_map;
    const size_t dedup = sizeof(SelectState) + sizeof(uint4) * (size_t)n_map + sizeof(uint32_t) * (size_t)table_slots(n_map);
    const size_t update = sizeof(ScanState) + sizeof(uint32_t) * (size_t)(chunks_of(n_map) + chunks_of(n_new));
    size_t r = prune > dedup ? prune : dedup;
    r = r > update ? r : update;
    return ((r + 255) & ~(size_t)255) + 256;   // 256: the caller's buffer may start anywhere
}

// The scratch from its first 32-byte boundary (16-byte records; 8 slots of the table to a sector).
template <typename T> static T* scratch_base(void* scratch) {
    return reinterpret_cast<T*>(((uintptr_t)scratch + 31) & ~(uintptr_t)31);
}

cudaError_t launch_prune_plan(const float* logits, int64_t n, float thr, double max_ratio, uint8_t* keep,
                              void* scratch, unsigned long long* kept_host, cudaStream_t st) {
    SelectState* s = scratch_base<SelectState>(scratch);
    unsigned long long* list = reinterpret_cast<unsigned long long*>(s + 1);
    const unsigned long long k_max = (unsigned long long)floor(max_ratio * (double)n);
    int idx_bits = 1;
    while ((1ull << idx_bits) < (unsigned long long)n) idx_bits++;
    const int rounds = (32 + idx_bits + kDigitBits - 1) / kDigitBits;
    cudaError_t e = cudaMemsetAsync(s, 0, offsetof(SelectState, hist) + sizeof(s->hist[0]) * rounds, st);
    if (e != cudaSuccess) return e;
    if (n > 0) {
        const int64_t g = (n + kMuThreads * kCollectRows - 1) / (kMuThreads * kCollectRows);
        prune_collect_kernel<<<(unsigned)g, kMuThreads, 0, st>>>(logits, n, thr, k_max, idx_bits,
                                                                 (rounds - 1) * kDigitBits, list, keep, s);
        // blocks of the passes over the list: its length is known on the device alone
        const unsigned gl = (unsigned)(g < 2 * device_sms() ? g : 2 * device_sms());
        for (int r = 1; r < rounds; r++)
            if ((e = launch_pdl(prune_round_kernel, dim3(gl), dim3(kMuThreads), 0, st, list, r,
                                (rounds - 1 - r) * kDigitBits, s)) != cudaSuccess) return e;
        if ((e = launch_pdl(prune_mark_kernel, dim3(gl), dim3(kMuThreads), 0, st, list, idx_bits, s, keep)) != cudaSuccess)
            return e;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaMemcpyAsync(kept_host, &s->kept, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
}

cudaError_t launch_dedup_plan(const float* map_means, int64_t n, const float* new_means, int64_t nq, float radius,
                              uint8_t* accept, void* scratch, unsigned long long* accepted_host, cudaStream_t st) {
    SelectState* s = scratch_base<SelectState>(scratch);
    const uint64_t T = table_slots(n);
    uint32_t* head = reinterpret_cast<uint32_t*>(s + 1);
    uint4* node = reinterpret_cast<uint4*>(head + T);
    const double inv_cell = 1.0 / (1.001 * (double)radius);
    CellScale cs;
    cs.hi = (float)inv_cell;
    cs.lo = (float)(inv_cell - (double)cs.hi);
    const uint32_t mask = (uint32_t)(T - 1);
    cudaError_t e = cudaMemsetAsync(s, 0, offsetof(SelectState, hist), st);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(head, 0, sizeof(uint32_t) * T, st)) != cudaSuccess) return e;
    if (n > 0) {
        constexpr int kRows = kMuThreads * kBuildRows;
        hash_build_kernel<<<(unsigned)((n + kRows - 1) / kRows), kMuThreads, 0, st>>>(map_means, n, cs, mask, head, node);
    }
    if (nq > 0) {
        constexpr int kQueries = kMuThreads / 32 * kQueriesPerWarp;
        dedup_query_kernel<<<(unsigned)((nq + kQueries - 1) / kQueries), kMuThreads, 0, st>>>(
            new_means, nq, cs, radius * radius, mask, head, node, accept, s);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaMemcpyAsync(accepted_host, &s->kept, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
}

cudaError_t launch_map_scan(const uint8_t* keep, int64_t n, const uint8_t* accept, int64_t n_new, void* scratch,
                            const uint32_t** chunk_pos, uint32_t* totals_host, cudaStream_t st) {
    ScanState* s = scratch_base<ScanState>(scratch);
    uint32_t* sum = reinterpret_cast<uint32_t*>(s + 1);
    const int64_t nc = chunks_of(n), nc_new = accept ? chunks_of(n_new) : 0;
    cudaError_t e = cudaMemsetAsync(s, 0, sizeof(ScanState), st);
    if (e != cudaSuccess) return e;
    constexpr int kChunks = kMuThreads / 32;
    const int64_t g = (nc + nc_new + kChunks - 1) / kChunks;
    if (g > 0) chunk_sum_kernel<<<(unsigned)g, kMuThreads, 0, st>>>(keep, n, accept, n_new, nc, nc_new, sum, s);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *chunk_pos = sum;
    return cudaMemcpyAsync(totals_host, s->totals, sizeof(uint32_t) * 2, cudaMemcpyDeviceToHost, st);
}

cudaError_t launch_compact(MapUpdateArgs& a, cudaStream_t st) {
    a.n_chunks = (uint32_t)chunks_of(a.n);
    const int64_t g = a.n_chunks + chunks_of(a.n_new);
    if (g > 0)
        compact_kernel<<<dim3((unsigned)g, (a.n_planes + kCompactPlanes - 1) / kCompactPlanes), kMuThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace gs
