// a2-a4: tile binning, the stable LSD radix sorts and the per-tile ranges.  Tile-based
// rasterizer of §II-A / §III-C: every Gaussian is listed, in depth order, in each tile its
// alpha >= alpha_min box covers.
//
// The required order is (global tile, depth, view, Gaussian index).  Instead of one sort on
// a (tile << 32 | bits(z)) key over all pairs, the binning sorts twice:
//   1. the visible (view, Gaussian) entries -- compacted in (view, index) order -- by the
//      32-bit depth key (4 passes over the entries, about a fifth of the pairs);
//   2. the pairs, emitted from the depth-sorted entries, by the global tile id alone
//      (ceil(tile bits / 8) passes with 32-bit keys).
// Both sorts are stable, so pass 2 keeps the depth order within a tile and pass 1 keeps
// (view, index) order between equal depths: the result is the order above.
//
// Element counts are read on the device, so no host round trip is needed between the stages and
// the whole sequence can be captured in a CUDA graph.  A sort pass is one kernel: every block
// counts the digits of its run of chunks, gets the counts of the blocks before it by look-back
// (gs_internal.cuh), and scatters its chunks, ranked by warp ballots, in digit runs; the digit
// totals a pass needs are counted by the kernel before it.  With separate histogram, scan and
// scatter kernels a pass took 20 us however few the keys (launches and latency).
#include "gs_kernels.cuh"

namespace gs {

// ----------------------------------------------------------------------------------------
// Block-wide scans.  The sums of a warp are taken in 32 bits, those across warps in U.
// ----------------------------------------------------------------------------------------
template <typename U>
__device__ __forceinline__ U block_exclusive_scan_1024(uint32_t x, U* s_warp, U& total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
        U t = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : U(0);
        U ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const U y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        s_warp[lane] = ti - t;
        if (lane == 31) s_warp[32] = ti;
    }
    __syncthreads();
    total = s_warp[32];
    const U r = s_warp[w] + (inc - x);
    __syncthreads();
    return r;
}

// ----------------------------------------------------------------------------------------
// Entry compaction.  The projection leaves one bit word per view and 32 Gaussians (vis_bits,
// each view padded to whole words).  A block of kEntryThreads threads takes WPW words per warp;
// each warp writes the entries of its words, one word at a time with a lane per slot, so entries
// stay in (view, index) order.  32 words per warp on large maps; 8 (two rounds of gathers
// instead of eight) shorten the chain of dependent gathers where few blocks are resident anyway.
// The blocks' first positions come from a look-back scan while the blocks are about one wave
// (9 us in all at 10k slots, 25 us with separate count and scan kernels), else from a count
// kernel whose last block scans the totals: a look-back stalls each further wave of blocks (58
// against 49 us at 16M slots).
// ----------------------------------------------------------------------------------------
constexpr int kEntryThreads = 256;
constexpr int kEntryWarps = kEntryThreads / 32;
static_assert(kEntryMinWords == 8 * kEntryWarps && kEntryThreads == 32 * kEntryWarps, "words per block of the short form");

// Entries of every block's words (blocks of `wpb` words), and their exclusive scan by the last
// block to finish; the total goes to the counters.  A thread counts four words.
constexpr int kCountWords = 4 * kEntryThreads;

__global__ void __launch_bounds__(kEntryThreads) entry_count_kernel(BinArgs a, int64_t n_words, int wpb, int n_blocks) {
    pdl_begin();
    constexpr int GT = kEntryMinWords / 4;   // threads per kEntryMinWords words
    __shared__ uint32_t s[kEntryThreads / GT], s_w[33];
    __shared__ bool last;
    if (a.counters->status != 0) return;
    const int64_t word = (int64_t)blockIdx.x * kCountWords + 4 * threadIdx.x;
    uint32_t sum = 0;
    if (word + 3 < n_words) {
        const uint4 q = *reinterpret_cast<const uint4*>(a.vis_bits + word);
        sum = __popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w);
    } else {
        for (int64_t k = word; k < n_words; k++) sum += __popc(a.vis_bits[k]);
    }
#pragma unroll
    for (int o = GT / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (threadIdx.x % GT == 0) s[threadIdx.x / GT] = sum;
    __syncthreads();
    const int per = kCountWords / wpb, groups = wpb / kEntryMinWords;   // totals of this block; groups of each
    if ((int)threadIdx.x < per) {
        uint32_t t = 0;
        for (int k = 0; k < groups; k++) t += s[threadIdx.x * groups + k];
        const int64_t b = (int64_t)blockIdx.x * per + threadIdx.x;
        if (b < n_blocks) a.entry_scan[b] = t;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&a.tickets[0], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    unsigned long long carry = 0;
    constexpr int PT = 8;   // totals per thread and round
    for (int base = 0; base < n_blocks; base += PT * kEntryThreads) {
        uint32_t x[PT], sum8 = 0, tot;
#pragma unroll
        for (int k = 0; k < PT; k++) {
            const int j = base + (int)threadIdx.x * PT + k;
            x[k] = j < n_blocks ? (uint32_t)__ldcg(&a.entry_scan[j]) : 0u;
            sum8 += x[k];
        }
        unsigned long long run = carry + block_exclusive_scan_1024(sum8, s_w, tot);
#pragma unroll
        for (int k = 0; k < PT; k++) {
            const int j = base + (int)threadIdx.x * PT + k;
            if (j < n_blocks) a.entry_scan[j] = run;
            run += x[k];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        a.counters->n_entries = carry;
        a.counters->n_entries32 = (uint32_t)carry;
    }
}

template <int WPW, bool LOOKBACK>
__global__ void __launch_bounds__(kEntryThreads, 4) entry_compact_kernel(BinArgs a, int64_t n_words) {
    pdl_begin();
    constexpr int WPB = WPW * kEntryWarps;   // words per block
    __shared__ uint32_t s[33];
    __shared__ uint32_t s_off[WPB], s_word[WPB];
    __shared__ uint32_t s_base, s_chunk;
    __shared__ uint32_t s_hist[kSortBins];
    __shared__ bool s_ok;
    static_assert(kEntryThreads == kSortBins, "a thread per digit");
    if (!LOOKBACK && a.counters->status != 0) return;   // (this form does not set it)
    s_hist[threadIdx.x] = 0;
    if (LOOKBACK) {
        if (threadIdx.x == 0) s_chunk = lb_ticket(&a.tickets[0], a.counters);
        __syncthreads();
        if (s_chunk == kLbStop) return;
    }
    const int64_t chunk = LOOKBACK ? s_chunk : blockIdx.x, word = chunk * WPB + threadIdx.x;
    const uint32_t b = (int)threadIdx.x < WPB && word < n_words ? a.vis_bits[word] : 0u;
    const uint32_t nw = (uint32_t)((a.n + 31) >> 5);   // words per view
    uint32_t tot;
    const uint32_t off = block_exclusive_scan_1024((uint32_t)__popc(b), s, tot);
    if (!LOOKBACK) {
        if (threadIdx.x == 0) {
            s_base = (uint32_t)a.entry_scan[chunk];
            s_ok = true;
        }
    } else if (threadIdx.x < 32) {
        bool ok = true;
        const unsigned long long before = lb_scan_warp(a.entry_scan, chunk, tot, a.counters, a.spin, ok);
        if (threadIdx.x == 0) {
            s_base = (uint32_t)before;
            s_ok = ok;
            if (ok && chunk == gridDim.x - 1) {
                a.counters->n_entries = before + tot;
                a.counters->n_entries32 = (uint32_t)(before + tot);
            }
        }
    }
    if ((int)threadIdx.x < WPB) {
        s_off[threadIdx.x] = off;
        s_word[threadIdx.x] = b;
    }
    __syncthreads();
    if (!s_ok) return;
    const uint32_t base = s_base;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t ltm;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(ltm));
    // four bit words per iteration: their record gathers are issued together
    for (int k = 0; k < WPW; k += 4) {
        bool hit[4];
        float4 g0[4];
        int grx[4], gry[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int lw = w * WPW + k + u;
            hit[u] = (s_word[lw] >> lane) & 1u;
            const uint32_t gw = (uint32_t)(chunk * WPB) + lw;   // < V * nw
            const uint32_t v = gw / nw;
            const uint32_t idx = v * (uint32_t)a.n + (gw - v * nw) * 32 + lane;
            if (hit[u]) {
                g0[u] = __ldg(a.proj + 3 * (size_t)idx);
                grx[u] = __float_as_int(__ldg(a.proj + 3 * (size_t)idx + 1).w);
                gry[u] = __float_as_int(__ldg(a.proj + 3 * (size_t)idx + 2).w);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int lw = w * WPW + k + u;
            const uint32_t bw = s_word[lw];
            if (hit[u]) {
                const uint32_t pos = base + s_off[lw] + (uint32_t)__popc(bw & ltm);
                const uint32_t gw = (uint32_t)(chunk * WPB) + lw;
                const uint32_t v = gw / nw;
                const uint32_t idx = v * (uint32_t)a.n + (gw - v * nw) * 32 + lane;
                const float4 r0 = g0[u];
                const int rx = grx[u];
                const int ry = gry[u];
                const View& V = a.views[v];
                // the rectangle the projection found non-empty
                int xa = 0, xb = 0, ya = 0, yb = 0;
                tile_span(r0.x, rx, a.tile, V.tiles_x, xa, xb);
                tile_span(r0.y, ry, a.tile, V.tiles_y, ya, yb);
                const uint32_t zk = __float_as_uint(r0.z);   // z > 0: bits are monotone
                a.ekeys[pos] = zk;
                atomicAdd(&s_hist[zk & 255u], 1u);   // the depth sort's first digit
                a.evals[pos] = pos;
                a.entries[pos] = idx;
                a.erect[pos] = make_uint4((uint32_t)(V.tile_off + ya * V.tiles_x + xa),
                                          (uint32_t)(xb - xa + 1) | ((uint32_t)(yb - ya + 1) << 16), idx, 0u);
            }
        }
    }
    __syncthreads();
    if (s_hist[threadIdx.x]) atomicAdd(&a.ehist[threadIdx.x], s_hist[threadIdx.x]);
}

size_t entry_scan_words(int64_t n, int n_views) {
    return (size_t)(((int64_t)n_views * ((n + 31) >> 5) + kEntryMinWords - 1) / kEntryMinWords) + 1;
}

cudaError_t launch_entries(const BinArgs& a, cudaStream_t st) {
    const int64_t n_words = (int64_t)a.n_views * ((a.n + 31) >> 5);
    if (n_words == 0) return cudaSuccess;
    // the short form while its blocks fit the device a few times over (4 resident per SM)
    const int64_t small = (n_words + kEntryMinWords - 1) / kEntryMinWords, sms = device_sms();
    if (small <= 4 * sms) {
        launch_pdl(entry_compact_kernel<8, true>, (unsigned)small, kEntryThreads, 0, st, a, n_words);
        return cudaGetLastError();
    }
    const int wpb = small <= 16 * sms ? kEntryMinWords : 32 * kEntryWarps;
    const int nb = (int)((n_words + wpb - 1) / wpb);
    launch_pdl(entry_count_kernel, (unsigned)((n_words + kCountWords - 1) / kCountWords), kEntryThreads, 0, st, a, n_words, wpb, nb);
    if (wpb == kEntryMinWords)
        launch_pdl(entry_compact_kernel<8, false>, nb, kEntryThreads, 0, st, a, n_words);
    else
        launch_pdl(entry_compact_kernel<32, false>, nb, kEntryThreads, 0, st, a, n_words);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Pair emission from the depth-sorted entries: the tile counts of their rectangles, taken
// in that order, are scanned into pair offsets (total = pair count), then each entry writes
// one (global tile id, view * n + index) pair per covered tile, tiles in row-major order.
// The rectangles and indices are read from the compact per-entry records of the compaction (16
// bytes, one gather an entry), not from the projected records.
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t rect_count(uint2 r) { return (r.y & 0xFFFFu) * (r.y >> 16); }

// Pair offsets of the depth-sorted entries (poff[e] = pairs of the entries before e), for every
// output chunk of kEmitChunk pairs the entry holding its first pair, and each entry's tile
// rectangle and index in depth order (srt), which the emission then reads without the gather
// through the sorted compact indices.  The entry count is known only on the device: resident
// blocks take chunks of kPairScanChunk entries in turn.
__global__ void __launch_bounds__(kPairScanThreads) pair_offsets_kernel(BinArgs a) {
    pdl_begin();
    __shared__ unsigned long long s[33], s_base;
    __shared__ uint32_t s_chunk;
    __shared__ bool s_ok;
    const int64_t E = (int64_t)a.counters->n_entries, VN = (int64_t)a.n_views * a.n;
    const int64_t n_chunks = (E + kPairScanChunk - 1) / kPairScanChunk;
    const uint64_t emit_chunks = ((uint64_t)a.max_pairs + kEmitChunk - 1) / kEmitChunk;
    for (;;) {
        if (threadIdx.x == 0) s_chunk = lb_ticket(&a.tickets[1], a.counters);
        __syncthreads();
        const int64_t ch = s_chunk;
        if (ch >= n_chunks) return;   // (kLbStop is past every chunk)
        // thread t takes entries 4 t .. 4 t + 3 of the chunk
        const int64_t e0 = ch * kPairScanChunk + (int64_t)threadIdx.x * kPairScanItems;
        uint32_t c[kPairScanItems], t[kPairScanItems], sum = 0;
        if (e0 + kPairScanItems <= E) {
            const uint4 q = *reinterpret_cast<const uint4*>(a.sorted_evals + e0);
            c[0] = q.x; c[1] = q.y; c[2] = q.z; c[3] = q.w;
        } else {
#pragma unroll
            for (int k = 0; k < kPairScanItems; k++) c[k] = e0 + k < E ? a.sorted_evals[e0 + k] : 0u;
        }
        uint4 r[kPairScanItems];   // one 16-byte gather an entry
#pragma unroll
        for (int k = 0; k < kPairScanItems; k++) r[k] = e0 + k < E ? a.erect[c[k]] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int k = 0; k < kPairScanItems; k++) {
            t[k] = rect_count(make_uint2(r[k].x, r[k].y));
            sum += t[k];
            if (e0 + k < E) {
                a.srt[e0 + k] = r[k].x;
                a.srt[VN + e0 + k] = r[k].y;
                a.srt[2 * VN + e0 + k] = r[k].z;
            }
        }
        // an entry covers at most (16384 / 8)^2 = 2^22 tiles: a warp's 128 entries fit 32 bits, the
        // chunk's 2048 do not
        unsigned long long tot;
        const unsigned long long local = block_exclusive_scan_1024(sum, s, tot);
        if (threadIdx.x < 32) {
            bool ok = true;
            const unsigned long long before = lb_scan_warp(a.pair_scan, ch, tot, a.counters, a.spin, ok);
            if (threadIdx.x == 0) {
                s_base = before;
                s_ok = ok;
                if (ok && ch == n_chunks - 1) {
                    a.counters->n_pairs = before + tot;
                    if (before + tot > (unsigned long long)a.max_pairs) set_status(a.counters, GS_ERR_CAPACITY);
                }
            }
        }
        __syncthreads();
        if (!s_ok) return;
        unsigned long long off = s_base + local;
#pragma unroll
        for (int k = 0; k < kPairScanItems; k++) {
            if (e0 + k < E) {
                a.poff[e0 + k] = (uint32_t)off;
                // chunk starts c * kEmitChunk inside [off, off + t), of the chunks that exist
                for (uint64_t m = (off + kEmitChunk - 1) / kEmitChunk; m < emit_chunks && m * kEmitChunk < off + t[k]; m++)
                    a.chunk_first[m] = (uint32_t)(e0 + k);
            }
            off += t[k];
        }
    }
}

size_t pair_scan_words(int64_t n, int n_views) { return (size_t)(((int64_t)n_views * n) / kPairScanChunk) + 2; }

// Adds one to bin d of a shared histogram for every valid lane: once, with the count, where the
// valid lanes share the digit -- the rule for a depth's or a tile id's upper digits -- instead of
// 32 serial additions to one address.  All lanes of the warp call it.
// hist_add_all: every lane is valid.
__device__ __forceinline__ void hist_add_all(uint32_t* h, uint32_t d) {
    const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
    if (__all_sync(0xffffffffu, d == d0)) {
        if ((threadIdx.x & 31) == 0) atomicAdd(&h[d0], 32u);
    } else {
        atomicAdd(&h[d], 1u);
    }
}
__device__ __forceinline__ void hist_add(uint32_t* h, uint32_t d, bool valid) {
    const uint32_t v = __ballot_sync(0xffffffffu, valid);
    if (!v) return;
    const int lead = __ffs(v) - 1;
    const uint32_t d0 = __shfl_sync(0xffffffffu, d, lead);
    if (__all_sync(0xffffffffu, !valid || d == d0)) {
        if ((int)(threadIdx.x & 31) == lead) atomicAdd(&h[d0], (uint32_t)__popc(v));
    } else if (valid) {
        atomicAdd(&h[d], 1u);
    }
}

// Emission balanced over the output: a block takes a chunk of kEmitChunk consecutive pairs,
// stages the entries they come from (at most kEmitChunk + 1) with their tile rectangles in
// shared memory, marks the slot where each entry starts, and finds every slot's entry with a
// running maximum over the chunk.  A few entries
// with very many tiles no longer serialise on one warp.
__global__ void __launch_bounds__(kEmitThreads) pair_emit_kernel(BinArgs a) {
    pdl_begin();
    static_assert(kEmitChunk == 8 * kEmitThreads, "each thread owns 8 consecutive slots of the chunk");
    __shared__ uint32_t s_off[kEmitChunk + 1], s_t0[kEmitChunk + 1], s_id[kEmitChunk + 1];
    __shared__ uint16_t s_wx[kEmitChunk + 1], s_tx[kEmitChunk + 1];
    __shared__ __align__(16) uint16_t s_own[kEmitChunk];   // slot -> local entry index
    __shared__ uint32_t s_wmax[kEmitThreads / 32];
    __shared__ uint16_t s_view_tx[GS_MAX_VIEWS];   // tiles per row of each view
    __shared__ uint32_t s_hist[kSortMaxBins];      // the tile sort's first digit
    if (a.counters->status != 0) return;
    for (int k = threadIdx.x; k < kSortMaxBins; k += kEmitThreads) s_hist[k] = 0;
    for (int v = threadIdx.x; v < a.n_views; v += blockDim.x) s_view_tx[v] = (uint16_t)a.views[v].tiles_x;
    const uint64_t P = a.counters->n_pairs;
    const int64_t E = (int64_t)a.counters->n_entries;
    const uint64_t n_chunks = (P + kEmitChunk - 1) / kEmitChunk;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // the chunks in turn over the grid (a resident grid: the pair count is known only here)
    for (uint64_t c = blockIdx.x; c < n_chunks; c += gridDim.x) {
        const uint64_t p0 = c * kEmitChunk, p1 = p0 + kEmitChunk < P ? p0 + kEmitChunk : P;
        const int64_t e0 = a.chunk_first[c];
        const int64_t e1 = c + 1 < n_chunks ? (int64_t)a.chunk_first[c + 1] : E - 1;
        const int ne = (int)(e1 - e0 + 1);   // <= kEmitChunk + 1: every entry has >= 1 pair
        for (int i = threadIdx.x; i < kEmitChunk; i += blockDim.x) s_own[i] = 0;
        __syncthreads();
        const int64_t VN = (int64_t)a.n_views * a.n;
        for (int j = threadIdx.x; j < ne; j += blockDim.x) {
            const int64_t e = e0 + j;
            const uint32_t idx = a.srt[2 * VN + e];
            const uint2 r = make_uint2(a.srt[e], a.srt[VN + e]);
            const uint32_t off = a.poff[e];
            s_off[j] = off;
            s_t0[j] = r.x;
            s_id[j] = idx;
            s_wx[j] = (uint16_t)(r.y & 0xFFFFu);
            s_tx[j] = s_view_tx[idx / (uint32_t)a.n];
            // the entry's first pair slot in this chunk (entry 0 starts at or before p0)
            if (j > 0 && off < p1) s_own[off - p0] = (uint16_t)j;
        }
        __syncthreads();
        // slot owner = the last entry starting at or before the slot: a running maximum over
        // the chunk (8 slots per thread, then warp and block maxima of the thread maxima)
        uint32_t own[8], mx = 0;
        {
            const uint4 q = *reinterpret_cast<const uint4*>(s_own + 8 * threadIdx.x);
            const uint32_t wd[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int h = 0; h < 4; h++) {
                mx = max(mx, wd[h] & 0xFFFFu);
                own[2 * h] = mx;
                mx = max(mx, wd[h] >> 16);
                own[2 * h + 1] = mx;
            }
        }
        uint32_t inc = mx;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc = max(inc, y);
        }
        if (lane == 31) s_wmax[w] = inc;
        uint32_t before = __shfl_up_sync(0xffffffffu, inc, 1);
        if (lane == 0) before = 0;
        __syncthreads();
        for (int ww = 0; ww < w; ww++) before = max(before, s_wmax[ww]);
        __syncthreads();   // every thread has read its slots
#pragma unroll
        for (int h = 0; h < 8; h++) s_own[8 * threadIdx.x + h] = (uint16_t)max(before, own[h]);
        __syncthreads();
        // coalesced writes: thread t writes slots t, t + 256, ...
        for (uint64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
            const uint32_t j = s_own[p - p0];
            const uint32_t kk = (uint32_t)p - s_off[j], wx = s_wx[j];
            const uint32_t ty = kk / wx, tx = kk - ty * wx;
            const uint32_t tile = s_t0[j] + ty * (uint32_t)s_tx[j] + tx;
            a.pkeys[p] = tile;
            a.pvals[p] = s_id[j];
            if (a.phist_mask) atomicAdd(&s_hist[tile & a.phist_mask], 1u);
        }
        __syncthreads();
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kSortMaxBins; k += kEmitThreads)
        if (s_hist[k]) atomicAdd(&a.phist[k], s_hist[k]);
}

// Blocks of `kernel` resident on the device at once (occupancy times SMs), kept per device.
template <class Kernel>
static int resident_grid(int (&cache)[kMaxDevices], Kernel kernel, int threads, size_t smem = 0) {
    const int d = current_device();
    if (d >= 0 && cache[d] > 0) return cache[d];
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int g = per_sm * device_sms();
    if (d >= 0) cache[d] = g;
    return g;
}

cudaError_t launch_emit(const BinArgs& a, cudaStream_t st) {
    static int g_offsets[kMaxDevices] = {}, g_emit[kMaxDevices] = {};
    const int64_t nb = ((int64_t)a.n_views * a.n + kPairScanChunk - 1) / kPairScanChunk;   // at most
    if (nb > 0) {
        const int64_t g = resident_grid(g_offsets, pair_offsets_kernel, kPairScanThreads);
        launch_pdl(pair_offsets_kernel, (unsigned)(g < nb ? g : nb), kPairScanThreads, 0, st, a);
    }
    // one chunk of kEmitChunk pairs per block and turn; the pair count is known only on the
    // device, so the grid is the resident one (capped by the capacity's chunks)
    const int64_t emit_chunks = (a.max_pairs + kEmitChunk - 1) / kEmitChunk;
    const int64_t ge = resident_grid(g_emit, pair_emit_kernel, kEmitThreads);
    const int64_t emit_grid = emit_chunks < ge ? emit_chunks : ge;
    launch_pdl(pair_emit_kernel, (unsigned)(emit_grid > 0 ? emit_grid : 1), kEmitThreads, 0, st, a);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Radix sort with BITS-bit digits (8 or 9), keys K = uint32_t or unsigned long long.
// ----------------------------------------------------------------------------------------
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kItemsPerWarp = kSortChunk / kSortWarps;   // 256
constexpr int kHistThreads = 512;
constexpr int kHistItems = kSortChunk / kHistThreads;    // 8

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// The pass's digit: BITS bits of the key from `shift`, restricted by the pass's digit mask (a
// sort by the low b bits ends with a pass whose mask keeps only the bits below b).
template <int BITS, typename K>
__device__ __forceinline__ uint32_t digit_of(K k, int shift, uint32_t mask) {
    return (uint32_t)(k >> shift) & ((1u << BITS) - 1u) & mask;
}

// Digit counts of one pass of 8-bit digits (a sort whose keys no kernel of the library counts).
__global__ void __launch_bounds__(kHistThreads) sort_count_kernel(SortArgs a, int shift) {
    __shared__ uint32_t h[kSortBins];
    if (a.counters->status != 0) return;
    const int64_t count = (int64_t)*a.count;
    for (int t = threadIdx.x; t < kSortBins; t += kHistThreads) h[t] = 0;
    __syncthreads();
    const unsigned long long* keys = static_cast<const unsigned long long*>(a.keys[0]);
    for (int64_t base = (int64_t)blockIdx.x * kSortChunk; base < count; base += (int64_t)gridDim.x * kSortChunk) {
        unsigned long long k[kHistItems];
#pragma unroll
        for (int j = 0; j < kHistItems; j++) {
            const int64_t i = base + (int64_t)j * kHistThreads + threadIdx.x;
            k[j] = i < count ? keys[i] : 0ull;
        }
#pragma unroll
        for (int j = 0; j < kHistItems; j++)
            hist_add(h, (uint32_t)(k[j] >> shift) & 255u & a.digit_mask,
                     base + (int64_t)j * kHistThreads + threadIdx.x < count);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kSortBins; t += kHistThreads)
        if (h[t]) atomicAdd(&a.hist[t], h[t]);
}

// Digit-indexed shared arrays are stored at dix(d) = d with its low 5 bits XORed with the next
// ones: digits 32 m apart (tile ids one or more tile rows apart, which a warp step often holds)
// then fall in different banks.  A bijection on [0, 2^BITS).
__device__ __forceinline__ int dix(uint32_t d) { return (int)(d ^ ((d >> 5) & 31u)); }

// Chunk position k is stored at k + k / 32: ranked keys of one warp step often land at a
// fixed stride (consecutive digits with similar counts), which without the skew would hit the
// same few shared-memory banks.
__device__ __forceinline__ int skew(int k) { return k + (k >> 5); }

template <typename K, int BITS>
struct SortSmem {
    static constexpr int BINS = 1 << BITS;
    K keys[kSortChunk + kSortChunk / 32];
    uint32_t vals[kSortChunk + kSortChunk / 32];
    uint32_t wcnt[kSortWarps][BINS];
    uint32_t run[BINS];      // next output position of each digit
    uint32_t gpos[BINS];     // the same for the chunk being written, less cstart
    uint32_t cstart[BINS];
    uint32_t next[kSortMaxBins];   // digit counts: of the block's run, then of the next pass
    uint32_t scan_w[33];
    uint32_t ticket;
};

// Exclusive scan of DPT consecutive values per thread over the block (kSortThreads threads);
// out[q] receives the prefix of value q.
template <int DPT>
__device__ __forceinline__ void block_exclusive_scan_dpt(const uint32_t (&x)[DPT], uint32_t (&out)[DPT],
                                                         uint32_t* scan_w) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t sum = 0;
#pragma unroll
    for (int q = 0; q < DPT; q++) sum += x[q];
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) scan_w[w] = inc;
    __syncthreads();
    if (w == 0) {
        const uint32_t t0 = lane < kSortWarps ? scan_w[lane] : 0u;
        uint32_t ti = t0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        if (lane < kSortWarps) scan_w[lane] = ti - t0;
    }
    __syncthreads();
    uint32_t r = scan_w[w] + inc - sum;
#pragma unroll
    for (int q = 0; q < DPT; q++) {
        out[q] = r;
        r += x[q];
    }
    __syncthreads();
}

constexpr int kLbBatch = 8;   // look-back words loaded at a time

// Sum of the words col[j << bits], j = last, last - 1, ..., first, up to and including the first
// that holds an inclusive prefix (state 2).  ok is cleared after `limit` polls of words not there.
template <typename W>
__device__ __forceinline__ uint32_t lb_sum(const W* col, int bits, int64_t last, int64_t first, uint32_t tag, int limit,
                                           bool& ok) {
    uint32_t sum = 0;
    int spin = 0;
    for (int64_t j = last; j >= first && ok; j -= kLbBatch) {
        W wd[kLbBatch];
#pragma unroll
        for (int u = 0; u < kLbBatch; u++) wd[u] = j - u >= first ? lb_load(col + ((size_t)(j - u) << bits)) : (W)0;
        bool full = false;
#pragma unroll
        for (int u = 0; u < kLbBatch; u++) {
            if (full || j - u < first || !ok) continue;
            uint32_t st = lb_state(wd[u], tag);
            while (st == 0) {
                if (++spin > limit) {
                    ok = false;
                    break;
                }
                wd[u] = lb_load(col + ((size_t)(j - u) << bits));
                st = lb_state(wd[u], tag);
            }
            if (!ok) continue;
            sum += (uint32_t)lb_value(wd[u]);
            full = st == 2;
        }
        if (full) break;
    }
    return sum;
}

// Digit counts of the first `lo` keys into run, by the whole block.  A function of its own: inline it
// made each pass half a microsecond longer (1499 and 1496 us, rendering 2M Gaussians in 8 views).
template <typename K, int BITS>
__device__ __noinline__ void recount(uint32_t* run, const K* keys, int64_t lo, int shift, uint32_t mask) {
    for (int d = threadIdx.x; d < (1 << BITS); d += kSortThreads) run[d] = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < lo; i += kSortThreads) atomicAdd(&run[digit_of<BITS>(keys[i], shift, mask)], 1u);
    __syncthreads();
}

// One pass.  Block t (in ticket order, so that the blocks it waits for are running) owns a
// contiguous run of chunks.  It counts the run's digits and publishes them, ranks its first chunk,
// and then sums the counts of the blocks before it (a thread per digit), by when those mostly are
// there; then it scatters its chunks one after another.  Blocks form groups of kSortGroup whose
// last block publishes the group's counts and then its inclusive prefix, so that a block reads
// at most 15 + grid / 16 words a digit: reading the words of every block in flight instead took
// most of the pass.  At 7k / 356k / 1.9M entries a pass takes 9 / 12 / 27 us, at 8.7M pairs 77 to 90
// (separate kernels: 20 / 26 / 38, 76).  (Chunks dealt out one by one, each with a look-back of its own, lose at large
// counts: a look-back step is about a microsecond across the two dies, 85 against 60 us a pass at
// 8.7M pairs.)  The next pass's digits are counted on the way out.  Every wait is bounded, and a
// block whose wait gives up counts the keys before its run itself, so that a pass has one result:
// the callers that sort without a status word to report would have nothing to tell a failure by.
template <typename K, int BITS>
__global__ void __launch_bounds__(kSortThreads, kSortBlocksPerSM)
    sort_pass_kernel(SortArgs a, int in_buf, int shift, int pass, int next_shift, uint32_t next_mask) {
    pdl_begin();
    constexpr int BINS = 1 << BITS;
    constexpr int DPT = (BINS + kSortThreads - 1) / kSortThreads;   // digits per thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SortSmem<K, BITS>& S = *reinterpret_cast<SortSmem<K, BITS>*>(smem_raw);
    if (a.counters->status != 0) return;
    const int64_t count = (int64_t)*a.count, nch = sort_chunks(count);
    if (threadIdx.x == 0) S.ticket = atomicAdd(&a.tickets[pass], 1u);
    for (int t = threadIdx.x; t < kSortMaxBins; t += kSortThreads) S.next[t] = 0;
    // (selects, not a runtime index into the parameter arrays, which would go to local memory)
    const K* kin = static_cast<const K*>(in_buf ? a.keys[1] : a.keys[0]);
    const uint32_t* vin = in_buf ? a.vals[1] : a.vals[0];
    K* kout = static_cast<K*>(in_buf ? a.keys[0] : a.keys[1]);
    uint32_t* vout = in_buf ? a.vals[0] : a.vals[1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int d0 = threadIdx.x * DPT;   // this thread's digits d0 .. d0 + DPT - 1 (if below BINS)
    const uint32_t tag = a.tag + (uint32_t)pass;
    uint32_t dbase[DPT];                // first output position of each digit
    {
        uint32_t x[DPT];
#pragma unroll
        for (int q = 0; q < DPT; q++) x[q] = d0 + q < BINS ? a.hist[pass * kSortMaxBins + d0 + q] : 0u;
        block_exclusive_scan_dpt<DPT>(x, dbase, S.scan_w);   // (begins and ends with barriers)
    }
    const int64_t blocks = nch < gridDim.x ? nch : gridDim.x, t = S.ticket;
    if (t >= blocks) return;   // (the same for the whole block)
    const int64_t lo = nch * t / blocks * kSortChunk, end = nch * (t + 1) / blocks * kSortChunk, hi = end < count ? end : count;
    const uint32_t ltm = lanemask_lt();
    K key[kSortItems];
    uint32_t val[kSortItems];
    auto load = [&](int64_t base, int m) {
        // all loads first: the chunk's reads are in flight together
#pragma unroll
        for (int j = 0; j < kSortItems; j++) {
            const int item = w * kItemsPerWarp + j * 32 + lane;
            const bool valid = item < m;
            key[j] = valid ? kin[base + item] : (K)0;
            val[j] = valid ? vin[base + item] : 0u;
        }
    };
    auto chunk_size = [&](int64_t base) { return (int)(hi - base < kSortChunk ? hi - base : kSortChunk); };
    // the digits of the run, two chunks' keys in flight at a time (of a single chunk, from the
    // registers it is ranked from below)
    if (hi - lo > kSortChunk) {
        for (int64_t base = lo; base < hi; base += 2 * kSortChunk) {
            K k[2][kSortItems];
#pragma unroll
            for (int j = 0; j < 2 * kSortItems; j++) {
                const int64_t i = base + (int64_t)j * kSortThreads + threadIdx.x;
                k[j / kSortItems][j % kSortItems] = i < hi ? kin[i] : (K)0;
            }
            if (base + 2 * kSortChunk <= hi) {
#pragma unroll
                for (int j = 0; j < 2 * kSortItems; j++)
                    hist_add_all(S.next, digit_of<BITS>(k[j / kSortItems][j % kSortItems], shift, a.digit_mask));
            } else {
#pragma unroll
                for (int j = 0; j < 2 * kSortItems; j++)
                    hist_add(S.next, digit_of<BITS>(k[j / kSortItems][j % kSortItems], shift, a.digit_mask),
                             base + (int64_t)j * kSortThreads + threadIdx.x < hi);
            }
        }
    }
    load(lo, chunk_size(lo));
    if (hi - lo <= kSortChunk) {
#pragma unroll
        for (int j = 0; j < kSortItems; j++)
            hist_add(S.next, digit_of<BITS>(key[j], shift, a.digit_mask), w * kItemsPerWarp + j * 32 + lane < chunk_size(lo));
    }
    __syncthreads();
    lbword* const groups = a.lookback;
    uint32_t* const words = reinterpret_cast<uint32_t*>(groups + kSortGroupBytes / sizeof(lbword));
    uint32_t mine[DPT];
#pragma unroll
    for (int q = 0; q < DPT; q++) {
        if (d0 + q >= BINS) continue;
        mine[q] = S.next[d0 + q];
        lb_store(words + ((size_t)t << BITS) + d0 + q, tag, 1, mine[q]);
        S.next[d0 + q] = 0;
    }
    for (int64_t base = lo; base < hi; base += kSortChunk) {
        const int m = chunk_size(base);
        for (int k = threadIdx.x; k < kSortWarps * BINS; k += kSortThreads) (&S.wcnt[0][0])[k] = 0;
        if (base != lo) load(base, m);
        uint32_t rank[kSortItems / 2];   // two 16-bit ranks a word
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSortItems; j++) {
            const int item = w * kItemsPerWarp + j * 32 + lane;
            const bool valid = item < m;
            const uint32_t dg = valid ? digit_of<BITS>(key[j], shift, a.digit_mask) : (uint32_t)BINS;
            // lanes holding the same digit: one ballot per digit bit, and one for validity (a
            // fixed cost; __match_any_sync is slower when a warp holds many distinct digits)
            uint32_t peers = __ballot_sync(0xffffffffu, valid);
            if (!valid) peers = ~peers;
#pragma unroll
            for (int bit = 0; bit < BITS; bit++) {
                const bool set = (dg >> bit) & 1u;
                const uint32_t bb = __ballot_sync(0xffffffffu, set);
                peers &= set ? bb : ~bb;
            }
            uint32_t r = __popc(peers & ltm);
            if (valid) r += S.wcnt[w][dix(dg)];
            __syncwarp();
            if (valid && lane == 31 - __clz(peers)) S.wcnt[w][dix(dg)] += __popc(peers);
            __syncwarp();
            rank[j / 2] = j % 2 ? rank[j / 2] | r << 16 : r;
        }
        __syncthreads();
        // per digit: prefix over warps and the chunk total, then the chunk's digit starts
        uint32_t tot[DPT], cs[DPT];
#pragma unroll
        for (int q = 0; q < DPT; q++) {
            tot[q] = 0;
            if (d0 + q >= BINS) continue;
#pragma unroll
            for (int ww = 0; ww < kSortWarps; ww++) {
                const uint32_t c = S.wcnt[ww][dix(d0 + q)];
                S.wcnt[ww][dix(d0 + q)] = tot[q];
                tot[q] += c;
            }
        }
        block_exclusive_scan_dpt<DPT>(tot, cs, S.scan_w);
#pragma unroll
        for (int q = 0; q < DPT; q++)
            if (d0 + q < BINS) S.cstart[dix(d0 + q)] = cs[q];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSortItems; j++) {
            const int item = w * kItemsPerWarp + j * 32 + lane;
            if (item < m) {
                const uint32_t dg = digit_of<BITS>(key[j], shift, a.digit_mask);
                const int pos = skew((int)(S.cstart[dix(dg)] + S.wcnt[w][dix(dg)] + (rank[j / 2] >> (16 * (j % 2)) & 0xFFFFu)));
                S.keys[pos] = key[j];
                S.vals[pos] = val[j];
            }
        }
        if (base == lo) {
            // counts of the blocks before this one: those of its group, then the groups before
            const int64_t g = t / kSortGroup;
            const bool last = t % kSortGroup == kSortGroup - 1;
            bool ok = a.spin > 0;
#pragma unroll
            for (int q = 0; q < DPT; q++) {
                const int d = d0 + q;
                if (d >= BINS) continue;
                uint32_t before = lb_sum(words + d, BITS, t - 1, g * kSortGroup, tag, a.spin, ok);
                if (last && ok)
                    lb_store(groups + ((size_t)g << BITS) + d, tag, g == 0 ? 2u : 1u, (unsigned long long)(before + mine[q]));
                if (g > 0 && ok) {
                    before += lb_sum(groups + d, BITS, g - 1, 0, tag, a.spin, ok);
                    if (last && ok) lb_store(groups + ((size_t)g << BITS) + d, tag, 2, (unsigned long long)(before + mine[q]));
                }
                S.run[d] = dbase[q] + before;
            }
            // a wait that gives up: the counts from the keys before the run, which the pass only reads
            if (__builtin_expect(__syncthreads_or(!ok), 0)) {
                recount<K, BITS>(S.run, kin, lo, shift, a.digit_mask);
#pragma unroll
                for (int q = 0; q < DPT; q++) {
                    const int d = d0 + q;
                    if (d >= BINS) continue;
                    if (last) lb_store(groups + ((size_t)g << BITS) + d, tag, 2, (unsigned long long)(S.run[d] + mine[q]));
                    S.run[d] += dbase[q];
                }
            }
        }
#pragma unroll
        for (int q = 0; q < DPT; q++) {
            if (d0 + q >= BINS) continue;
            const uint32_t r = S.run[d0 + q];
            S.gpos[dix(d0 + q)] = r - cs[q];
            S.run[d0 + q] = r + tot[q];
        }
        __syncthreads();
        auto put = [&](int k) {
            const K kk = S.keys[skew(k)];
            const uint32_t g = S.gpos[dix(digit_of<BITS>(kk, shift, a.digit_mask))] + (uint32_t)k;   // (mod 2^32)
            kout[g] = kk;
            vout[g] = S.vals[skew(k)];
            return kk;
        };
        if (m == kSortChunk) {
#pragma unroll 4
            for (int k = threadIdx.x; k < kSortChunk; k += kSortThreads) {
                const K kk = put(k);
                if (next_mask) hist_add_all(S.next, (uint32_t)(kk >> next_shift) & next_mask);
            }
        } else {
            for (int k0 = 0; k0 < m; k0 += kSortThreads) {
                const int k = k0 + (int)threadIdx.x;
                K kk = 0;
                if (k < m) kk = put(k);
                if (next_mask) hist_add(S.next, (uint32_t)(kk >> next_shift) & next_mask, k < m);
            }
        }
        __syncthreads();
    }
    if (next_mask)
        for (int k = threadIdx.x; k < kSortMaxBins; k += kSortThreads)
            if (S.next[k]) atomicAdd(&a.hist[(pass + 1) * kSortMaxBins + k], S.next[k]);
}

// One pass (in_buf -> in_buf ^ 1) with BITS-bit digits at `shift`.
template <typename K, int BITS>
static cudaError_t launch_pass(const SortArgs& a, int in_buf, int shift, int pass, int next_shift, uint32_t next_mask,
                               cudaStream_t st) {
    static bool attr_set[kMaxDevices] = {};
    const size_t smem = sizeof(SortSmem<K, BITS>);
    cudaError_t e = once_per_device(attr_set, [&] {
        return cudaFuncSetAttribute(sort_pass_kernel<K, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e != cudaSuccess) return e;
    launch_pdl(sort_pass_kernel<K, BITS>, sort_grid(a.capacity, device_sms()), kSortThreads, smem, st, a, in_buf, shift, pass, next_shift,
                                                                              next_mask);
    return cudaGetLastError();
}

template <typename K>
static cudaError_t launch_passes(const SortArgs& a, int n_passes, const int* shifts, const int* bits, cudaStream_t st) {
    if (n_passes > kSortMaxPasses) return cudaErrorInvalidValue;
    for (int p = 0; p < n_passes; p++) {
        const bool more = p + 1 < n_passes;
        const int ns = more ? shifts[p + 1] : 0;
        const uint32_t nm = more ? ((1u << bits[p + 1]) - 1u) & a.digit_mask : 0u;
        cudaError_t e = cudaErrorInvalidValue;
        if (bits[p] == 8) e = launch_pass<K, 8>(a, p & 1, shifts[p], p, ns, nm, st);
        if constexpr (sizeof(K) == 4)
            if (bits[p] == 9) e = launch_pass<K, 9>(a, p & 1, shifts[p], p, ns, nm, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_sort32(const SortArgs& a, int n_passes, const int* shifts, const int* bits, cudaStream_t st) {
    return launch_passes<uint32_t>(a, n_passes, shifts, bits, st);
}

cudaError_t launch_sort64(const SortArgs& a, int n_passes, const int* shifts, cudaStream_t st) {
    const int bits[kSortMaxPasses] = {8, 8, 8, 8, 8, 8, 8, 8};
    return launch_passes<unsigned long long>(a, n_passes, shifts, bits, st);
}

cudaError_t launch_sort_count64(const SortArgs& a, int shift, cudaStream_t st) {
    sort_count_kernel<<<sort_grid(a.capacity, device_sms()), kHistThreads, 0, st>>>(a, shift);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Tile ranges.
// ----------------------------------------------------------------------------------------
// Each thread takes 4 consecutive sorted tile ids (one 16-byte load) and the id before them
// (from the previous lane, or loaded by lane 0); a start boundary j (key[j] != key[j - 1])
// opens key[j]'s range and closes key[j - 1]'s.
__global__ void __launch_bounds__(256) ranges_kernel(RangeArgs a) {
    pdl_begin();
    if (a.counters->status != 0) return;
    const int64_t P = (int64_t)a.counters->n_pairs;
    const int64_t groups = (P + 3) / 4;
    const int lane = threadIdx.x & 31;
    for (int64_t g0 = (int64_t)blockIdx.x * blockDim.x; g0 < groups; g0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = g0 + threadIdx.x;
        const int64_t i0 = 4 * g;
        uint32_t k[4] = {0u, 0u, 0u, 0u};
        if (i0 + 3 < P) {
            const uint4 q = *reinterpret_cast<const uint4*>(a.keys + i0);
            k[0] = q.x; k[1] = q.y; k[2] = q.z; k[3] = q.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) k[j] = i0 + j < P ? a.keys[i0 + j] : 0u;
        }
        uint32_t prev = __shfl_up_sync(0xffffffffu, k[3], 1);
        if (lane == 0 && i0 > 0 && i0 < P) prev = a.keys[i0 - 1];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t i = i0 + j;
            if (i >= P) break;
            const uint32_t before = j == 0 ? prev : k[j - 1];
            if (i == 0 || before != k[j]) {
                a.ranges[k[j]].x = (uint32_t)i;
                if (i > 0) a.ranges[before].y = (uint32_t)i;
            }
            if (i == P - 1) a.ranges[k[j]].y = (uint32_t)P;
        }
    }
}

cudaError_t launch_ranges(const RangeArgs& a, cudaStream_t st) {
    launch_pdl(ranges_kernel, device_sms() * 12, 256, 0, st, a);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Work order of the compositing kernels: (view, tile) items by decreasing pair count, in
// power-of-two buckets (bucket b holds counts in [2^(b-1), 2^b)), so that the largest tiles
// are scheduled first and the tail of the launch is made of short items.
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ int order_bucket(uint2 r) {
    const uint32_t c = r.y - r.x;
    return c ? 33 - __clz(c) : 0;   // 0 = empty, 1..33
}

// Bucket counts; the last block to finish turns them into the buckets' first positions, largest
// counts first (tmp: counts, then positions, then the blocks done).
__global__ void tile_order_hist_kernel(const uint2* ranges, int n_tiles, uint32_t* tmp, const Counters* c) {
    pdl_begin();
    __shared__ uint32_t h[kOrderBuckets];
    __shared__ bool last;
    for (int b = threadIdx.x; b < kOrderBuckets; b += blockDim.x) h[b] = 0;
    __syncthreads();
    if (c->status == 0)
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_tiles; t += gridDim.x * blockDim.x)
            atomicAdd(&h[order_bucket(ranges[t])], 1u);
    __syncthreads();
    for (int b = threadIdx.x; b < kOrderBuckets; b += blockDim.x)
        if (h[b]) atomicAdd(&tmp[b], h[b]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&tmp[2 * kOrderBuckets], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int b = threadIdx.x; b < kOrderBuckets; b += blockDim.x) h[b] = __ldcg(&tmp[b]);
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int b = kOrderBuckets - 1; b >= 0; b--) {
            tmp[kOrderBuckets + b] = run;
            run += h[b];
        }
    }
}

__global__ void tile_order_scatter_kernel(const uint2* ranges, int n_tiles, uint32_t* cursor, uint32_t* order,
                                          const Counters* c) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    for (int t0 = blockIdx.x * blockDim.x; t0 < n_tiles; t0 += gridDim.x * blockDim.x) {
        const int t = t0 + threadIdx.x;
        const bool ok = t < n_tiles;
        const int b = ok ? (c->status == 0 ? order_bucket(ranges[t]) : 0) : kOrderBuckets;
        // one atomic per bucket per warp
        const uint32_t peers = __match_any_sync(0xffffffffu, b);
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0;
        if (ok && lane == leader) base = atomicAdd(&cursor[b], (uint32_t)__popc(peers));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (ok) order[base + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)t;
    }
}

cudaError_t launch_tile_order(const uint2* ranges, int n_tiles, uint32_t* order, uint32_t* tmp, const Counters* c,
                              cudaStream_t st) {
    if (n_tiles <= 0) return cudaSuccess;
    const int blocks = (n_tiles + 255) / 256 < 1024 ? (n_tiles + 255) / 256 : 1024;
    launch_pdl(tile_order_hist_kernel, blocks, 256, 0, st, ranges, n_tiles, tmp, c);
    launch_pdl(tile_order_scatter_kernel, blocks, 256, 0, st, ranges, n_tiles, tmp + kOrderBuckets, order, c);
    return cudaGetLastError();
}

}  // namespace gs
