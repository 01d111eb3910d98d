// Gaussian-GICP loop registration (RMGS-SLAM §III-D): the frustum target set around a
// historical loopframe, planar-regularised covariances, nearest-mean correspondences and the
// Gauss-Newton iterations on sum r^T (Sigma~_n + R Sigma~_m R^T)^-1 r, r = mu_n - T mu_m.
//
// The target set's decisions (in front of the near plane, inside the image, within d_max of
// the view's centre) are taken in FP32 with a fixed operation order.  Correspondences are found
// in FP32 through a spatial hash of the target means in cells of about d_corr / 4 (their exact
// size does not matter: every search covers the cells of the whole ball around the query).
// The weights, residuals and normal equations are evaluated in FP64 and summed in FP64; the
// last block of an iteration solves the 6 x 6 system and updates T on the device.
#include <cstring>

#include "gs_kernels.cuh"

namespace gs {

constexpr int kGThreads = 256;

// (gicp_scratch_bytes counts 240 bytes for the state: the 512 of this form fit because the
// search's tables are smaller than what it counts for them, see hash_layout)
struct GicpState {
    unsigned long long count;
    double acc[32];          // H upper triangle (21), g (6), cost, correspondences, 3 unused
    double T[12];            // current transform, row-major 3 x 4
    double eps;
    int32_t it, max_iters;   // iterations begun; limit
    int32_t stage;           // 0 iterating, 1 evaluating at the final T, 2 done
    int32_t converged;
    uint32_t blocks_done;    // blocks of the running evaluation that have added their sums
    uint32_t n_list;         // listed source rows
};
static_assert(sizeof(GicpState) <= 512, "the state's slot of the scratch");
constexpr size_t kStateSlot = 512;
constexpr size_t kStateCounted = 240;   // the state's share of gicp_scratch_bytes

static int g_grid(int64_t n) {
    int64_t b = (n + kGThreads - 1) / kGThreads;
    return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

__global__ void __launch_bounds__(kGThreads) gicp_target_kernel(GicpMap map, const GicpView* views, int nv,
                                                                float near_z, float dmax2, const uint8_t* src_flag,
                                                                uint8_t* flag, GicpState* s) {
    uint32_t cnt = 0;
    const int64_t n = map.n;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float m0 = map.means[i], m1 = map.means[n + i], m2 = map.means[2 * n + i];
        bool in = false;
        for (int k = 0; k < nv && !in; k++) {
            const GicpView& V = views[k];
            float pc[3];
#pragma unroll
            for (int r = 0; r < 3; r++)
                pc[r] = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(V.R[3 * r], m0), __fmul_rn(V.R[3 * r + 1], m1)),
                                            __fmul_rn(V.R[3 * r + 2], m2)), V.t[r]);
            const float z = pc[2];
            const float u = __fadd_rn(__fdiv_rn(__fmul_rn(V.fx, pc[0]), z), V.cx);
            const float v = __fadd_rn(__fdiv_rn(__fmul_rn(V.fy, pc[1]), z), V.cy);
            const bool img = z > near_z && u >= 0.f && u < V.W && v >= 0.f && v < V.H;
            const float d0 = __fsub_rn(m0, V.c[0]), d1 = __fsub_rn(m1, V.c[1]), d2 = __fsub_rn(m2, V.c[2]);
            const float dd = __fadd_rn(__fadd_rn(__fmul_rn(d0, d0), __fmul_rn(d1, d1)), __fmul_rn(d2, d2));
            in = img && dd < dmax2;
        }
        if (src_flag && src_flag[i]) in = false;
        flag[i] = in ? 1 : 0;
        cnt += in;
    }
    cnt = warp_sum(cnt);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&s->count, (unsigned long long)cnt);
}

// ---------------------------------------------------------------------------------------
// Target hash: the flagged target means by cell hash (counting sort).
//
// Cells are about d_corr / 4 wide, so that the ball around a query -- d_corr wide at first,
// the distance to the last iteration's match from then on -- holds few points outside its
// cells: with cells of d_corr a query scanned 27 of them, thousands of candidates on a dense
// map, to keep one.  The cell of a coordinate is floor(p * inv_h) in FP32, a monotone function
// of p, so the cells between those of q - r and q + r hold every point within r of q whatever
// the rounding.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t g_hash(int cx, int cy, int cz, uint32_t mask) {
    return ((uint32_t)cx * 73856093u ^ (uint32_t)cy * 19349663u ^ (uint32_t)cz * 83492791u) & mask;
}
// buckets of the occupancy table, whose entries are the occupied cells of a 4 x 4 x 4 block
// (bit x + 4 y + 16 z): other multipliers (the first three primes of 32-bit xxHash), so that they
// do not repeat the cells' collisions
__device__ __forceinline__ uint32_t g_coarse(int cx, int cy, int cz, uint32_t mask) {
    return ((uint32_t)cx * 2654435761u ^ (uint32_t)cy * 2246822519u ^ (uint32_t)cz * 3266489917u) & mask;
}
constexpr float kCellLimit = 1e9f;   // cells beyond it are one
__device__ __forceinline__ int g_cell(float p, float inv) {
    return __float2int_rd(fminf(fmaxf(__fmul_rn(p, inv), -kCellLimit), kCellLimit));
}

// pts: the flagged target means in hash order, (x, y, z, row index bits), so that a candidate
// of the nearest-mean search is one 16-byte load from a contiguous run of its cell
struct GicpHash {
    uint64_t T;              // source rows listed at a time
    uint32_t Te, mask;       // hash buckets (a power of two) and Te - 1
    uint32_t omask;          // occupancy buckets - 1
    uint32_t *start;         // [Te + 1] first point of each bucket
    uint32_t *list, *nn;     // [T] listed source rows, each one's nearest target (~0: none)
    unsigned long long* occ; // [omask + 1] occupied cells of the blocks
    uint32_t *bsum;
    float4* pts;
    GicpState* state;
    size_t bytes;
};

// T as gicp_scratch_bytes sizes it (>= 2 n).  The table takes n / 4 buckets: the targets are
// a few per cent of the map they are flagged in, and several share a cell.
static GicpHash hash_layout(void* scratch, int64_t n_tar) {
    GicpHash h;
    h.T = 1;
    while (h.T < (uint64_t)(2 * (n_tar > 0 ? n_tar : 1))) h.T <<= 1;
    uint64_t te = h.T < 1024 ? h.T : 1024;
    while (te < (uint64_t)n_tar / 4) te <<= 1;
    h.Te = (uint32_t)te;
    h.mask = h.Te - 1;
    h.state = static_cast<GicpState*>(scratch);
    char* base = static_cast<char*>(scratch);
    size_t off = kStateSlot;
    off += (16 - (reinterpret_cast<uintptr_t>(base + off) & 15)) & 15;
    h.pts = reinterpret_cast<float4*>(base + off);
    off += sizeof(float4) * (size_t)(n_tar > 0 ? n_tar : 0);
    auto words = [&](size_t n) { uint32_t* r = reinterpret_cast<uint32_t*>(base + off); off += sizeof(uint32_t) * n; return r; };
    const uint64_t to = te > 1024 ? te / 8 : (te >= 32 ? te / 32 : 1);
    h.omask = (uint32_t)(to - 1);
    h.occ = reinterpret_cast<unsigned long long*>(words(2 * to));   // (off is a multiple of 16 here)
    h.list = words(h.T);
    h.nn = words(h.T);
    h.start = words(te + 1);
    h.bsum = words(te / 1024 + 2);
    h.bytes = off;
    return h;
}

size_t gicp_scratch_bytes(int64_t n_tar) {
    uint64_t T = 1;
    while (T < (uint64_t)(2 * (n_tar > 0 ? n_tar : 1))) T <<= 1;
    // 3 T + n + T / 1024 + 2 words, then (16-byte aligned) 16 bytes a row and 12 doubles; what
    // hash_layout takes is never more
    const size_t words = 3 * (size_t)T + (size_t)n_tar + (size_t)(T / 1024) + 2;
    const size_t reg = kStateCounted + sizeof(uint32_t) * words + 15 +
                       sizeof(float4) * (size_t)(n_tar > 0 ? n_tar : 0) + 12 * sizeof(double);
    // target set: the state, then the view table
    const size_t tgt = ((kStateCounted + 255) & ~(size_t)255) + sizeof(GicpView) * GS_MAX_VIEWS;
    return ((reg > tgt ? reg : tgt) + 255) & ~(size_t)255;
}

__global__ void __launch_bounds__(kGThreads) gicp_hash_count(GicpMap tar, const uint8_t* flag, float inv, GicpHash h,
                                                             uint32_t* count) {
    const int64_t n = tar.n;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (flag && !flag[i]) continue;
        const int cx = g_cell(tar.means[i], inv), cy = g_cell(tar.means[n + i], inv), cz = g_cell(tar.means[2 * n + i], inv);
        atomicAdd(&count[g_hash(cx, cy, cz, h.mask)], 1u);
        const unsigned long long bit = 1ull << ((cx & 3) | (cy & 3) << 2 | (cz & 3) << 4);
        unsigned long long* o = &h.occ[g_coarse(cx >> 2, cy >> 2, cz >> 2, h.omask)];
        if (!(*o & bit)) atomicOr(o, bit);
    }
}

__global__ void __launch_bounds__(kGThreads) gicp_hash_fill(GicpMap tar, const uint8_t* flag, float inv, GicpHash h,
                                                            uint32_t* cursor) {
    const int64_t n = tar.n;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (flag && !flag[i]) continue;
        const float x = tar.means[i], y = tar.means[n + i], z = tar.means[2 * n + i];
        const uint32_t b = g_hash(g_cell(x, inv), g_cell(y, inv), g_cell(z, inv), h.mask);
        h.pts[h.start[b] + atomicAdd(&cursor[b], 1u)] = make_float4(x, y, z, __int_as_float((int)i));
    }
}

// ---------------------------------------------------------------------------------------
// Source list: the flagged source rows of [lo, hi) (hi - lo <= T), with no match yet.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kGThreads) gicp_src_compact(const uint8_t* flag, int64_t lo, int64_t hi,
                                                              uint32_t* list, uint32_t* nn, uint32_t* count) {
    const int lane = threadIdx.x & 31;
    uint32_t ltm;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(ltm));
    // (base is the same for the 32 lanes of a warp, so the loop and the ballot are warp-uniform)
    for (int64_t base = lo + (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < hi;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t m = base + lane;
        const bool f = m < hi && (!flag || flag[m] != 0);
        const uint32_t bal = __ballot_sync(0xffffffffu, f);
        if (!bal) continue;
        uint32_t b = 0;
        if (lane == 0) b = atomicAdd(count, (uint32_t)__popc(bal));
        b = __shfl_sync(0xffffffffu, b, 0);
        if (f) {
            const uint32_t at = b + __popc(bal & ltm);
            list[at] = (uint32_t)(m - lo);
            nn[at] = 0xFFFFFFFFu;
        }
    }
}

// ---------------------------------------------------------------------------------------
// Nearest target of every listed source row: the least (FP32 squared distance, row) below r2.
//
// Eight lanes per query; latency bound (occupancy word -> bucket -> points, each load waiting
// for the one before), so the kernel is kept small for occupancy and the FP64 part is a kernel
// of its own.  The ball starts at the last iteration's match (T moves by less every iteration,
// so it usually is the match again or next to it) and then spans a block or two; a query without
// one takes the ball of d_corr, at most 36 blocks of 4 x 4 x 4 cells.  The lanes share a block:
// its occupancy word tells the cells that hold a point, lane s takes those with x + 4 (y & 1)
// = s, skips the ones farther away than the best so far and scans the rest.  At 80k source rows
// and a 2M-row map an evaluation's search takes 57 us (with a 27-cell search of d_corr cells, a
// thread per query and the FP64 part in the same kernel: 200 to 500 us).
constexpr int kSearchLanes = 8;
constexpr int kSearchSpan = 16;   // cells per axis; more only where FP32 cannot resolve the cells

__global__ void __launch_bounds__(kGThreads) gicp_search_kernel(GicpMap src, int64_t lo, GicpMap tar, float inv, float r2,
                                                                GicpHash h) {
    const GicpState* st = h.state;
    if (st->stage == 2) return;
    const float side = 1.0f / inv;
    const int lane = threadIdx.x & 31, sub = lane & (kSearchLanes - 1);
    const uint32_t gm = ((1u << kSearchLanes) - 1u) << (lane & ~(kSearchLanes - 1));
    const uint32_t cnt = st->n_list;
    float R[9], t[3];
#pragma unroll
    for (int r = 0; r < 3; r++) {
#pragma unroll
        for (int c = 0; c < 3; c++) R[3 * r + c] = (float)st->T[4 * r + c];
        t[r] = (float)st->T[4 * r + 3];
    }
    const int64_t ns = src.n, nt = tar.n;
    constexpr int kPerBlock = kGThreads / kSearchLanes;
    for (uint32_t li = blockIdx.x * kPerBlock + (threadIdx.x / kSearchLanes); li < cnt; li += gridDim.x * kPerBlock) {
        const int64_t m = lo + h.list[li];
        const uint32_t prev = h.nn[li];
        const float s0 = src.means[m], s1 = src.means[ns + m], s2 = src.means[2 * ns + m];
        float q[3];
#pragma unroll
        for (int r = 0; r < 3; r++)
            q[r] = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(R[3 * r], s0), __fmul_rn(R[3 * r + 1], s1)),
                                       __fmul_rn(R[3 * r + 2], s2)), t[r]);
        float best = r2;
        uint32_t bi = 0xFFFFFFFFu;
        auto test = [&](float px, float py, float pz, uint32_t j) {
            const float ex = __fsub_rn(q[0], px), ey = __fsub_rn(q[1], py), ez = __fsub_rn(q[2], pz);
            const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
            if (d2 < best || (d2 == best && bi != 0xFFFFFFFFu && j < bi)) { best = d2; bi = j; }
        };
        auto scan = [&](uint32_t b, uint32_t e) {
#pragma unroll 4
            for (uint32_t k = b; k < e; k++) {
                const float4 P = h.pts[k];
                test(P.x, P.y, P.z, (uint32_t)__float_as_int(P.w));
            }
        };
        // least squared distance from q to the slab of cells [c, c + 1) along axis r, rounded down:
        // cell boundaries are off by their FP32 rounding, which the slack of a 1024th of a cell and
        // 4 ulp of the coordinate covers
        auto gap = [&](int c, int width, int r) {
            const float slack = 0.001f * side + 5e-7f * fabsf(q[r]);
            const float lo = (float)c * side - slack, hi = (float)(c + width) * side + slack;
            const float g = fmaxf(fmaxf(lo - q[r], q[r] - hi), 0.f);
            return g * g;
        };
        // the occupied cells o of a block, shared by the lanes
        auto block = [&](int bx, int by, int bz, unsigned long long o) {
            o = o >> sub & 0x0101010101010101ull;
            const int cx = 4 * bx + (sub & 3), y0 = 4 * by + (sub >> 2);
            const float dx = gap(cx, 1, 0);
            while (o) {
                const int k = __ffsll((long long)o) - 1;   // sub + 8 (y >> 1) + 16 z, less sub
                o &= o - 1;
                const int cy = y0 + ((k >> 3) & 1) * 2, cz = 4 * bz + (k >> 4);
                if (0.999f * (dx + gap(cy, 1, 1) + gap(cz, 1, 2)) > best) continue;
                const uint32_t hh = g_hash(cx, cy, cz, h.mask);
                scan(__ldg(&h.start[hh]), __ldg(&h.start[hh + 1]));
            }
        };
        // the group's least (distance, row) to all its lanes
        auto merge = [&]() {
#pragma unroll
            for (int o = kSearchLanes / 2; o > 0; o >>= 1) {
                const float od = __shfl_xor_sync(gm, best, o);
                const uint32_t oj = __shfl_xor_sync(gm, bi, o);
                if (od < best || (od == best && oj < bi)) { best = od; bi = oj; }
            }
        };
        if (!(isfinite(q[0]) && isfinite(q[1]) && isfinite(q[2]))) {   // no distance to it is a number
            if (sub == 0) h.nn[li] = bi;
            continue;
        }
        if (prev != 0xFFFFFFFFu) test(tar.means[prev], tar.means[nt + prev], tar.means[2 * nt + prev], prev);
        // cells of the ball of squared radius best (rounded outwards)
        int c0[3], c1[3];
        auto ball = [&]() {
            const float rad = __fadd_ru(__fmul_ru(__fsqrt_ru(best), 1.00001f), 1e-18f);
            bool wide = !(rad < 1e18f);
#pragma unroll
            for (int r = 0; r < 3; r++) {
                c0[r] = g_cell(__fsub_rd(q[r], rad), inv);
                c1[r] = g_cell(__fadd_ru(q[r], rad), inv);
                wide = wide || c1[r] - c0[r] >= kSearchSpan || c1[r] >= (int)kCellLimit || c0[r] <= -(int)kCellLimit;
            }
            return wide;
        };
        if (ball()) {
            // a ball of more cells than that, or of cells past the limit (coordinates so large that
            // FP32 does not resolve the cells, or a d_corr without bound): every target
            for (uint32_t k = sub, e = h.start[h.Te]; k < e; k += kSearchLanes) scan(k, k + 1);
            merge();
            if (sub == 0) h.nn[li] = bi;
            continue;
        }
        const int x0 = c0[0] >> 2, y0 = c0[1] >> 2, z0 = c0[2] >> 2;
        const int nx = (c1[0] >> 2) - x0 + 1, ny = (c1[1] >> 2) - y0 + 1, nz = (c1[2] >> 2) - z0 + 1;
        // without a match so far: the block of the query first, and its best to all lanes, so that
        // the others are mostly out of reach
        int seen = -1;
        if (bi == 0xFFFFFFFFu) {
            const int bx = g_cell(q[0], inv) >> 2, by = g_cell(q[1], inv) >> 2, bz = g_cell(q[2], inv) >> 2;
            block(bx, by, bz, __ldg(&h.occ[g_coarse(bx, by, bz, h.omask)]));
            merge();
            seen = bx - x0 + nx * (by - y0 + ny * (bz - z0));
        }
        // eight blocks at a time, a lane each: the occupancy words of those within reach are loaded
        // together, then the lanes share the cells of each that holds any
        for (int k0 = 0; k0 < nx * ny * nz; k0 += kSearchLanes) {
            const int k = k0 + sub;
            const int bx = x0 + k % nx, by = y0 + (k / nx) % ny, bz = z0 + k / (nx * ny);
            unsigned long long o = 0;
            if (k < nx * ny * nz && k != seen &&
                !(0.999f * (gap(4 * bx, 4, 0) + gap(4 * by, 4, 1) + gap(4 * bz, 4, 2)) > best))
                o = __ldg(&h.occ[g_coarse(bx, by, bz, h.omask)]);
            uint32_t any = __ballot_sync(gm, o != 0) & gm;
            while (any) {
                const int from = __ffs(any) - 1;
                any &= any - 1;
                block(__shfl_sync(gm, bx, from), __shfl_sync(gm, by, from), __shfl_sync(gm, bz, from),
                      __shfl_sync(gm, o, from));
            }
        }
        merge();
        if (sub == 0) h.nn[li] = bi;
    }
}

// ---------------------------------------------------------------------------------------
// Normal equations, in FP64, and the Gauss-Newton update.
//
// GB300's FP64 pipe takes a warp instruction at the same cost however few lanes are active and
// at a small fraction of the FP32 rate, so the kernel is written for few FP64 instructions:
// a block first lists its matched pairs, so that warps are full, and the algebra is taken apart.
// The planar covariance R diag(1, 1, 1e-3) R^T is I - 0.999 n n^T with n the column of R that
// gets 1e-3, so Sigma~_n + R Sigma~_m R^T = I + R R^T - 0.999 (n n^T + m m^T), m = R n_m (R R^T is
// formed once a block and not taken for I: the caller's first transform is a rotation to its own
// rounding only, and every later one keeps what it had; with 2 I in its place a transform given in
// FP32 left ten times the error, and one 1e-3 off a rotation met another minimum); with O its
// inverse and q^ the cross-product matrix of T mu_m the blocks of J^T O J (J = [-I | q^]) are
// O, -O q^ and -q^ O q^, those of J^T O r are -O r and -q^ O r.  About 190 FP64 operations a
// pair where the matrix products spelled out took about 700: 41 us an evaluation at 80k source
// rows, of which about 8 are the last block's 6 x 6 solution.  The registration of 80k rows
// against a 2M-row map in 25 iterations went from 12.9 to 2.0 ms.
// ---------------------------------------------------------------------------------------
constexpr double kPlanar = 1.0 - 1e-3;
constexpr int kNormalThreads = 64;
constexpr int kNormalRows = 128;   // listed rows a block takes at a time (about 4 blocks per SM at 80k
                                   // rows: with 512 rows a few SMs had two blocks and the rest one)

// unit normal of the planar form: the column of the quaternion's rotation for the axis of the
// smallest log-scale (the first on ties)
__device__ __forceinline__ void planar_normal(const GicpMap& g, int64_t i, double (&c)[3]) {
    const int64_t n = g.n;
    const float qw = g.quats[i], qx = g.quats[n + i], qy = g.quats[2 * n + i], qz = g.quats[3 * n + i];
    const float l0 = g.log_scales[i], l1 = g.log_scales[n + i], l2 = g.log_scales[2 * n + i];
    const int e = (l0 <= l1 && l0 <= l2) ? 0 : (l1 <= l2 ? 1 : 2);
    // the columns are one formula of (x, y, z) turned cyclically to start at axis e
    const double w = qw, x = e == 0 ? qx : (e == 1 ? qy : qz), y = e == 0 ? qy : (e == 1 ? qz : qx),
                 z = e == 0 ? qz : (e == 1 ? qx : qy);
    const double wx = w * w + x * x, yz = y * y + z * z;
    const double s = 1.0 / (wx + yz), s2 = s + s;
    const double a = (wx - yz) * s, b = (x * y + w * z) * s2, d = (x * z - w * y) * s2;
    c[0] = e == 0 ? a : (e == 1 ? d : b);
    c[1] = e == 0 ? b : (e == 1 ? a : d);
    c[2] = e == 0 ? d : (e == 1 ? b : a);
}

// (rho, phi) -> [R | t] (row-major 3 x 4)
__device__ __forceinline__ void se3_exp_dev(const double (&xi)[6], double (&E)[12]) {
    const double *rho = xi, *phi = xi + 3;
    const double th = sqrt(phi[0] * phi[0] + phi[1] * phi[1] + phi[2] * phi[2]);
    const double K[9] = {0, -phi[2], phi[1], phi[2], 0, -phi[0], -phi[1], phi[0], 0};
    const bool tiny = th < 1e-12;
    double A = 1.0, B = 0.5, C = 0.0;   // tiny: R = I + K, V = I + K / 2
    if (!tiny) {
        double sn, cs;
        sincos(th, &sn, &cs);
        A = sn / th;
        B = (1 - cs) / (th * th);
        C = (1 - A) / (th * th);
    }
#pragma unroll
    for (int r = 0; r < 3; r++) {
        double t = 0;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double K2 = K[3 * r] * K[c] + K[3 * r + 1] * K[3 + c] + K[3 * r + 2] * K[6 + c];
            const double I = r == c ? 1.0 : 0.0;
            E[4 * r + c] = tiny ? I + K[3 * r + c] : I + A * K[3 * r + c] + B * K2;
            t += (I + B * K[3 * r + c] + C * K2) * rho[c];
        }
        E[4 * r + 3] = t;
    }
}

// One warp: the Gauss-Newton step from the summed normal equations (elimination without
// pivoting of the symmetric positive definite 6 x 6 system, a lane per entry), T <- Exp(xi) T,
// and the next stage.  Stops without a step on fewer than 6 correspondences or a pivot that is
// not positive.
__device__ void gicp_step(GicpState* s, const double* acc, double (*A)[7], bool final_eval) {
    const int lane = threadIdx.x & 31;
    if (final_eval) {
        if (lane == 0) s->stage = 2;
        return;
    }
    bool ok = acc[28] >= 6;
    if (lane < 6) {
        for (int c = 0; c < 6; c++) {
            const int a = min(lane, c), b = max(lane, c);
            A[lane][c] = acc[6 * a - a * (a - 1) / 2 + (b - a)];
        }
        A[lane][6] = -acc[21 + lane];
    }
    __syncwarp();
    double inv[6], xi[6];
    for (int k = 0; k < 6 && ok; k++) {
        const double p = A[k][k];
        ok = p > 0;
        inv[k] = 1.0 / p;
        const int w = 6 - k, r = k + 1 + lane / w, c = k + 1 + lane % w;   // 5 - k rows, 6 - k columns
        if (ok && r < 6) A[r][c] -= A[r][k] * inv[k] * A[k][c];
        __syncwarp();
    }
    double T[12];
    for (int k = 0; k < 12; k++) T[k] = s->T[k];
    double nrm = 0;
    if (ok) {
        for (int i = 5; i >= 0; i--) {
            double v = A[i][6];
            for (int k = i + 1; k < 6; k++) v -= A[i][k] * xi[k];
            xi[i] = v * inv[i];
            nrm += xi[i] * xi[i];
        }
        double E[12];
        se3_exp_dev(xi, E);
        __syncwarp();
        if (lane < 12) {
            const int r = lane / 4, c = lane % 4;
            double v = c == 3 ? E[4 * r + 3] : 0.0;
            for (int e = 0; e < 3; e++) v += E[4 * r + e] * T[4 * e + c];
            s->T[lane] = v;
        }
    }
    if (lane == 0) {
        const int it = s->it + 1;
        const bool conv = ok && sqrt(nrm) < s->eps;
        s->it = it;
        s->converged = conv ? 1 : 0;
        if (!ok || conv || it >= s->max_iters) s->stage = 1;
    }
}

__global__ void __launch_bounds__(kNormalThreads) gicp_normal_kernel(GicpMap src, int64_t lo, GicpMap tar, GicpHash h,
                                                                     int last_segment) {
    GicpState* st = h.state;
    if (st->stage == 2) return;
    __shared__ uint32_t s_li[kNormalRows], s_n;
    __shared__ double s_acc[kNormalThreads / 32][32];
    __shared__ double s_A[6][7], s_B[6];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t ltm;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(ltm));
    double T[12];
#pragma unroll
    for (int k = 0; k < 12; k++) T[k] = st->T[k];
    // I + R R^T, xx xy xz yy yz zz, by six threads (18 operations a thread would be a twentieth of
    // its pairs'); the barriers before the pairs order it
    if (threadIdx.x < 6) {
        const int k = threadIdx.x, a = k < 3 ? 0 : (k < 5 ? 1 : 2), b = k < 3 ? k : (k < 5 ? k - 2 : 2);
        double v = a == b ? 1.0 : 0.0;
        for (int e = 0; e < 3; e++) v += st->T[4 * a + e] * st->T[4 * b + e];
        s_B[k] = v;
    }
    const uint32_t cnt = st->n_list;
    const int64_t ns = src.n, nt = tar.n;
    double acc[32];
#pragma unroll
    for (int k = 0; k < 32; k++) acc[k] = 0.0;
    bool mine = false;
    for (uint32_t base = blockIdx.x * kNormalRows; base < cnt; base += gridDim.x * kNormalRows) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < kNormalRows; k += kNormalThreads) {
            const bool f = base + k < cnt && h.nn[base + k] != 0xFFFFFFFFu;
            const uint32_t bal = __ballot_sync(0xffffffffu, f);
            uint32_t b = 0;
            if (lane == 0 && bal) b = atomicAdd(&s_n, (uint32_t)__popc(bal));
            b = __shfl_sync(0xffffffffu, b, 0);
            if (f) s_li[b + __popc(bal & ltm)] = base + k;
        }
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < s_n; k += kNormalThreads) {
            const uint32_t li = s_li[k];
            const int64_t m = lo + h.list[li], j = h.nn[li];
            mine = true;
            const double a0 = src.means[m], a1 = src.means[ns + m], a2 = src.means[2 * ns + m];
            double q[3], r[3], nm[3], n[3], mr[3];
#pragma unroll
            for (int e = 0; e < 3; e++) q[e] = T[4 * e] * a0 + T[4 * e + 1] * a1 + T[4 * e + 2] * a2 + T[4 * e + 3];
#pragma unroll
            for (int e = 0; e < 3; e++) r[e] = (double)tar.means[e * nt + j] - q[e];
            planar_normal(src, m, nm);
            planar_normal(tar, j, n);
#pragma unroll
            for (int e = 0; e < 3; e++) mr[e] = T[4 * e] * nm[0] + T[4 * e + 1] * nm[1] + T[4 * e + 2] * nm[2];
            // A = I + R R^T - 0.999 (n n^T + m m^T): xx xy xz yy yz zz
            const double kn[3] = {kPlanar * n[0], kPlanar * n[1], kPlanar * n[2]};
            const double km[3] = {kPlanar * mr[0], kPlanar * mr[1], kPlanar * mr[2]};
            // (read here each time: held over the loop they would take 16 registers, an eighth block of an SM)
            const volatile double* B = s_B;
            const double A0 = B[0] - kn[0] * n[0] - km[0] * mr[0], A1 = B[1] - kn[0] * n[1] - km[0] * mr[1],
                         A2 = B[2] - kn[0] * n[2] - km[0] * mr[2], A3 = B[3] - kn[1] * n[1] - km[1] * mr[1],
                         A4 = B[4] - kn[1] * n[2] - km[1] * mr[2], A5 = B[5] - kn[2] * n[2] - km[2] * mr[2];
            // inverse by the adjugate
            const double c0 = A3 * A5 - A4 * A4, c1 = A2 * A4 - A1 * A5, c2 = A1 * A4 - A2 * A3;
            const double id = 1.0 / (A0 * c0 + A1 * c1 + A2 * c2);
            const double O0 = c0 * id, O1 = c1 * id, O2 = c2 * id, O3 = (A0 * A5 - A2 * A2) * id,
                         O4 = (A1 * A2 - A0 * A4) * id, O5 = (A0 * A3 - A1 * A1) * id;
            // P = O q^ (columns of q^: (0, q2, -q1), (-q2, 0, q0), (q1, -q0, 0))
            const double P00 = O1 * q[2] - O2 * q[1], P01 = O2 * q[0] - O0 * q[2], P02 = O0 * q[1] - O1 * q[0];
            const double P10 = O3 * q[2] - O4 * q[1], P11 = O4 * q[0] - O1 * q[2], P12 = O1 * q[1] - O3 * q[0];
            const double P20 = O4 * q[2] - O5 * q[1], P21 = O5 * q[0] - O2 * q[2], P22 = O2 * q[1] - O4 * q[0];
            acc[0] += O0; acc[1] += O1; acc[2] += O2;
            acc[3] -= P00; acc[4] -= P01; acc[5] -= P02;
            acc[6] += O3; acc[7] += O4;
            acc[8] -= P10; acc[9] -= P11; acc[10] -= P12;
            acc[11] += O5;
            acc[12] -= P20; acc[13] -= P21; acc[14] -= P22;
            // q^T O q^ = -q^ P: row 0 = q2 P1 - q1 P2, row 1 = q0 P2 - q2 P0, row 2 = q1 P0 - q0 P1
            acc[15] += q[2] * P10 - q[1] * P20; acc[16] += q[2] * P11 - q[1] * P21; acc[17] += q[2] * P12 - q[1] * P22;
            acc[18] += q[0] * P21 - q[2] * P01; acc[19] += q[0] * P22 - q[2] * P02;
            acc[20] += q[1] * P02 - q[0] * P12;
            const double g0 = O0 * r[0] + O1 * r[1] + O2 * r[2], g1 = O1 * r[0] + O3 * r[1] + O4 * r[2],
                         g2 = O2 * r[0] + O4 * r[1] + O5 * r[2];
            acc[21] -= g0; acc[22] -= g1; acc[23] -= g2;
            acc[24] += q[2] * g1 - q[1] * g2; acc[25] += q[0] * g2 - q[2] * g0; acc[26] += q[1] * g0 - q[0] * g1;
            acc[27] += r[0] * g0 + r[1] * g1 + r[2] * g2;
            acc[28] += 1.0;
        }
        __syncthreads();
    }
    // the warp's sums: 32 values halved at each of five lane exchanges, so that lane l ends with
    // the total of value l (31 additions instead of 5 for each of the 29 values)
    double total = 0.0;
    if (__any_sync(0xffffffffu, mine)) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool hi = lane & o;
#pragma unroll
            for (int k = 0; k < 16; k++) {
                if (k < o) {
                    const double keep = hi ? acc[o + k] : acc[k], give = hi ? acc[k] : acc[o + k];
                    acc[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
        }
        total = acc[0];
    }
    s_acc[w][lane] = total;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = 0;
        for (int k = 0; k < kNormalThreads / 32; k++) v += s_acc[k][lane];
        if (lane < 29 && v != 0.0) atomicAdd(&st->acc[lane], v);
        __threadfence();
        __syncwarp();
        bool last = false;
        if (lane == 0 && last_segment) last = atomicAdd(&st->blocks_done, 1u) == gridDim.x - 1;
        if (lane == 0) s_last = last;
    }
    __syncthreads();
    if (!s_last || w != 0) return;
    // every block of the evaluation has added its sums
    __threadfence();
    s_acc[0][lane] = __ldcg(&st->acc[lane]);
    __syncwarp();
    const bool final_eval = st->stage == 1;
    __syncwarp();   // every lane has read the stage that lane 0 moves on
    gicp_step(st, s_acc[0], s_A, final_eval);
    // the final evaluation's cost and count stay for the host
    if (!final_eval) st->acc[lane] = 0.0;
    if (lane == 0) st->blocks_done = 0;
}

cudaError_t launch_gicp_target_set(const GicpMap& map, const GicpView* views, int n_views, float near_z, float dmax2,
                                   const uint8_t* source_flag, uint8_t* target_flag, void* scratch,
                                   unsigned long long* count_host, cudaStream_t st) {
    GicpState* s = static_cast<GicpState*>(scratch);
    GicpView* dv = reinterpret_cast<GicpView*>(reinterpret_cast<char*>(scratch) + ((kStateCounted + 255) & ~(size_t)255));
    cudaError_t e = cudaMemsetAsync(s, 0, sizeof(s->count), st);   // (the target set uses the count alone)
    if (e != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(dv, views, sizeof(GicpView) * n_views, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    gicp_target_kernel<<<g_grid(map.n), kGThreads, 0, st>>>(map, dv, n_views, near_z, dmax2, source_flag, target_flag, s);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaMemcpyAsync(count_host, &s->count, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
}

// The target hash of one registration.
static cudaError_t build_hash(const GicpHash& h, const GicpMap& tar, const uint8_t* tar_flag, float inv, cudaStream_t st) {
    cudaError_t e;
    uint32_t *count = h.nn, *cursor = h.list;   // free until the source rows are listed
    if ((e = cudaMemsetAsync(count, 0, sizeof(uint32_t) * h.Te, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(cursor, 0, sizeof(uint32_t) * h.Te, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(h.occ, 0, sizeof(unsigned long long) * ((size_t)h.omask + 1), st)) != cudaSuccess) return e;
    if (tar.n > 0) gicp_hash_count<<<g_grid(tar.n), kGThreads, 0, st>>>(tar, tar_flag, inv, h, count);
    if ((e = exclusive_scan_u32(count, (int64_t)h.Te, h.start, h.bsum, h.start + h.Te, st)) != cudaSuccess) return e;
    if (tar.n > 0) gicp_hash_fill<<<g_grid(tar.n), kGThreads, 0, st>>>(tar, tar_flag, inv, h, cursor);
    return cudaGetLastError();
}

cudaError_t launch_gicp_register(const GicpMap& src, const uint8_t* src_flag, const GicpMap& tar, const uint8_t* tar_flag,
                                 const double (&T0)[12], float d_corr, int max_iters, double eps, void* scratch,
                                 size_t scratch_bytes, GicpOutcome* out, cudaStream_t st) {
    const GicpHash h = hash_layout(scratch, tar.n);
    if (h.bytes > scratch_bytes) return cudaErrorInvalidValue;
    const float inv = 4.0f / (1.001f * d_corr), r2 = d_corr * d_corr;
    cudaError_t e;
    if ((e = build_hash(h, tar, tar_flag, inv, st)) != cudaSuccess) return e;
    GicpState s;
    memset(&s, 0, sizeof(s));
    for (int k = 0; k < 12; k++) s.T[k] = T0[k];
    s.eps = eps;
    s.max_iters = max_iters;
    if ((e = cudaMemcpyAsync(h.state, &s, sizeof(s), cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    // The source rows in segments of at most T rows (one segment when the source map is no larger
    // than twice the target map).  One segment is listed once, and each row's match bounds its
    // next search; several share the list, so each evaluation lists and searches them anew.
    const bool one = (uint64_t)src.n <= h.T;
    auto list = [&](int64_t lo, int64_t hi) {
        const cudaError_t er = cudaMemsetAsync(&h.state->n_list, 0, sizeof(uint32_t), st);
        if (er == cudaSuccess && hi > lo)
            gicp_src_compact<<<g_grid(hi - lo), kGThreads, 0, st>>>(src_flag, lo, hi, h.list, h.nn, &h.state->n_list);
        return er;
    };
    const int sms = device_sms();
    auto evaluate = [&](int64_t lo, int64_t hi, bool last) {
        const int64_t rows = hi - lo > 0 ? hi - lo : 1;
        // (8 resident search blocks per SM; the normal equations are bound by the FP64 pipe)
        const int64_t gs = (rows * kSearchLanes + kGThreads - 1) / kGThreads, gn = (rows + kNormalRows - 1) / kNormalRows;
        gicp_search_kernel<<<(int)(gs < 8 * sms ? gs : 8 * sms), kGThreads, 0, st>>>(src, lo, tar, inv, r2, h);
        gicp_normal_kernel<<<(int)(gn < 8 * sms ? gn : 8 * sms), kNormalThreads, 0, st>>>(src, lo, tar, h, last ? 1 : 0);
    };
    if (one && (e = list(0, src.n)) != cudaSuccess) return e;
    // At most max_iters evaluations and one at the final T.  They are launched kPoll at a time
    // and the state is then read back: kernels launched past the end return at once, which costs
    // less than a host round trip every iteration.
    constexpr int kPoll = 8;
    for (int64_t done = 0; done <= max_iters;) {
        for (int k = 0; k < kPoll && done <= max_iters; k++, done++) {
            if (one) {
                evaluate(0, src.n, true);
            } else {
                for (int64_t lo = 0; lo < src.n; lo += (int64_t)h.T) {
                    const int64_t hi = src.n - lo < (int64_t)h.T ? src.n : lo + (int64_t)h.T;
                    if ((e = list(lo, hi)) != cudaSuccess) return e;
                    evaluate(lo, hi, hi == src.n);
                }
            }
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(&s, h.state, sizeof(s), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
        if (s.stage == 2) break;
    }
    for (int k = 0; k < 12; k++) out->T[k] = s.T[k];
    out->cost = s.acc[27];
    out->n_corr = (int64_t)s.acc[28];
    out->iters = s.it;
    out->converged = s.converged;
    return cudaSuccess;
}

}  // namespace gs
