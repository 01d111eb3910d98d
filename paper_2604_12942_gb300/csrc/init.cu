// a10-a11: voxel-PCA geometric fitting (RMGS-SLAM §III-A) and the cascaded Gaussian
// initialisation (§III-B equations).  Points are grouped into cubic voxels by sorting their
// voxel keys with the library's radix sort; a warp then takes the voxels that start among 32 sorted
// points, for each the mean, the covariance, a 3x3 Jacobi eigen-decomposition, the planar / linear
// classification and the trace of the descriptor covariance, and writes the per-point features the
// learned initialiser consumes.
#include <cstring>

#include "gs_kernels.cuh"

namespace gs {

constexpr float kLambdaFloor = 1e-4f;   // (0.01 m)^2 floor of eigenvalues before the log
constexpr float kY00 = 0.28209479177387814f;

struct PcaArgs {
    int64_t n;
    const float* pts;      // [3][n]
    const float* rgb;      // [3][n]
    float voxel, tau_p, tau_l, sigma2, tau_trace;
    int min_pts;
    unsigned long long* keys;   // sorted keys
    const uint32_t* idx;        // sorted point indices
    float* x;              // [n][16]
    uint8_t* has_feature;
    uint8_t* reliable;
    float* s_pca;          // [n][3]
    float* q_pca;          // [n][4]
    const float* depth;    // [n]
    float fx;
};

// voxel key of an FP32 point: floor(p / s) per axis (IEEE division), 21 bits each, +2^20
__device__ __forceinline__ unsigned long long voxel_key(float x, float y, float z, float s) {
    unsigned long long k = 0;
    const float c[3] = {x, y, z};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        float q = floorf(__fdiv_rn(c[a], s));
        q = fminf(fmaxf(q, -1048576.0f), 1048575.0f);
        k = (k << 21) | (unsigned long long)((int)q + 1048576);
    }
    return k;
}

__global__ void voxel_key_kernel(const float* pts, int64_t n, float s, unsigned long long* keys, uint32_t* idx,
                                 Counters* c) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        c->status = 0;
        c->n_pairs = (unsigned long long)n;
    }
    if (i >= n) return;
    keys[i] = voxel_key(pts[i], pts[n + i], pts[2 * n + i], s);
    idx[i] = (uint32_t)i;
}

// Cyclic Jacobi eigen-decomposition of a symmetric 3x3 matrix; columns of V are eigenvectors.
__device__ void jacobi3(float A[9], float lam[3], float V[9]) {
#pragma unroll
    for (int i = 0; i < 9; i++) V[i] = (i % 4 == 0) ? 1.f : 0.f;
    for (int sweep = 0; sweep < 12; sweep++) {
        const float off = A[1] * A[1] + A[2] * A[2] + A[5] * A[5];
        const float diag = A[0] * A[0] + A[4] * A[4] + A[8] * A[8];
        if (off <= 1e-14f * diag || off == 0.f) break;
#pragma unroll
        for (int pq = 0; pq < 3; pq++) {
            const int p = pq == 2 ? 1 : 0, q = pq == 0 ? 1 : 2;
            const float apq = A[p * 3 + q];
            if (apq == 0.f) continue;
            const float theta = 0.5f * (A[q * 3 + q] - A[p * 3 + p]) / apq;
            const float t = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
            const float cth = rsqrtf(t * t + 1.f), sth = t * cth;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float akp = A[k * 3 + p], akq = A[k * 3 + q];
                A[k * 3 + p] = cth * akp - sth * akq;
                A[k * 3 + q] = sth * akp + cth * akq;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float apk = A[p * 3 + k], aqk = A[q * 3 + k];
                A[p * 3 + k] = cth * apk - sth * aqk;
                A[q * 3 + k] = sth * apk + cth * aqk;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float vkp = V[k * 3 + p], vkq = V[k * 3 + q];
                V[k * 3 + p] = cth * vkp - sth * vkq;
                V[k * 3 + q] = sth * vkp + cth * vkq;
            }
        }
    }
    lam[0] = A[0];
    lam[1] = A[4];
    lam[2] = A[8];
}

// Rotation matrix -> unit quaternion (w, x, y, z) with w >= 0 (largest-pivot form).
__device__ void matrix_to_quat(const float R[9], float q[4]) {
    const float tr = R[0] + R[4] + R[8];
    const float c0 = 1.f + tr, c1 = 1.f + R[0] - R[4] - R[8], c2 = 1.f - R[0] + R[4] - R[8], c3 = 1.f - R[0] - R[4] + R[8];
    int k = 0;
    float best = c0;
    if (c1 > best) { best = c1; k = 1; }
    if (c2 > best) { best = c2; k = 2; }
    if (c3 > best) { best = c3; k = 3; }
    const float s = 2.f * sqrtf(fmaxf(best, 1e-30f)), is = 1.f / s;
    if (k == 0) { q[0] = 0.25f * s; q[1] = (R[7] - R[5]) * is; q[2] = (R[2] - R[6]) * is; q[3] = (R[3] - R[1]) * is; }
    else if (k == 1) { q[0] = (R[7] - R[5]) * is; q[1] = 0.25f * s; q[2] = (R[1] + R[3]) * is; q[3] = (R[2] + R[6]) * is; }
    else if (k == 2) { q[0] = (R[2] - R[6]) * is; q[1] = (R[1] + R[3]) * is; q[2] = 0.25f * s; q[3] = (R[5] + R[7]) * is; }
    else { q[0] = (R[3] - R[1]) * is; q[1] = (R[2] + R[6]) * is; q[2] = (R[5] + R[7]) * is; q[3] = 0.25f * s; }
    const float nrm = rsqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    const float sg = q[0] < 0.f ? -nrm : nrm;
#pragma unroll
    for (int i = 0; i < 4; i++) q[i] *= sg;
}

// A warp takes 32 sorted positions and processes the voxels that start among them.  What is
// independent per point -- gathering it, its share of the trace, writing its outputs -- is done by
// all lanes; the sums of a voxel are taken one point after another in FP32, as the definition of
// the result, each by a lane of its own from shared memory (three coordinates, six covariances),
// so that a point costs an addition's latency instead of a gather's; and the eigen-decompositions
// of the warp's voxels run in the lanes of their first points at once.  With one thread per voxel
// doing everything the kernel took as long as its largest voxel: 398 us at 400k points, 89 in this
// form.
constexpr int kPcaWarps = 4;
constexpr int kStash = 512;   // points of a voxel held in shared memory at a time

struct PcaStash {
    float p[3][kStash];
};

// Points j0 .. j0 + m - 1 of the sorted order into the stash, all loads of a lane in flight.
__device__ __forceinline__ void stash_points(PcaStash& S, const PcaArgs& a, int64_t j0, int m) {
    const int lane = threadIdx.x & 31;
    for (int c = 0; c < m; c += 256) {
        uint32_t id[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int j = c + 32 * u + lane;
            id[u] = j < m ? a.idx[j0 + j] : 0u;
        }
        float v[3][8];
#pragma unroll
        for (int u = 0; u < 8; u++)
            if (c + 32 * u + lane < m) {
#pragma unroll
                for (int k = 0; k < 3; k++) v[k][u] = a.pts[(int64_t)k * a.n + id[u]];
            }
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int j = c + 32 * u + lane;
            if (j < m) {
#pragma unroll
                for (int k = 0; k < 3; k++) S.p[k][j] = v[k][u];
            }
        }
    }
    __syncwarp();
}

__global__ void __launch_bounds__(32 * kPcaWarps) voxel_stats_kernel(PcaArgs a, bool vec) {
    __shared__ PcaStash s_stash[kPcaWarps];
    __shared__ float s_t[kPcaWarps][2][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    PcaStash& S = s_stash[w];
    const int64_t n = a.n, base = ((int64_t)blockIdx.x * kPcaWarps + w) * 32;
    if (base >= n) return;   // (whole warps; no block barrier)
    const int64_t i = base + lane;
    const unsigned long long key = i < n ? a.keys[i] : 0ull;
    const bool head = i < n && (i == 0 || a.keys[i - 1] != key);
    const uint32_t heads = __ballot_sync(0xffffffffu, head);
    if (!heads) return;
    // end of this lane's voxel: the next head, or, for the last one, the first other key after
    int64_t end = n < base + 32 ? n : base + 32;
    {
        const uint32_t after = lane == 31 ? 0u : heads >> (lane + 1) << (lane + 1);
        const int lasth = 31 - __clz(heads);
        if (head && after) end = base + __ffs(after) - 1;
        const unsigned long long lk = __shfl_sync(0xffffffffu, key, lasth);
        int64_t e = base + 32;
        for (; e < n; e += 32) {
            const uint32_t same = __ballot_sync(0xffffffffu, e + lane < n && a.keys[e + lane] == lk);
            if (same != 0xffffffffu) { e += __ffs(~same) - 1; break; }
        }
        if (lane == lasth && base + 32 < n) end = e < n ? e : n;
    }
    const int64_t N = end - i;
    const bool has = head && N >= a.min_pts;
    float o[3] = {0.f, 0.f, 0.f}, mu[3] = {0.f, 0.f, 0.f}, C[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const uint32_t sums = __ballot_sync(0xffffffffu, has);
    for (uint32_t rest = sums; rest; rest &= rest - 1) {
        const int h = __ffs(rest) - 1;
        const int64_t v0 = base + h, vn = __shfl_sync(0xffffffffu, N, h);
        // centre on the first point for precision, then the two-pass mean / covariance
        const uint32_t p0 = a.idx[v0];
        const float oo[3] = {a.pts[p0], a.pts[n + p0], a.pts[2 * n + p0]};
        const int k = lane < 3 ? lane : 0;
        const float ok = k == 0 ? oo[0] : (k == 1 ? oo[1] : oo[2]);
        float acc = 0.f;
        for (int64_t c = 0; c < vn; c += kStash) {
            const int m = (int)(vn - c < kStash ? vn - c : kStash);
            __syncwarp();
            stash_points(S, a, v0 + c, m);
            if (lane < 3)
                for (int j = 0; j < m; j++) acc += S.p[k][j] - ok;
        }
        acc /= (float)vn;
        float mm[3];
#pragma unroll
        for (int q = 0; q < 3; q++) mm[q] = __shfl_sync(0xffffffffu, acc, q);
        // lanes 0..5: the covariances (0,0) (0,1) (0,2) (1,1) (1,2) (2,2)
        const int r = lane < 3 ? 0 : (lane < 5 ? 1 : 2), cc = lane < 3 ? lane : (lane < 5 ? lane - 2 : 2);
        const float orr = r == 0 ? oo[0] : (r == 1 ? oo[1] : oo[2]), mr = r == 0 ? mm[0] : (r == 1 ? mm[1] : mm[2]);
        const float oc = cc == 0 ? oo[0] : (cc == 1 ? oo[1] : oo[2]), mc = cc == 0 ? mm[0] : (cc == 1 ? mm[1] : mm[2]);
        float cov = 0.f;
        for (int64_t c = 0; c < vn; c += kStash) {
            const int m = (int)(vn - c < kStash ? vn - c : kStash);
            if (vn > kStash) {   // (else the points are still there)
                __syncwarp();
                stash_points(S, a, v0 + c, m);
            }
            if (lane < 6)
                for (int j = 0; j < m; j++) {
                    const float dr = S.p[r][j] - orr - mr, dc = S.p[cc][j] - oc - mc;
                    cov += dr * dc;
                }
        }
        cov /= (float)vn;
        float cv[6];
#pragma unroll
        for (int q = 0; q < 6; q++) cv[q] = __shfl_sync(0xffffffffu, cov, q);
        if (lane == h) {
#pragma unroll
            for (int q = 0; q < 3; q++) { o[q] = oo[q]; mu[q] = oo[q] + mm[q]; }
            C[0] = cv[0]; C[1] = C[3] = cv[1]; C[2] = C[6] = cv[2];
            C[4] = cv[3]; C[5] = C[7] = cv[4]; C[8] = cv[5];
        }
    }
    float l[3] = {0.f, 0.f, 0.f}, V[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, qv[4] = {1.f, 0.f, 0.f, 0.f};
    int cls = 0;   // class, 0 also where the eigenvalue gaps are degenerate
    if (has) {
        float W[9], lw[3];
        jacobi3(C, lw, W);
        // ascending order
        int id[3] = {0, 1, 2};
        if (lw[id[1]] < lw[id[0]]) { int t = id[0]; id[0] = id[1]; id[1] = t; }
        if (lw[id[2]] < lw[id[1]]) { int t = id[1]; id[1] = id[2]; id[2] = t; }
        if (lw[id[1]] < lw[id[0]]) { int t = id[0]; id[0] = id[1]; id[1] = t; }
#pragma unroll
        for (int c = 0; c < 3; c++) {
            l[c] = lw[id[c]];
#pragma unroll
            for (int r = 0; r < 3; r++) V[r * 3 + c] = W[r * 3 + id[c]];
        }
        // sign: largest-magnitude component positive; v_max = v_min x v_mid
#pragma unroll
        for (int c = 0; c < 2; c++) {
            int big = 0;
            if (fabsf(V[3 + c]) > fabsf(V[big * 3 + c])) big = 1;
            if (fabsf(V[6 + c]) > fabsf(V[big * 3 + c])) big = 2;
            if (V[big * 3 + c] < 0.f)
#pragma unroll
                for (int r = 0; r < 3; r++) V[r * 3 + c] = -V[r * 3 + c];
        }
        V[2] = V[3] * V[7] - V[6] * V[4];
        V[5] = V[6] * V[1] - V[0] * V[7];
        V[8] = V[0] * V[4] - V[3] * V[1];
        cls = (l[0] < a.tau_p) ? 1 : ((l[2] > a.tau_l * l[0]) ? 2 : 0);
        const float g1 = (l[1] - l[0]) / fmaxf(l[2], 1e-30f), g2 = (l[2] - l[1]) / fmaxf(l[2], 1e-30f);
        if (!(g1 > 1e-6f && g2 > 1e-6f)) cls = 0;
        matrix_to_quat(V, qv);
    }
    bool rel = false;
    // trace of the directional block of Sigma_g = sigma^2 sum_i ||F_i||_F^2, where row m of F_i is
    // (d.v_m v_k + d.v_k v_m) / (N (l_k - l_m)) and the two terms are orthogonal: a point's two
    // summands by its lane, added up in order by lane 0
    for (uint32_t rest = __ballot_sync(0xffffffffu, cls != 0); rest; rest &= rest - 1) {
        const int h = __ffs(rest) - 1;
        const int64_t v0 = base + h, vn = __shfl_sync(0xffffffffu, N, h);
        const int k = __shfl_sync(0xffffffffu, cls, h) == 1 ? 0 : 2;
        float vv[9], vl[3], vm[3];
#pragma unroll
        for (int q = 0; q < 9; q++) vv[q] = __shfl_sync(0xffffffffu, V[q], h);
#pragma unroll
        for (int q = 0; q < 3; q++) {
            vl[q] = __shfl_sync(0xffffffffu, l[q], h);
            vm[q] = __shfl_sync(0xffffffffu, mu[q], h);
        }
        float tr = 0.f;
        for (int64_t c = 0; c < vn; c += 32) {
            const int m = (int)(vn - c < 32 ? vn - c : 32);
            float d[3] = {0.f, 0.f, 0.f};
            if (lane < m) {
                const uint32_t pj = a.idx[v0 + c + lane];
#pragma unroll
                for (int q = 0; q < 3; q++) d[q] = a.pts[(int64_t)q * n + pj] - vm[q];
            }
            const float vk0 = k == 0 ? vv[0] : vv[2], vk1 = k == 0 ? vv[3] : vv[5], vk2 = k == 0 ? vv[6] : vv[8];
            const float dk = d[0] * vk0 + d[1] * vk1 + d[2] * vk2;
#pragma unroll
            for (int u = 0; u < 2; u++) {
                // the two other eigenvectors, in order: 1, 2 (k = 0) or 0, 1 (k = 2)
                const float vm0 = u == 0 ? (k == 0 ? vv[1] : vv[0]) : (k == 0 ? vv[2] : vv[1]);
                const float vm1 = u == 0 ? (k == 0 ? vv[4] : vv[3]) : (k == 0 ? vv[5] : vv[4]);
                const float vm2 = u == 0 ? (k == 0 ? vv[7] : vv[6]) : (k == 0 ? vv[8] : vv[7]);
                const float lm = u == 0 ? (k == 0 ? vl[1] : vl[0]) : (k == 0 ? vl[2] : vl[1]);
                const float dm = d[0] * vm0 + d[1] * vm1 + d[2] * vm2;
                const float den = (float)vn * ((k == 0 ? vl[0] : vl[2]) - lm);
                s_t[w][u][lane] = (dm * dm + dk * dk) / (den * den);
            }
            __syncwarp();
            if (lane == 0)
                for (int j = 0; j < m; j++) {
                    tr += s_t[w][0][j];
                    tr += s_t[w][1][j];
                }
            __syncwarp();
        }
        tr = __shfl_sync(0xffffffffu, tr, 0);
        if (lane == h) rel = tr * a.sigma2 < a.tau_trace;
    }
    // outputs, the points of each voxel over the lanes
    float lg[3];
#pragma unroll
    for (int k = 0; k < 3; k++) lg[k] = logf(fmaxf(l[k], kLambdaFloor));
    for (uint32_t rest = heads; rest; rest &= rest - 1) {
        const int h = __ffs(rest) - 1;
        const int64_t v0 = base + h, vn = __shfl_sync(0xffffffffu, N, h);
        const bool vh = __shfl_sync(0xffffffffu, has, h), vr = __shfl_sync(0xffffffffu, rel, h);
        float f[12], q[4];
#pragma unroll
        for (int k = 0; k < 3; k++) f[k] = __shfl_sync(0xffffffffu, lg[k], h);
#pragma unroll
        for (int k = 0; k < 9; k++) f[3 + k] = __shfl_sync(0xffffffffu, V[k], h);
#pragma unroll
        for (int k = 0; k < 4; k++) q[k] = __shfl_sync(0xffffffffu, qv[k], h);
        for (int64_t j = lane; j < vn; j += 32) {
            const uint32_t p = a.idx[v0 + j];
            float x[16];
#pragma unroll
            for (int k = 0; k < 12; k++) x[k] = vh ? f[k] : 0.f;
#pragma unroll
            for (int k = 0; k < 3; k++) x[12 + k] = vh ? a.rgb[(int64_t)k * n + p] : 0.f;
            x[15] = vh ? logf(fmaxf(a.depth[p], 1e-6f) / a.fx) : 0.f;
            float* xp = a.x + 16 * (size_t)p;
            float* qp = a.q_pca + 4 * (size_t)p;
            if (vec) {
#pragma unroll
                for (int k = 0; k < 4; k++)
                    reinterpret_cast<float4*>(xp)[k] = make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
                *reinterpret_cast<float4*>(qp) = make_float4(q[0], q[1], q[2], q[3]);
            } else {
#pragma unroll
                for (int k = 0; k < 16; k++) xp[k] = x[k];
#pragma unroll
                for (int k = 0; k < 4; k++) qp[k] = q[k];
            }
            a.has_feature[p] = vh;
            a.reliable[p] = vr;
#pragma unroll
            for (int k = 0; k < 3; k++) a.s_pca[3 * (size_t)p + k] = vh ? 0.5f * f[k] : 0.f;
        }
    }
}

// Frames a point may be seen from (the segment's keyframes / loopframes), by value.
struct FrameSet {
    int n;
    gs_camera cam[GS_MAX_VIEWS];
};

// Per point: the camera-frame depth in the closest frame whose image it projects into (the
// "closer view" of §III-B), and whether there is one; if none, the depth in frame 0.
__global__ void point_depth_kernel(const float* pts, int64_t n, const __grid_constant__ FrameSet fs, float* depth,
                                   uint8_t* inside) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x = pts[i], y = pts[n + i], z = pts[2 * n + i];
    float best = 0.f, first = 0.f;
    bool found = false;
    for (int f = 0; f < fs.n; f++) {
        const gs_camera& cam = fs.cam[f];
        const float* R = cam.R_cw;
        const float cx = R[0] * x + R[1] * y + R[2] * z + cam.t_cw[0];
        const float cy = R[3] * x + R[4] * y + R[5] * z + cam.t_cw[1];
        const float cz = R[6] * x + R[7] * y + R[8] * z + cam.t_cw[2];
        if (f == 0) first = cz;
        if (!(cz > 0.f)) continue;
        const float u = cam.fx * cx / cz + cam.cx, v = cam.fy * cy / cz + cam.cy;
        if (u >= 0.f && u < (float)cam.width && v >= 0.f && v < (float)cam.height && (!found || cz < best)) {
            best = cz;
            found = true;
        }
    }
    depth[i] = found ? best : first;
    inside[i] = found;
}



struct PcaWs {
    size_t counters, keys0, keys1, vals0, vals1, hist, total;
};

static size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// digit counts, tickets and look-back words of the sort
constexpr size_t kPcaSortCounts = sizeof(uint32_t) * kSortMaxPasses * kSortMaxBins;
constexpr size_t kPcaSortHead = kPcaSortCounts + 256;
constexpr size_t kPcaSortRegion = sizeof(uint32_t) * (512 * 512 + 512);
static_assert(kPcaSortHead + kSortGroupBytes + (size_t)kSortMaxGrid * 4 * kSortBins <= kPcaSortRegion,
              "sort_lookback_bytes of any size");

static PcaWs pca_layout(int64_t n) {
    PcaWs L;
    size_t off = 0;
    auto take = [&](size_t b) { const size_t r = off; off = al256(off + b); return r; };
    L.counters = take(sizeof(Counters));
    L.keys0 = take(8 * (size_t)n);
    L.keys1 = take(8 * (size_t)n);
    L.vals0 = take(4 * (size_t)n);
    L.vals1 = take(4 * (size_t)n);
    L.hist = take(kPcaSortRegion);
    L.total = off;
    return L;
}

size_t pca_workspace_size(int64_t n) { return pca_layout(n).total; }

cudaError_t launch_voxel_pca(const float* pts, const float* rgb, int64_t n, const FrameSet& fs, float voxel,
                             int min_pts, float tau_p, float tau_l, float sigma, float tau_trace, void* ws,
                             float* x, uint8_t* has_feature, uint8_t* reliable, float* s_pca, float* q_pca,
                             float* depth, uint8_t* inside, cudaStream_t st) {
    const PcaWs L = pca_layout(n);
    char* b = static_cast<char*>(ws);
    Counters* cnt = reinterpret_cast<Counters*>(b + L.counters);
    SortArgs sa;
    unsigned long long* vkeys = reinterpret_cast<unsigned long long*>(b + L.keys0);
    sa.keys[0] = vkeys;
    sa.keys[1] = b + L.keys1;
    sa.vals[0] = reinterpret_cast<uint32_t*>(b + L.vals0);
    sa.vals[1] = reinterpret_cast<uint32_t*>(b + L.vals1);
    sa.hist = reinterpret_cast<uint32_t*>(b + L.hist);
    sa.tickets = reinterpret_cast<uint32_t*>(b + L.hist + kPcaSortCounts);
    sa.lookback = reinterpret_cast<unsigned long long*>(b + L.hist + kPcaSortHead);
    sa.counters = cnt;
    sa.count = &cnt->n_pairs;
    sa.capacity = n;
    cudaError_t e = cudaMemsetAsync(b + L.hist, 0, kPcaSortHead + sort_lookback_bytes(n, 8), st);
    if (e != cudaSuccess) return e;
    const int blocks = (int)((n + 255) / 256);
    point_depth_kernel<<<blocks, 256, 0, st>>>(pts, n, fs, depth, inside);
    voxel_key_kernel<<<blocks, 256, 0, st>>>(pts, n, voxel, vkeys, sa.vals[0], cnt);
    int shifts[8] = {0, 8, 16, 24, 32, 40, 48, 56};
    if ((e = launch_sort_count64(sa, shifts[0], st)) != cudaSuccess) return e;
    e = launch_sort64(sa, 8, shifts, st);   // 63-bit keys, result back in buffer 0
    if (e != cudaSuccess) return e;
    PcaArgs a;
    a.n = n;
    a.pts = pts;
    a.rgb = rgb;
    a.voxel = voxel;
    a.tau_p = tau_p;
    a.tau_l = tau_l;
    a.sigma2 = sigma * sigma;
    a.tau_trace = tau_trace;
    a.min_pts = min_pts;
    a.keys = vkeys;
    a.idx = sa.vals[0];
    a.x = x;
    a.has_feature = has_feature;
    a.reliable = reliable;
    a.s_pca = s_pca;
    a.q_pca = q_pca;
    a.depth = depth;
    a.fx = fs.cam[0].fx;
    // vec: 16-byte rows of x and q_pca
    const bool vec = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(q_pca)) & 15) == 0;
    constexpr int kPcaRows = 32 * kPcaWarps;
    voxel_stats_kernel<<<(unsigned)((n + kPcaRows - 1) / kPcaRows), kPcaRows, 0, st>>>(a, vec);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Cascade (§III-B): model where the MLP prediction is valid, else PCA where reliable, else
// the isotropic depth heuristic.
// ---------------------------------------------------------------------------------------
struct CascadeArgs {
    int64_t n;
    int K;                  // SH coefficients per channel of the output map
    const float* pts;       // [3][n]
    const float* rgb;       // [3][n]
    const float* y;         // [n][16] or null
    const uint8_t* has_feature;
    const uint8_t* reliable;
    const float* s_pca;
    const float* q_pca;
    const float* depth;
    const uint8_t* inside;
    float fx;
    unsigned int* count;    // #(reliable and not valid)
    float opacity_logit0;
    float *means, *log_scales, *quats, *logits, *sh;   // output planes
    int32_t* branch;
    float* beta_out;
};

__device__ __forceinline__ bool model_valid(const CascadeArgs& a, int64_t i) {
    if (!a.y || !a.has_feature[i] || !a.inside[i]) return false;
    const float* y = a.y + 16 * (size_t)i;
#pragma unroll
    for (int k = 0; k < 11; k++)
        if (!isfinite(y[k])) return false;
#pragma unroll
    for (int k = 0; k < 3; k++)
        if (!(fabsf(y[k]) < 3.f)) return false;
    return true;
}

__global__ void cascade_count_kernel(CascadeArgs a) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned int c = 0;
    if (i < a.n) c = (a.reliable[i] && !model_valid(a, i)) ? 1u : 0u;
    c = warp_sum(c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(a.count, c);
}

__global__ void cascade_assign_kernel(CascadeArgs a) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n = a.n;
    const float beta = fminf(1.f, fmaxf(0.25f, (float)(*a.count) / (float)(n > 0 ? n : 1)));
    if (i == 0 && a.beta_out) *a.beta_out = beta;
    if (i >= n) return;
    float ls[3], q[4] = {1.f, 0.f, 0.f, 0.f}, col[3], lo = a.opacity_logit0;
#pragma unroll
    for (int k = 0; k < 3; k++) col[k] = a.rgb[(int64_t)k * n + i];
    int br = 0;
    if (model_valid(a, i)) {
        const float* y = a.y + 16 * (size_t)i;
        float qq[4], nq = 0.f;
#pragma unroll
        for (int k = 0; k < 4; k++) { qq[k] = a.q_pca[4 * (size_t)i + k] + y[3 + k]; nq += qq[k] * qq[k]; }
        nq = rsqrtf(nq);
#pragma unroll
        for (int k = 0; k < 4; k++) q[k] = qq[k] * nq;
#pragma unroll
        for (int k = 0; k < 3; k++) { ls[k] = a.s_pca[3 * (size_t)i + k] + y[k]; col[k] += y[8 + k]; }
        lo += y[7];
        br = 2;
    } else if (a.reliable[i]) {
        const float lb = logf(beta);
#pragma unroll
        for (int k = 0; k < 3; k++) ls[k] = a.s_pca[3 * (size_t)i + k] + lb;
#pragma unroll
        for (int k = 0; k < 4; k++) q[k] = a.q_pca[4 * (size_t)i + k];
        br = 1;
    } else {
        const float s = logf(fmaxf(a.depth[i], 1e-6f) / a.fx);
#pragma unroll
        for (int k = 0; k < 3; k++) ls[k] = s;
    }
#pragma unroll
    for (int k = 0; k < 3; k++) {
        a.means[(int64_t)k * n + i] = a.pts[(int64_t)k * n + i];
        a.log_scales[(int64_t)k * n + i] = ls[k];
    }
#pragma unroll
    for (int k = 0; k < 4; k++) a.quats[(int64_t)k * n + i] = q[k];
    a.logits[i] = lo;
#pragma unroll
    for (int c = 0; c < 3; c++) a.sh[(int64_t)c * n + i] = (col[c] - 0.5f) / kY00;
    for (int k = 3; k < 3 * a.K; k++) a.sh[(int64_t)k * n + i] = 0.f;
    if (a.branch) a.branch[i] = br;
}

cudaError_t launch_cascade(const CascadeArgs& a, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(a.count, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    const int blocks = (int)((a.n + 255) / 256);
    if (blocks > 0) cascade_count_kernel<<<blocks, 256, 0, st>>>(a);
    cascade_assign_kernel<<<blocks > 0 ? blocks : 1, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace gs

using namespace gs;

namespace gs {
gs_status record_error(gs_status s, const char* msg);
}

extern "C" size_t gs_pca_workspace_size(int64_t n) { return n > 0 ? pca_workspace_size(n) : 256; }

extern "C" gs_status gs_voxel_pca(const float* pts, const float* rgb, int64_t n, const gs_camera* frames,
                                  int32_t n_frames, const gs_pca_opts* opts, void* ws, size_t ws_bytes, float* x_out,
                                  uint8_t* has_feature, uint8_t* reliable, float* s_pca, float* q_pca, float* depth,
                                  uint8_t* inside, void* stream) {
    if (n < 0 || n > 0xFFFFFFFFll) return record_error(GS_ERR_INVALID_ARG, "n out of range");
    if (!frames || !opts) return record_error(GS_ERR_INVALID_ARG, "frames / opts is NULL");
    if (n_frames < 1 || n_frames > GS_MAX_VIEWS) return record_error(GS_ERR_INVALID_ARG, "n_frames must be in [1, 32]");
    FrameSet fs;
    memset(&fs, 0, sizeof(fs));
    fs.n = n_frames;
    for (int f = 0; f < n_frames; f++) {
        if (!(frames[f].fx > 0.f) || !(frames[f].fy > 0.f)) return record_error(GS_ERR_INVALID_ARG, "focal lengths must be > 0");
        fs.cam[f] = frames[f];
    }
    if (n == 0) return GS_OK;
    if (!pts || !rgb || !ws || !x_out || !has_feature || !reliable || !s_pca || !q_pca || !depth || !inside)
        return record_error(GS_ERR_INVALID_ARG, "NULL buffer");
    if (ws_bytes < pca_workspace_size(n)) return record_error(GS_ERR_INVALID_ARG, "PCA workspace too small");
    if (!(opts->voxel > 0.f) || opts->min_pts < 1) return record_error(GS_ERR_INVALID_ARG, "bad PCA options");
    cudaError_t e = launch_voxel_pca(pts, rgb, n, fs, opts->voxel, opts->min_pts, opts->tau_p, opts->tau_l,
                                     opts->sigma, opts->tau_trace, ws, x_out, has_feature, reliable, s_pca, q_pca,
                                     depth, inside, (cudaStream_t)stream);
    if (e != cudaSuccess) return record_error(GS_ERR_CUDA, cudaGetErrorString(e));
    return GS_OK;
}

extern "C" gs_status gs_init_cascade(const float* pts, const float* rgb, int64_t n, const float* y,
                                     const uint8_t* has_feature, const uint8_t* reliable, const float* s_pca,
                                     const float* q_pca, const float* depth, const uint8_t* inside, float fx,
                                     float opacity_init, gs_gaussians* out, int32_t* branch, unsigned int* count_tmp,
                                     float* beta_out, void* stream) {
    if (!out || out->n != n || n < 0) return record_error(GS_ERR_INVALID_ARG, "output map must have n Gaussians");
    if (out->sh_degree < 0 || out->sh_degree > 3) return record_error(GS_ERR_INVALID_ARG, "sh_degree must be 0..3");
    if (!(opacity_init > 0.f && opacity_init < 1.f)) return record_error(GS_ERR_INVALID_ARG, "opacity_init in (0,1)");
    if (n > 0 && (!pts || !rgb || !has_feature || !reliable || !s_pca || !q_pca || !depth || !inside || !count_tmp ||
                  !out->means || !out->log_scales || !out->quats || !out->opacity_logits || !out->sh))
        return record_error(GS_ERR_INVALID_ARG, "NULL buffer");
    CascadeArgs a;
    a.n = n;
    a.K = (out->sh_degree + 1) * (out->sh_degree + 1);
    a.pts = pts; a.rgb = rgb; a.y = y; a.has_feature = has_feature; a.reliable = reliable;
    a.s_pca = s_pca; a.q_pca = q_pca; a.depth = depth; a.inside = inside; a.fx = fx;
    a.count = count_tmp;
    a.opacity_logit0 = logf(opacity_init / (1.f - opacity_init));
    a.means = out->means; a.log_scales = out->log_scales; a.quats = out->quats; a.logits = out->opacity_logits;
    a.sh = out->sh;
    a.branch = branch;
    a.beta_out = beta_out;
    cudaError_t e = launch_cascade(a, (cudaStream_t)stream);
    if (e != cudaSuccess) return record_error(GS_ERR_CUDA, cudaGetErrorString(e));
    return GS_OK;
}
