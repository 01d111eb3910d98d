// a11-a12: the learned Gaussian initialiser's MLP (16 -> 128 -> 128 -> 128 -> 16, GELU),
// BF16 weights and activations with FP32 accumulation on the tensor cores
// (mma.sync m16n8k16), inference and one training step (MSE, backward GEMMs, Adam on FP32
// master weights).  It stands in for the paper's pretrained feed-forward model (§III-B).
//
// Parameters, packed:  weights BF16 [36864] = W1 (128x16) | W2 (128x128) | W3 (128x128) |
// W4 (16x128), each row-major [out][in];  biases FP32 [400] = b1 (128) | b2 | b3 | b4 (16).
#include <cuda_bf16.h>

#include "gs_kernels.cuh"

namespace gs {

constexpr int kIn = 16, kHid = 128, kOut = 16, kOutUsed = 11;
constexpr int kNW = 2048 + 32768 + 2048;
constexpr int kNB = 400;
__host__ __device__ __forceinline__ int woff(int l) { return l == 0 ? 0 : l == 1 ? 2048 : l == 2 ? 2048 + 16384 : 2048 + 32768; }
__host__ __device__ __forceinline__ int boff(int l) { return 128 * l; }
constexpr int kRows = 128;   // rows per CTA iteration (8 warps x 16)
constexpr int kThreads = 256;
constexpr int kLdIn = kIn + 8, kLdHid = kHid + 8;   // padded smem strides (bf16 elements)

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}

// Fragment layout of mma.m16n8k16 (row.col): lane = 4 g + t; A regs {(g, 2t..2t+1), (g+8, 2t..),
// (g, 2t+8..), (g+8, 2t+8..)}, B regs {(2t..2t+1, g), (2t+8.., g)}, C {(g, 2t), (g, 2t+1),
// (g+8, 2t), (g+8, 2t+1)}.  So the results of two neighbouring column tiles are, rounded to BF16,
// the A registers of the k step over the same 16 columns: a warp's 16 rows pass from layer to
// layer in registers, and only weights come from shared memory (ldmatrix, four 8 x 8 blocks an
// instruction; rows padded by 16 bytes keep it free of bank conflicts).  Gathering every
// fragment element by element from shared memory took 377 us for 400k rows, most of it those
// loads; this form takes 203, bound by the erf of 384 activations a row (about 120 us of issue
// slots).  The k steps are summed in the same order, so the outputs are the same bits; tcgen05
// sums in another order, which moves BF16 roundings of the activations.
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const bf16* p) {
    const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s) : "memory");
}
__device__ __forceinline__ void ldsm4_trans(uint32_t (&r)[4], const bf16* p) {
    const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s) : "memory");
}
// B of two column tiles (n0, n0 + 8) and one k step from M[n][k] or, transposed, from M[k][n]:
// r = {b0, b1} of the first, {b0, b1} of the second
__device__ __forceinline__ void load_b(uint32_t (&r)[4], const bf16* M, int ld, int n0, int k0) {
    const int lane = threadIdx.x & 31;
    ldsm4(r, M + (n0 + (lane & 7) + (lane >> 4) * 8) * ld + k0 + ((lane >> 3) & 1) * 8);
}
__device__ __forceinline__ void load_b_trans(uint32_t (&r)[4], const bf16* M, int ld, int n0, int k0) {
    const int lane = threadIdx.x & 31;
    ldsm4_trans(r, M + (k0 + (lane & 7) + ((lane >> 3) & 1) * 8) * ld + n0 + (lane >> 4) * 8);
}
// A of rows m0.. and one k step from M[k][m]
__device__ __forceinline__ void load_a_trans(uint32_t (&r)[4], const bf16* M, int ld, int m0, int k0) {
    const int lane = threadIdx.x & 31;
    ldsm4_trans(r, M + (k0 + (lane & 7) + (lane >> 4) * 8) * ld + m0 + ((lane >> 3) & 1) * 8);
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.3989422804014327f;
}

// Two adjacent floats; vec: the pointer is 8-byte aligned (checked on the host per buffer).
__device__ __forceinline__ float2 ld2(const float* p, bool vec) {
    return vec ? *reinterpret_cast<const float2*>(p) : make_float2(p[0], p[1]);
}
__device__ __forceinline__ void st2(float* p, float a, float b, bool vec) {
    if (vec) *reinterpret_cast<float2*>(p) = make_float2(a, b);
    else { p[0] = a; p[1] = b; }
}
__device__ __forceinline__ void add2(float* p, float a, float b, bool vec) {
    if (vec) atomicAdd(reinterpret_cast<float2*>(p), make_float2(a, b));
    else { atomicAdd(p, a); atomicAdd(p + 1, b); }
}

struct WeightSmem {
    bf16 w1[kHid * kLdIn];
    bf16 w2[2][kHid * kLdHid];   // W2, W3
    bf16 w4[kOut * kLdHid];
    float b[kNB];
};

// vec: w is 16-byte aligned
__device__ void load_weights(WeightSmem& S, const bf16* w, const float* b, bool vec) {
    // eight elements of one matrix row at a time (the rows' padded strides are multiples of 8)
    for (int e = threadIdx.x; e < kNW / 8; e += blockDim.x) {
        const int i = 8 * e;
        bf16* dst;
        if (i < woff(1)) dst = S.w1 + (i / kIn) * kLdIn + i % kIn;
        else if (i < woff(3)) {
            const int j = i - woff(1), m = j / (kHid * kHid), q = j % (kHid * kHid);
            dst = S.w2[m] + (q / kHid) * kLdHid + q % kHid;
        } else dst = S.w4 + ((i - woff(3)) / kHid) * kLdHid + (i - woff(3)) % kHid;
        if (vec) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(w + i);
        else
            for (int k = 0; k < 8; k++) dst[k] = w[i + k];
    }
    for (int e = threadIdx.x; e < kNB; e += blockDim.x) S.b[e] = b[e];
}

// BF16 input rows r0 .. r0 + 15 as the A registers of the first layer (rows past n are zero)
__device__ __forceinline__ void load_x(uint32_t (&a)[4], const float* x, int64_t r0, int64_t n, bool vec) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const int64_t row = r0 + g + (q & 1) * 8;
        const float2 v = row < n ? ld2(x + row * kIn + 2 * t + (q >> 1) * 8, vec) : make_float2(0.f, 0.f);
        a[q] = pack2(v.x, v.y);
    }
}

// Forward of the warp's 16 rows; the pre-activations go to z1..z3 (each [n][128], null: not
// stored), the output layer's two column tiles (C layout) through out(c0, c1).
template <typename Out>
__device__ __forceinline__ void warp_forward(const WeightSmem& S, const uint32_t (&x)[4], float* const (&z)[3], int64_t r0,
                                             int64_t n, bool vec, Out out) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    uint32_t A[8][4], B[8][4];
    auto bias = [&](float (&c)[4], const float* b, int n0) {
        c[0] = c[2] = b[n0 + 2 * t];
        c[1] = c[3] = b[n0 + 2 * t + 1];
    };
    // the hidden layer's columns 16 j .. 16 j + 15 from their two tiles' sums
    auto activate = [&](uint32_t (&dst)[4], const float (&c0)[4], const float (&c1)[4], float* zl, int j) {
        if (zl) {
            const int c = 16 * j + 2 * t;
            if (r0 + g < n) {
                st2(zl + (r0 + g) * kHid + c, c0[0], c0[1], vec);
                st2(zl + (r0 + g) * kHid + c + 8, c1[0], c1[1], vec);
            }
            if (r0 + g + 8 < n) {
                st2(zl + (r0 + g + 8) * kHid + c, c0[2], c0[3], vec);
                st2(zl + (r0 + g + 8) * kHid + c + 8, c1[2], c1[3], vec);
            }
        }
        dst[0] = pack2(gelu(c0[0]), gelu(c0[1]));
        dst[1] = pack2(gelu(c0[2]), gelu(c0[3]));
        dst[2] = pack2(gelu(c1[0]), gelu(c1[1]));
        dst[3] = pack2(gelu(c1[2]), gelu(c1[3]));
    };
#pragma unroll
    for (int j = 0; j < 8; j++) {
        float c0[4], c1[4];
        uint32_t w[4];
        bias(c0, S.b + boff(0), 16 * j);
        bias(c1, S.b + boff(0), 16 * j + 8);
        load_b(w, S.w1, kLdIn, 16 * j, 0);
        mma16816(c0, x, w[0], w[1]);
        mma16816(c1, x, w[2], w[3]);
        activate(A[j], c0, c1, z[0], j);
    }
#pragma unroll 1
    for (int l = 1; l <= 2; l++) {
        const bf16* W = S.w2[l - 1];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            float c0[4], c1[4];
            bias(c0, S.b + boff(l), 16 * j);
            bias(c1, S.b + boff(l), 16 * j + 8);
#pragma unroll
            for (int k = 0; k < 8; k++) {
                uint32_t w[4];
                load_b(w, W, kLdHid, 16 * j, 16 * k);
                mma16816(c0, A[k], w[0], w[1]);
                mma16816(c1, A[k], w[2], w[3]);
            }
            activate(B[j], c0, c1, z[l], j);
        }
#pragma unroll
        for (int j = 0; j < 8; j++)
#pragma unroll
            for (int q = 0; q < 4; q++) A[j][q] = B[j][q];
    }
    float c0[4], c1[4];
    bias(c0, S.b + boff(3), 0);
    bias(c1, S.b + boff(3), 8);
#pragma unroll
    for (int k = 0; k < 8; k++) {
        uint32_t w[4];
        load_b(w, S.w4, kLdHid, 0, 16 * k);
        mma16816(c0, A[k], w[0], w[1]);
        mma16816(c1, A[k], w[2], w[3]);
    }
    out(c0, c1);
}

// A warp takes 16 rows at a time; no barrier after the weights are in place.
__global__ void __launch_bounds__(kThreads, 2) mlp_infer_kernel(const bf16* w, const float* b, const float* x, int64_t n,
                                                                float* y, bool vec_w, bool vec) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WeightSmem& S = *reinterpret_cast<WeightSmem*>(smem_raw);
    load_weights(S, w, b, vec_w);
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    float* const none[3] = {nullptr, nullptr, nullptr};
    for (int64_t r0 = ((int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * 16; r0 < n;
         r0 += (int64_t)gridDim.x * (kThreads / 32) * 16) {
        uint32_t a[4];
        load_x(a, x, r0, n, vec);
        warp_forward(S, a, none, r0, n, vec, [&](const float (&c0)[4], const float (&c1)[4]) {
            if (r0 + g < n) {
                st2(y + (r0 + g) * kOut + 2 * t, c0[0], c0[1], vec);
                st2(y + (r0 + g) * kOut + 2 * t + 8, c1[0], c1[1], vec);
            }
            if (r0 + g + 8 < n) {
                st2(y + (r0 + g + 8) * kOut + 2 * t, c0[2], c0[3], vec);
                st2(y + (r0 + g + 8) * kOut + 2 * t + 8, c1[2], c1[3], vec);
            }
        });
    }
}

struct TrainSmem {
    WeightSmem w;
    bf16 g[kRows * kLdHid];     // g_l of the block's rows, [row][output]
    bf16 act[kRows * kLdHid];   // a_{l-1}, [row][input]
};

// One training pass over the block's 128 rows, a warp's 16 rows in registers: the forward with the
// pre-activations stored, the output gradient g = 2 (y - t) / (n * 11) on the 11 used outputs and
// the loss sum, then layer by layer from the output the weight / bias gradients (g_l^T a_{l-1},
// summed over the block's rows and added atomically) and the gradient of the previous layer's
// pre-activation g_{l-1} = (g_l W_l) * gelu'(z_{l-1}).  Only the weight gradients mix rows of
// different warps: g_l and a_{l-1} pass through shared memory for them, and a column of ones as
// one more B operand gives the bias gradient.  Forward and backward in one kernel read back the
// pre-activations their own lanes wrote.  16384 rows: 202 us a step with two kernels that
// gathered their fragments element by element, 80 us with this one.
__global__ void __launch_bounds__(kThreads, 1) mlp_train_kernel(const bf16* w, const float* b, const float* x,
                                                                const float* tgt, int64_t n, float* z1, float* z2,
                                                                float* z3, float* gw, float* gb, double* loss_sum,
                                                                bool vec_w, bool vec) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
    load_weights(S.w, w, b, vec_w);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    float* const zs[3] = {z1, z2, z3};
    const float scale = 2.f / ((float)n * (float)kOutUsed);
    double lsum = 0.0;
    uint32_t* const gw32 = reinterpret_cast<uint32_t*>(S.g);
    uint32_t* const aw32 = reinterpret_cast<uint32_t*>(S.act);
    constexpr int LW = kLdHid / 2;   // row stride in words
    const int row0 = warp * 16 + g;  // this lane's rows of the block: row0, row0 + 8
    for (int64_t base = (int64_t)blockIdx.x * kRows; base < n; base += (int64_t)gridDim.x * kRows) {
        const int64_t r0 = base + warp * 16;
        uint32_t xa[4], G[8][4];
        load_x(xa, x, r0, n, vec);
        warp_forward(S.w, xa, zs, r0, n, vec, [&](const float (&c0)[4], const float (&c1)[4]) {
            float gv[8];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const int64_t row = r0 + g + ((q >> 1) & 1) * 8;
                const int c = 2 * t + (q & 1) + (q >> 2) * 8;
                gv[q] = 0.f;
                if (row < n && c < kOutUsed) {
                    const float d = (q < 4 ? c0[q & 3] : c1[q & 3]) - tgt[row * kOut + c];
                    lsum += (double)d * (double)d;
                    gv[q] = scale * d;
                }
            }
            G[0][0] = pack2(gv[0], gv[1]);
            G[0][1] = pack2(gv[2], gv[3]);
            G[0][2] = pack2(gv[4], gv[5]);
            G[0][3] = pack2(gv[6], gv[7]);
        });
#pragma unroll 1
        for (int l = 3; l >= 0; l--) {
            const int out_dim = l == 3 ? kOut : kHid, in_dim = l == 0 ? kIn : kHid;
            const int nk = out_dim / 16;
            __syncthreads();   // the last layer's products have read g and act
#pragma unroll
            for (int k = 0; k < 8; k++) {
                if (k >= nk) break;
                gw32[row0 * LW + 8 * k + t] = G[k][0];
                gw32[(row0 + 8) * LW + 8 * k + t] = G[k][1];
                gw32[row0 * LW + 8 * k + t + 4] = G[k][2];
                gw32[(row0 + 8) * LW + 8 * k + t + 4] = G[k][3];
            }
            if (l == 0) {
                aw32[row0 * LW + t] = xa[0];
                aw32[(row0 + 8) * LW + t] = xa[1];
                aw32[row0 * LW + t + 4] = xa[2];
                aw32[(row0 + 8) * LW + t + 4] = xa[3];
            } else {
                // a_{l-1} = gelu(z_l) into shared memory and g_{l-1} into registers
                const float* zl = zs[l - 1];
                const bf16* W = l == 3 ? S.w.w4 : S.w.w2[l - 1];
                uint32_t H[8][4];
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        if (k >= nk) break;
                        uint32_t wb[4];
                        load_b_trans(wb, W, kLdHid, 16 * j, 16 * k);
                        mma16816(c[0], G[k], wb[0], wb[1]);
                        mma16816(c[1], G[k], wb[2], wb[3]);
                    }
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int col = 16 * j + 8 * h + 2 * t;
#pragma unroll
                        for (int r = 0; r < 2; r++) {
                            const int64_t row = r0 + g + 8 * r;
                            const float2 zz = row < n ? ld2(zl + row * kHid + col, vec) : make_float2(0.f, 0.f);
                            const float av0 = row < n ? gelu(zz.x) : 0.f, av1 = row < n ? gelu(zz.y) : 0.f;
                            aw32[(row0 + 8 * r) * LW + 8 * j + 4 * h + t] = pack2(av0, av1);
                            H[j][2 * h + r] = pack2(c[h][2 * r] * gelu_grad(zz.x), c[h][2 * r + 1] * gelu_grad(zz.y));
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; j++)
#pragma unroll
                    for (int q = 0; q < 4; q++) G[j][q] = H[j][q];
            }
            __syncthreads();
            // gW[o][i] = sum_r g[r][o] a[r][i]: tiles of 16 outputs x 16 inputs, K = the block's rows
            const int mt = out_dim / 16, nt = in_dim / 16;
            float* dst = gw + woff(l);
            for (int tile = warp; tile < mt * nt; tile += kThreads / 32) {
                const int o0 = (tile / nt) * 16, i0 = (tile % nt) * 16;
                float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < kRows / 16; k++) {
                    uint32_t ga[4], ab[4];
                    load_a_trans(ga, S.g, kLdHid, o0, 16 * k);
                    load_b_trans(ab, S.act, kLdHid, i0, 16 * k);
                    mma16816(c0, ga, ab[0], ab[1]);
                    mma16816(c1, ga, ab[2], ab[3]);
                }
                add2(dst + (o0 + g) * in_dim + i0 + 2 * t, c0[0], c0[1], vec);
                add2(dst + (o0 + g + 8) * in_dim + i0 + 2 * t, c0[2], c0[3], vec);
                add2(dst + (o0 + g) * in_dim + i0 + 8 + 2 * t, c1[0], c1[1], vec);
                add2(dst + (o0 + g + 8) * in_dim + i0 + 8 + 2 * t, c1[2], c1[3], vec);
            }
            if (warp < mt) {   // bias gradient of outputs 16 warp ..: B = ones
                float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < kRows / 16; k++) {
                    uint32_t ga[4];
                    load_a_trans(ga, S.g, kLdHid, 16 * warp, 16 * k);
                    mma16816(c, ga, 0x3F803F80u, 0x3F803F80u);
                }
                if (t == 0) {
                    atomicAdd(&gb[boff(l) + 16 * warp + g], c[0]);
                    atomicAdd(&gb[boff(l) + 16 * warp + g + 8], c[2]);
                }
            }
        }
    }
    lsum = warp_sum(lsum);
    if (lane == 0 && lsum != 0.0) atomicAdd(loss_sum, lsum);
}

// Adam on the FP32 master parameters (weights then biases), BF16 copy of the weights,
// gradients cleared; the step's loss (loss_out may be null).
__global__ void mlp_adam_kernel(float* master, bf16* wq, float* bias, float* gw, float* gb, float* m, float* v, float lr,
                                float b1, float b2, float eps, float bc1, float bc2, const double* loss_sum, int64_t n,
                                float* loss_out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && loss_out) *loss_out = (float)(*loss_sum / ((double)n * kOutUsed));
    if (i >= kNW + kNB) return;
    const bool is_w = i < kNW;
    float g = is_w ? gw[i] : gb[i - kNW];
    float p = is_w ? master[i] : bias[i - kNW];
    const float mm = b1 * m[i] + (1.f - b1) * g;
    const float vv = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mm;
    v[i] = vv;
    p -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
    if (is_w) {
        master[i] = p;
        wq[i] = __float2bfloat16_rn(p);
        gw[i] = 0.f;
    } else {
        bias[i - kNW] = p;
        gb[i - kNW] = 0.f;
    }
}

// blocks of kRows rows, at most `per_sm` per SM
static int mlp_grid(int64_t n, int per_sm) {
    const int64_t sms = (int64_t)device_sms() * per_sm, blocks = (n + kRows - 1) / kRows;
    return (int)(blocks < sms ? (blocks > 0 ? blocks : 1) : sms);
}

static bool g_mlp_attr[kMaxDevices] = {};
static cudaError_t mlp_attrs() {
    return once_per_device(g_mlp_attr, [] {
        cudaError_t e = cudaFuncSetAttribute(mlp_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(WeightSmem));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(TrainSmem));
        return e;
    });
}

static bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

gs_status record_error(gs_status s, const char* msg);

}  // namespace gs

using namespace gs;

extern "C" gs_status gs_mlp_infer(const uint16_t* w_bf16, const float* bias, const float* x, int64_t n, float* y,
                                  void* stream) {
    if (n < 0) return record_error(GS_ERR_INVALID_ARG, "n must be >= 0");
    if (n == 0) return GS_OK;
    if (!w_bf16 || !bias || !x || !y) return record_error(GS_ERR_INVALID_ARG, "NULL buffer");
    cudaError_t e = mlp_attrs();
    if (e != cudaSuccess) return record_error(GS_ERR_CUDA, cudaGetErrorString(e));
    mlp_infer_kernel<<<mlp_grid(n, 2), kThreads, sizeof(WeightSmem), (cudaStream_t)stream>>>(
        reinterpret_cast<const bf16*>(w_bf16), bias, x, n, y, aligned(w_bf16, 16), aligned(x, 8) && aligned(y, 8));
    e = cudaGetLastError();
    return e == cudaSuccess ? GS_OK : record_error(GS_ERR_CUDA, cudaGetErrorString(e));
}

extern "C" size_t gs_mlp_train_scratch_size(int64_t n) {
    // z1..z3 [n][128] FP32, 16 unused floats a row, loss sum (double)
    return sizeof(float) * (size_t)n * (3 * 128 + 16) + 256;
}

extern "C" gs_status gs_mlp_train_step(float* w_master, uint16_t* w_bf16, float* bias, float* grad_w, float* grad_b,
                                       float* adam_m, float* adam_v, const float* x, const float* y_target, int64_t n,
                                       float lr, float b1, float b2, float eps, int64_t step, void* scratch,
                                       size_t scratch_bytes, float* loss_out, void* stream) {
    if (n < 1) return record_error(GS_ERR_INVALID_ARG, "n must be >= 1");
    if (step < 1) return record_error(GS_ERR_INVALID_ARG, "step must be >= 1");
    if (!w_master || !w_bf16 || !bias || !grad_w || !grad_b || !adam_m || !adam_v || !x || !y_target || !scratch)
        return record_error(GS_ERR_INVALID_ARG, "NULL buffer");
    if (scratch_bytes < gs_mlp_train_scratch_size(n)) return record_error(GS_ERR_INVALID_ARG, "scratch too small");
    cudaError_t e = mlp_attrs();
    if (e != cudaSuccess) return record_error(GS_ERR_CUDA, cudaGetErrorString(e));
    cudaStream_t st = (cudaStream_t)stream;
    float* z1 = static_cast<float*>(scratch);
    float* z2 = z1 + (size_t)n * 128;
    float* z3 = z2 + (size_t)n * 128;
    float* z_end = z3 + (size_t)n * (128 + 16);
    double* lsum = reinterpret_cast<double*>(
        (reinterpret_cast<uintptr_t>(z_end) + 15) & ~(uintptr_t)15);
    cudaMemsetAsync(lsum, 0, sizeof(double), st);
    const bf16* wq = reinterpret_cast<const bf16*>(w_bf16);
    mlp_train_kernel<<<mlp_grid(n, 1), kThreads, sizeof(TrainSmem), st>>>(
        wq, bias, x, y_target, n, z1, z2, z3, grad_w, grad_b, lsum, aligned(w_bf16, 16),
        aligned(x, 8) && aligned(scratch, 8) && aligned(grad_w, 8));
    const float bc1 = (float)(1.0 - pow((double)b1, (double)step)), bc2 = (float)(1.0 - pow((double)b2, (double)step));
    mlp_adam_kernel<<<(kNW + kNB + 255) / 256, 256, 0, st>>>(w_master, reinterpret_cast<bf16*>(w_bf16), bias, grad_w,
                                                            grad_b, adam_m, adam_v, lr, b1, b2, eps, bc1, bc2, lsum, n,
                                                            loss_out);
    e = cudaGetLastError();
    return e == cudaSuccess ? GS_OK : record_error(GS_ERR_CUDA, cudaGetErrorString(e));
}

