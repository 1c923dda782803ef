// mlp.cu -- the learned warm start: a 5 -> 128 -> 128 -> 128 -> 128 -> 1 SiLU
// network trained and evaluated on the GPU by the library's own kernels (BF16
// operands on the tensor cores, FP32 accumulation, FP32 master weights, Adam),
// and lbm_init_droplet_learned, which starts a droplet from the network's
// steady-profile prediction instead of the tanh profile.
//
// Parameter vector (FP32, compact): W1 [5][128], b1, W2 [128][128], b2, W3, b3,
// W4, b4, W5 [128][1], b5; z_l = h_{l-1} W_l + b_l, h_l = silu(z_l), y = h_4 W_5 + b_5.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/lbm.h"
#include "internal.h"
#include "trace.h"

namespace lbm {

// Feature scaling of the warm-start network (shared by training data and inference).
// The radius enters as the curvature 10/R: the steady profile depends on R
// through the Laplace pressure sigma/R, and a droplet larger than any trained
// one then lies next to the trained range (curvature near 0) instead of far
// outside it.  The curvature is capped at that of R = 5, below the smallest
// trained droplets, so that the small radii the mass bisection tries stay in
// range.  d spans the interface and the bulk plateaus on both sides.
__host__ __device__ inline void mlp_features(double G, double tau, double order, double R, double d, float* x)
{
    const double kappa = R > 5.0 ? 10.0 / R : 2.0;
    x[0] = (float)((G + 4.9) / 0.6);
    x[1] = (float)((tau - 0.8) / 0.2);
    x[2] = (float)((order - 7.0) / 3.0);
    x[3] = (float)((kappa - 0.5) / 0.4);
    x[4] = (float)(d / kMlpDmax);
}

namespace {

using bf16 = __nv_bfloat16;

constexpr int kIn = 5, kH = 128, kLayers = 5;
constexpr int kInPad = 16, kOutPad = 8;

__host__ __device__ constexpr int kFanD(int l) { return l == 0 ? kIn : (l == kLayers ? 1 : kH); }
__host__ __device__ constexpr long long param_offset_w(int l)
{
    long long o = 0;
    for (int i = 0; i < l; ++i) o += (long long)kFanD(i) * kFanD(i + 1) + kFanD(i + 1);
    return o;
}
__host__ __device__ constexpr long long param_offset_b(int l)
{
    return param_offset_w(l) + (long long)kFanD(l) * kFanD(l + 1);
}
constexpr long long kNParam = param_offset_w(kLayers);
static_assert(kNParam == 50433, "parameter count");

// padded GEMM shapes of layer l: [K_l][N_l]
constexpr int kK[kLayers] = {kInPad, kH, kH, kH, kH};
constexpr int kN[kLayers] = {kH, kH, kH, kH, kOutPad};

// ---- BF16 tensor-core pieces ------------------------------------------------------
// mma.sync m16n8k16 (row.col, bf16, f32 accumulators), operands from padded
// shared-memory tiles by ldmatrix.  Every product accumulates its K in steps of
// 16 in rising order, so a result does not depend on how the tiles are split.
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t s32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
// 16-byte asynchronous copy; `bytes` < 16 fills the rest with zeros.
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float silu_f(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float silu_grad_f(float z)
{
    const float s = 1.f / (1.f + __expf(-z));
    return s * (1.f + z * (1.f - s));
}

// ---- one pass through the network for a tile of rows ---------------------------------
// A block keeps all weights (107 KB of BF16) in shared memory and takes tiles of
// 32 rows through every layer, and in training back again to dZ_1, without
// leaving the SM: the 4096 x 128 x 128 products are too small to be launched
// layer by layer (a training step was some 40 launches of 2 to 400 us).  With 32
// rows a 4096-row batch gives 128 blocks, one per SM; eight warps split a tile
// into 16 x 32 pieces.  Forward and backward of 4096 rows, with the activations
// and dZ written for the weight gradients: see k_mlp_grad for the times.
constexpr int kTileRows = 32;
constexpr int kPassThreads = 256;
constexpr int kPitch = 136;   // bf16 row pitch of weights and activations (272 B: ldmatrix without conflicts)
constexpr int kZPitch = 132;  // f32 row pitch of the pre-activations

struct NetView {
    const bf16* W[kLayers];  // padded [kK][kN]
    const float* b[kLayers];
};
struct PassIn {      // where a row's features come from
    const float* X;  // [rows][5], or nullptr: a table of signed distances
    double G, tau, order, r_in, dmax;
    const double* R;  // table: radius of each candidate; row r is distance r % T of candidate r / T
    int T;
};
struct TrainBuf {  // per batch row; what the weight and bias gradients read
    const float* t;
    bf16* Xp;        // [rows][16]
    bf16* h[4];      // [rows][128] activations
    bf16* dZ[4];     // [rows][128]
    float* dZ32[4];  // the same in f32, for the bias gradients
    float* err;      // y - t
    float* dY;       // 2 (y - t) / rows
    bf16* dYb;       // [rows][kOutPad], column 0: a 16-byte row for the asynchronous copies
};

struct PassSmem {
    bf16 w1[kInPad][kPitch];
    bf16 w[3][kH][kPitch];
    bf16 w5[kH];
    float g[kTileRows];
    bf16 h[2][kTileRows][kPitch];
};
constexpr size_t kPassBytes = sizeof(PassSmem);
constexpr size_t kTrainBytes = sizeof(PassSmem) + sizeof(float) * 4 * kTileRows * kZPitch;

template <bool TRAIN>
__global__ void __launch_bounds__(kPassThreads, 1) k_mlp_pass(NetView net, PassIn in, int rows, float* __restrict__ y,
                                                              TrainBuf tb)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    PassSmem& sm = *reinterpret_cast<PassSmem*>(smem_raw);
    float* zs = reinterpret_cast<float*>(smem_raw + sizeof(PassSmem));  // [4][32][kZPitch], training only
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = (warp & 1) * 16, wn = (warp >> 1) * 32;
    const int g = lane >> 2, t = lane & 3;

    // weights: rows of 256 bytes, 16 copies each
    for (int i = tid; i < kInPad * 16; i += kPassThreads)
        cp16(s32(&sm.w1[i >> 4][(i & 15) * 8]), net.W[0] + (i >> 4) * kH + (i & 15) * 8, 16);
    cp_commit();
    for (int l = 0; l < 3; ++l) {  // a group per layer: the first layer starts on its own weights
        for (int i = tid; i < kH * 16; i += kPassThreads)
            cp16(s32(&sm.w[l][i >> 4][(i & 15) * 8]), net.W[l + 1] + (i >> 4) * kH + (i & 15) * 8, 16);
        cp_commit();
    }
    if (tid < kH) sm.w5[tid] = net.W[4][tid * kOutPad];

    // acc = A W (A: 32 x K tile of activations) for this warp's 16 x 32 piece
    auto product = [&](const bf16* A, const bf16* W, int K, float (&acc)[4][4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
        const uint32_t aa = s32(A + (wm + (lane & 15)) * kPitch + (lane >> 4) * 8);
        const uint32_t wa = s32(W + (lane & 15) * kPitch + wn + (lane >> 4) * 8);
        for (int k0 = 0; k0 < K; k0 += 16) {
            uint32_t a[4], b0[4], b1[4];
            ldsm4(a, aa + k0 * 2);
            ldsm4t(b0, wa + k0 * kPitch * 2);
            ldsm4t(b1, wa + k0 * kPitch * 2 + 32);
            mma_bf16(acc[0], a, b0[0], b0[1]);
            mma_bf16(acc[1], a, b0[2], b0[3]);
            mma_bf16(acc[2], a, b1[0], b1[1]);
            mma_bf16(acc[3], a, b1[2], b1[3]);
        }
    };
    // acc = A W^T
    auto product_t = [&](const bf16* A, const bf16* W, float (&acc)[4][4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
        const uint32_t aa = s32(A + (wm + (lane & 15)) * kPitch + (lane >> 4) * 8);
        const uint32_t wa = s32(W + (wn + (lane >> 4) * 8 + (lane & 7)) * kPitch + ((lane >> 3) & 1) * 8);
        for (int k0 = 0; k0 < kH; k0 += 16) {
            uint32_t a[4], b0[4], b1[4];
            ldsm4(a, aa + k0 * 2);
            ldsm4(b0, wa + k0 * 2);
            ldsm4(b1, wa + 16 * kPitch * 2 + k0 * 2);
            mma_bf16(acc[0], a, b0[0], b0[1]);
            mma_bf16(acc[1], a, b0[2], b0[3]);
            mma_bf16(acc[2], a, b1[0], b1[1]);
            mma_bf16(acc[3], a, b1[2], b1[3]);
        }
    };

    const int ntiles = (rows + kTileRows - 1) / kTileRows;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int r0 = tile * kTileRows;
        if (tid < kTileRows) {
            const int r = r0 + tid;
            float x[kIn] = {};
            if (r < rows) {
                if (in.X) {
                    for (int c = 0; c < kIn; ++c) x[c] = in.X[(long long)r * kIn + c];
                } else {
                    const int k = r % in.T;
                    const double d = -in.dmax + 2.0 * in.dmax * k / (in.T - 1);
                    mlp_features(in.G, in.tau, in.order, in.r_in * in.R[r / in.T], d, x);
                }
            }
            for (int c = 0; c < kInPad; ++c) {
                const bf16 v = __float2bfloat16(c < kIn ? x[c] : 0.f);
                sm.h[0][tid][c] = v;
                if (TRAIN && r < rows) tb.Xp[(long long)r * kInPad + c] = v;
            }
        }
        cp_wait<3>();  // the first layer's weights, first time round
        __syncthreads();
        int cur = 0;
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            float acc[4][4];
            product(&sm.h[cur][0][0], l == 0 ? &sm.w1[0][0] : &sm.w[l == 0 ? 0 : l - 1][0][0],
                    l == 0 ? kInPad : kH, acc);
#pragma unroll
            for (int ni = 0; ni < 4; ++ni) {
                const int c = wn + ni * 8 + 2 * t;
                const float2 bias = __ldg(reinterpret_cast<const float2*>(net.b[l] + c));
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int r = wm + g + hf * 8;
                    const float z0 = acc[ni][2 * hf] + bias.x, z1 = acc[ni][2 * hf + 1] + bias.y;
                    if (TRAIN) *reinterpret_cast<float2*>(zs + (l * kTileRows + r) * kZPitch + c) = make_float2(z0, z1);
                    __nv_bfloat162 hv;
                    hv.x = __float2bfloat16(silu_f(z0));
                    hv.y = __float2bfloat16(silu_f(z1));
                    *reinterpret_cast<__nv_bfloat162*>(&sm.h[cur ^ 1][r][c]) = hv;
                    if (TRAIN && r0 + r < rows)
                        *reinterpret_cast<__nv_bfloat162*>(tb.h[l] + (long long)(r0 + r) * kH + c) = hv;
                }
            }
            cur ^= 1;
            if (l == 0) cp_wait<2>();
            if (l == 1) cp_wait<1>();
            if (l == 2) cp_wait<0>();
            __syncthreads();
        }
        if (wn == 0) {  // output column, one warp per 16 rows
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            const uint32_t aa = s32(&sm.h[cur][wm + (lane & 15)][(lane >> 4) * 8]);
            for (int k0 = 0; k0 < kH; k0 += 16) {
                uint32_t a[4], b0 = 0, b1 = 0;
                ldsm4(a, aa + k0 * 2);
                if (g == 0) {
                    b0 = *reinterpret_cast<const uint32_t*>(&sm.w5[k0 + 2 * t]);
                    b1 = *reinterpret_cast<const uint32_t*>(&sm.w5[k0 + 2 * t + 8]);
                }
                mma_bf16(acc, a, b0, b1);
            }
            if (t == 0) {
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int rl = wm + g + hf * 8, r = r0 + rl;
                    const float v = acc[2 * hf] + net.b[4][0];
                    float gr = 0.f;
                    if (r < rows) {
                        if (y) y[r] = v;
                        if (TRAIN) {
                            const float e = v - tb.t[r];
                            gr = 2.f * e / rows;
                            tb.err[r] = e;
                            tb.dY[r] = gr;
                            uint4 row = make_uint4(0u, 0u, 0u, 0u);
                            row.x = __bfloat16_as_ushort(__float2bfloat16(gr));
                            *reinterpret_cast<uint4*>(tb.dYb + (long long)r * kOutPad) = row;
                        }
                    }
                    if (TRAIN) sm.g[rl] = __bfloat162float(__float2bfloat16(gr));
                }
            }
        }
        __syncthreads();
        if constexpr (TRAIN) {
#pragma unroll
            for (int l = 3; l >= 0; --l) {  // dH_l, then dZ_l = dH_l silu'(Z_l)
                float acc[4][4];
                if (l < 3) product_t(&sm.h[cur][0][0], &sm.w[l][0][0], acc);
#pragma unroll
                for (int ni = 0; ni < 4; ++ni) {
                    const int c = wn + ni * 8 + 2 * t;
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        const int r = wm + g + hf * 8;
                        float d0, d1;
                        if (l == 3) {  // the output layer's product has one column: exact in f32
                            d0 = sm.g[r] * __bfloat162float(sm.w5[c]);
                            d1 = sm.g[r] * __bfloat162float(sm.w5[c + 1]);
                        } else {
                            d0 = acc[ni][2 * hf];
                            d1 = acc[ni][2 * hf + 1];
                        }
                        const float2 z = *reinterpret_cast<const float2*>(zs + (l * kTileRows + r) * kZPitch + c);
                        const float v0 = d0 * silu_grad_f(z.x), v1 = d1 * silu_grad_f(z.y);
                        __nv_bfloat162 dv;
                        dv.x = __float2bfloat16(v0);
                        dv.y = __float2bfloat16(v1);
                        *reinterpret_cast<__nv_bfloat162*>(&sm.h[cur ^ 1][r][c]) = dv;
                        if (r0 + r < rows) {
                            const long long o = (long long)(r0 + r) * kH + c;
                            *reinterpret_cast<__nv_bfloat162*>(tb.dZ[l] + o) = dv;
                            *reinterpret_cast<float2*>(tb.dZ32[l] + o) = make_float2(v0, v1);
                        }
                    }
                }
                cur ^= 1;
                __syncthreads();
            }
        }
    }
    cp_wait<0>();  // a block without a tile leaves no copy in flight
}

// ---- weight and bias gradients, and the loss, of one batch -------------------------------
// dW_l = h_{l-1}^T dZ_l sums over the batch rows.  Each 32 x 32 piece of a dW, each
// group of 32 columns of a db and the loss are one block that streams its columns
// of the batch through shared memory (cp.async, chunks of 64 rows): 74 blocks, so
// all layers run at once and a sum still runs over the rows in order.  Bounded by
// that order: 256 dependent mma steps for a dW, 4096 dependent additions for a db.
// Eight chunks of 64 rows are in flight per block, and all parts
// come by asynchronous copies; W5's, a value a row, were loaded and stored by the
// threads, a memory latency per chunk.  Two training steps of 4096 rows, all kernels
// and copies: 3.94 ms -> 0.22 ms.
constexpr int kChunk = 64, kGStages = 8, kCPitch = 40;
constexpr size_t kGradBytes = sizeof(bf16) * kGStages * 2 * kChunk * kCPitch;  // 80 KB in flight per block
constexpr int kGradGemms = 3 * 16 + 4 + 4;  // 32 x 32 pieces of W2..W4, W1, W5
constexpr int kGradJobs = kGradGemms + 4 * 4 + 1 + 1;

__global__ void __launch_bounds__(128) k_mlp_grad(TrainBuf tb, int rows, float* __restrict__ grad,
                                                  double* __restrict__ loss)
{
    extern __shared__ __align__(128) unsigned char buf[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int job = blockIdx.x;
    const int nchunk = (rows + kChunk - 1) / kChunk;
    if (job < kGradGemms) {
        int l, m0, n0;
        if (job < 48) {
            l = 1 + job / 16;
            m0 = (job % 16) / 4 * 32;
            n0 = job % 4 * 32;
        } else if (job < 52) {
            l = 0;
            m0 = 0;
            n0 = (job - 48) * 32;
        } else {
            l = 4;
            m0 = (job - 52) * 32;
            n0 = 0;
        }
        const bf16* A = l == 0 ? tb.Xp : tb.h[l - 1];
        const int lda = l == 0 ? kInPad : kH;
        const bf16* Bm = l == 4 ? tb.dYb : tb.dZ[l];
        bf16(*As)[kChunk][kCPitch] = reinterpret_cast<bf16(*)[kChunk][kCPitch]>(buf);
        bf16(*Bs)[kChunk][kCPitch] = As + kGStages;
        if (l == 4) {  // one column, copied with its zero neighbours; zeros beyond
            for (int i = tid; i < kGStages * kChunk * kCPitch; i += 128) (&Bs[0][0][0])[i] = __float2bfloat16(0.f);
            __syncthreads();
        }
        auto load = [&](int c) {
            if (c < nchunk) {
                const int st = c % kGStages;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int idx = tid + i * 128, r = idx >> 2, q = (idx & 3) * 8;
                    const long long gr = (long long)c * kChunk + r;
                    const bool in = gr < rows;
                    const bool av = in && m0 + q < lda;
                    cp16(s32(&As[st][r][q]), av ? A + gr * lda + m0 + q : A, av ? 16 : 0);
                    if (l != 4) cp16(s32(&Bs[st][r][q]), in ? Bm + gr * kH + n0 + q : Bm, in ? 16 : 0);
                }
                if (l == 4 && tid < kChunk) {
                    const long long gr = (long long)c * kChunk + tid;
                    cp16(s32(&Bs[st][tid][0]), gr < rows ? Bm + gr * kOutPad : Bm, gr < rows ? 16 : 0);
                }
            }
            cp_commit();
        };
        for (int c = 0; c < kGStages - 1; ++c) load(c);
        const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
        float acc[2][4] = {};
        for (int c = 0; c < nchunk; ++c) {
            cp_wait<kGStages - 2>();
            __syncthreads();
            load(c + kGStages - 1);  // the stage consumed in the previous round
            const int st = c % kGStages;
            const uint32_t aa = s32(&As[st][(lane >> 4) * 8 + (lane & 7)][wm + ((lane >> 3) & 1) * 8]);
            const uint32_t ba = s32(&Bs[st][lane & 15][wn + (lane >> 4) * 8]);
#pragma unroll
            for (int k0 = 0; k0 < kChunk; k0 += 16) {
                uint32_t a[4], b[4];
                ldsm4t(a, aa + k0 * kCPitch * 2);
                ldsm4t(b, ba + k0 * kCPitch * 2);
                mma_bf16(acc[0], a, b[0], b[1]);
                mma_bf16(acc[1], a, b[2], b[3]);
            }
        }
        cp_wait<0>();
        const int K = kFanD(l), N = kFanD(l + 1);
        float* dst = grad + param_offset_w(l);
#pragma unroll
        for (int ni = 0; ni < 2; ++ni)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int m = m0 + wm + (lane >> 2) + ((e & 2) ? 8 : 0);
                const int nn = n0 + wn + ni * 8 + 2 * (lane & 3) + (e & 1);
                if (m < K && nn < N) dst[m * N + nn] = acc[ni][e];
            }
    } else if (job < kGradGemms + 16) {  // 32 columns of db_1 .. db_4, rows in order
        const int l = (job - kGradGemms) / 4, c0 = (job - kGradGemms) % 4 * 32;
        const float* Z = tb.dZ32[l];
        float(*Zs)[kChunk][32] = reinterpret_cast<float(*)[kChunk][32]>(buf);
        auto load = [&](int c) {
            if (c < nchunk)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int idx = tid + i * 128, r = idx >> 3, q = (idx & 7) * 4;
                    const long long gr = (long long)c * kChunk + r;
                    cp16(s32(&Zs[c % kGStages][r][q]), gr < rows ? Z + gr * kH + c0 + q : Z, gr < rows ? 16 : 0);
                }
            cp_commit();
        };
        for (int c = 0; c < kGStages - 1; ++c) load(c);
        float s = 0.f;
        for (int c = 0; c < nchunk; ++c) {
            cp_wait<kGStages - 2>();
            __syncthreads();
            load(c + kGStages - 1);
            if (tid < 32) {
                const int nr = rows - c * kChunk < kChunk ? rows - c * kChunk : kChunk;
                if (nr == kChunk) {
#pragma unroll
                    for (int r = 0; r < kChunk; ++r) s += Zs[c % kGStages][r][tid];
                } else {
                    for (int r = 0; r < nr; ++r) s += Zs[c % kGStages][r][tid];
                }
            }
        }
        cp_wait<0>();
        if (tid < 32) grad[param_offset_b(l) + c0 + tid] = s;
    } else if (job == kGradGemms + 16) {  // db_5
        float* ys = reinterpret_cast<float*>(buf);
        constexpr int kPart = 2048;
        float s = 0.f;
        for (int r0 = 0; r0 < rows; r0 += kPart) {
            const int nr = rows - r0 < kPart ? rows - r0 : kPart;
            __syncthreads();
            for (int i = tid; i < nr; i += 128) ys[i] = tb.dY[r0 + i];
            __syncthreads();
            if (tid == 0) {
#pragma unroll 32
                for (int i = 0; i < nr; ++i) s += ys[i];
            }
        }
        if (tid == 0) grad[param_offset_b(4)] = s;
    } else {  // loss: sums of 256 rows by a tree, then in order
        double* sh = reinterpret_cast<double*>(buf);
        auto sq = [&](int r) {
            if (r >= rows) return 0.0;
            const float e = tb.err[r];
            return (double)e * e;
        };
        double total = 0.0;
        for (int r0 = 0; r0 < rows; r0 += 256) {
            sh[tid] = sq(r0 + tid) + sq(r0 + tid + 128);
            __syncthreads();
            for (int s = 64; s > 0; s >>= 1) {
                if (tid < s) sh[tid] += sh[tid + s];
                __syncthreads();
            }
            if (tid == 0) total += sh[0];
            __syncthreads();
        }
        if (tid == 0) {
            const double v = total / rows;
            loss[0] += v;  // epoch sum: batches follow one another on the stream
            loss[1] = v;
        }
    }
}

// Where the BF16 copy of parameter i lives (nullptr: a bias).
__device__ __forceinline__ bf16* packed_slot(const NetView& net, int i)
{
    int l = 0;
#pragma unroll
    for (int q = 1; q < kLayers; ++q)
        if (i >= param_offset_w(q)) l = q;
    const int j = i - static_cast<int>(param_offset_w(l));
    const int K = kFanD(l), N = kFanD(l + 1);
    if (j >= K * N) return nullptr;
    return const_cast<bf16*>(net.W[l]) + (j / N) * (l == kLayers - 1 ? kOutPad : kH) + j % N;
}

// Adam (bias-corrected) on the FP32 master vector, and the BF16 copies of the weights.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2,
                       NetView net)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    if (bf16* w = packed_slot(net, i)) *w = __float2bfloat16(p[i]);
}

// BF16 padded weights [Kp][Np] from the compact master vector.
__global__ void k_pack_weights(const float* __restrict__ master, long long off, int K, int N, int Kp, int Np,
                               bf16* __restrict__ Wp)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Kp * Np) return;
    const int k = i / Np, n = i % Np;
    Wp[i] = __float2bfloat16((k < K && n < N) ? master[off + (long long)k * N + n] : 0.f);
}

inline unsigned blocks(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

}  // namespace lbm

using namespace lbm;

struct lbm_mlp {
    int device;
    cudaStream_t stream;
    uint64_t seed;
    long long adam_t;
    float* master;   // [kNParam]
    float* grad;     // [kNParam]
    float* m;
    float* v;
    bf16* W[kLayers];   // padded bf16 weights [kK][kN]
    float* b[kLayers];  // views into master
    // Work areas, one allocation each, kept until a larger one is needed.
    int icap;           // rows of the inference area
    float* Xi;          // [icap][5] features, then [icap] outputs
    int tcap;           // rows of the training area
    void* train;
    float* Xt;          // [tcap][5] features of the batch, then [tcap] targets
    TrainBuf tb;
    double* loss;       // epoch sum, last batch
    float* stage[2];    // pinned copies of a batch's features and targets
    cudaEvent_t staged[2];

    NetView view() const
    {
        NetView n;
        for (int l = 0; l < kLayers; ++l) {
            n.W[l] = W[l];
            n.b[l] = b[l];
        }
        return n;
    }
};

namespace {

#define MCK(call)                                                                                        \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess) return set_last_error(LBM_ECUDA, cudaGetErrorString(e_));                 \
    } while (0)

void free_train(lbm_mlp* n)
{
    cudaFree(n->train);
    for (int k = 0; k < 2; ++k) {
        if (n->stage[k]) cudaFreeHost(n->stage[k]);
        if (n->staged[k]) cudaEventDestroy(n->staged[k]);
        n->stage[k] = nullptr;
        n->staged[k] = nullptr;
    }
    n->train = nullptr;
    n->tcap = 0;
}

int ensure_infer(lbm_mlp* n, int rows)
{
    if (rows <= n->icap) return LBM_OK;
    cudaFree(n->Xi);
    n->Xi = nullptr;
    n->icap = 0;
    const int cap = std::max(rows, 1024);
    if (cudaMalloc(&n->Xi, sizeof(float) * (kIn + 1) * (size_t)cap) != cudaSuccess) {
        cudaGetLastError();
        return set_last_error(LBM_ENOMEM, "MLP work buffers");
    }
    n->icap = cap;
    return LBM_OK;
}

int ensure_train(lbm_mlp* n, int rows)
{
    if (rows <= n->tcap) return LBM_OK;
    free_train(n);
    const size_t cap = ((size_t)std::max(rows, 1024) + 63) / 64 * 64;  // every part starts on 128 bytes
    const size_t bytes = cap * (sizeof(float) * (kIn + 1) + sizeof(bf16) * kInPad + 8 * sizeof(bf16) * kH +
                                4 * sizeof(float) * kH + 2 * sizeof(float) + sizeof(bf16) * kOutPad) + 256;
    bool ok = cudaMalloc(&n->train, bytes) == cudaSuccess;
    for (int k = 0; k < 2 && ok; ++k)
        ok = cudaMallocHost(&n->stage[k], sizeof(float) * (kIn + 1) * cap) == cudaSuccess &&
             cudaEventCreateWithFlags(&n->staged[k], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        free_train(n);
        return set_last_error(LBM_ENOMEM, "MLP work buffers");
    }
    char* q = static_cast<char*>(n->train);
    auto take = [&](size_t b) {
        char* r = q;
        q += b;
        return static_cast<void*>(r);
    };
    n->loss = static_cast<double*>(take(256));
    n->Xt = static_cast<float*>(take(sizeof(float) * (kIn + 1) * cap));
    n->tb.Xp = static_cast<bf16*>(take(sizeof(bf16) * kInPad * cap));
    for (int l = 0; l < 4; ++l) {
        n->tb.h[l] = static_cast<bf16*>(take(sizeof(bf16) * kH * cap));
        n->tb.dZ[l] = static_cast<bf16*>(take(sizeof(bf16) * kH * cap));
        n->tb.dZ32[l] = static_cast<float*>(take(sizeof(float) * kH * cap));
    }
    n->tb.err = static_cast<float*>(take(sizeof(float) * cap));
    n->tb.dY = static_cast<float*>(take(sizeof(float) * cap));
    n->tb.dYb = static_cast<bf16*>(take(sizeof(bf16) * kOutPad * cap));
    n->tcap = (int)cap;
    return LBM_OK;
}

int pack_all(lbm_mlp* n)
{
    for (int l = 0; l < kLayers; ++l) {
        k_pack_weights<<<blocks(kK[l] * kN[l]), 256, 0, n->stream>>>(n->master, param_offset_w(l), kFanD(l),
                                                                     kFanD(l + 1), kK[l], kN[l], n->W[l]);
        MCK(cudaGetLastError());
    }
    return LBM_OK;
}

int sm_count(int device)
{
    int nsm = 1;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
    return nsm;
}

// One block per SM (the weights fill its shared memory), each walking its tiles.
unsigned pass_grid(const lbm_mlp* n, long long rows)
{
    return (unsigned)std::max(1LL, std::min<long long>((rows + kTileRows - 1) / kTileRows, sm_count(n->device)));
}

// y of `rows` feature rows at X (device).
int forward(lbm_mlp* n, const float* X, int rows, float* y)
{
    PassIn in{};
    in.X = X;
    k_mlp_pass<false><<<pass_grid(n, rows), kPassThreads, kPassBytes, n->stream>>>(n->view(), in, rows, y, TrainBuf{});
    MCK(cudaGetLastError());
    return LBM_OK;
}

// Loss (into n->loss) and gradient (into n->grad) of the batch in the training area.
int loss_and_grad(lbm_mlp* n, int rows)
{
    PassIn in{};
    in.X = n->Xt;
    TrainBuf tb = n->tb;
    tb.t = n->Xt + (size_t)rows * kIn;
    k_mlp_pass<true><<<pass_grid(n, rows), kPassThreads, kTrainBytes, n->stream>>>(n->view(), in, rows, nullptr, tb);
    MCK(cudaGetLastError());
    k_mlp_grad<<<kGradJobs, 128, kGradBytes, n->stream>>>(tb, rows, n->grad, n->loss);
    MCK(cudaGetLastError());
    return LBM_OK;
}

// SplitMix64, a counter-based generator (deterministic initialisation).
uint64_t splitmix64(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

}  // namespace

extern "C" {

int lbm_mlp_num_params(void) { return (int)kNParam; }

int lbm_mlp_create(lbm_mlp** out, uint64_t seed)
{
    if (!out) return set_last_error(LBM_EINVAL, "NULL argument");
    lbm_mlp* n = new (std::nothrow) lbm_mlp();
    if (!n) return set_last_error(LBM_ENOMEM, "host allocation failed");
    cudaGetDevice(&n->device);
    n->seed = seed;
    bool ok = cudaStreamCreateWithFlags(&n->stream, cudaStreamNonBlocking) == cudaSuccess &&
              cudaMalloc(&n->master, sizeof(float) * kNParam) == cudaSuccess &&
              cudaMalloc(&n->grad, sizeof(float) * kNParam) == cudaSuccess &&
              cudaMalloc(&n->m, sizeof(float) * kNParam) == cudaSuccess &&
              cudaMalloc(&n->v, sizeof(float) * kNParam) == cudaSuccess &&
              cudaFuncSetAttribute(k_mlp_pass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassBytes) ==
                  cudaSuccess &&
              cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradBytes) ==
                  cudaSuccess &&
              cudaFuncSetAttribute(k_mlp_pass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrainBytes) ==
                  cudaSuccess;
    for (int l = 0; l < kLayers && ok; ++l) ok = cudaMalloc(&n->W[l], sizeof(bf16) * kK[l] * kN[l]) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        lbm_mlp_destroy(n);
        return set_last_error(LBM_ENOMEM, "MLP allocation failed");
    }
    for (int l = 0; l < kLayers; ++l) n->b[l] = n->master + param_offset_b(l);
    // He-uniform weights from SplitMix64, zero biases
    std::vector<float> p(kNParam, 0.f);
    uint64_t ctr = seed * 0x100000001B3ull;
    for (int l = 0; l < kLayers; ++l) {
        const double lim = std::sqrt(6.0 / kFanD(l));
        for (long long i = 0; i < (long long)kFanD(l) * kFanD(l + 1); ++i) {
            const double u = (splitmix64(ctr++) >> 11) * (1.0 / 9007199254740992.0);
            p[param_offset_w(l) + i] = (float)((2.0 * u - 1.0) * lim);
        }
    }
    int rc = LBM_OK;
    if (cudaMemcpy(n->master, p.data(), sizeof(float) * kNParam, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(n->m, 0, sizeof(float) * kNParam) != cudaSuccess ||
        cudaMemset(n->v, 0, sizeof(float) * kNParam) != cudaSuccess)
        rc = set_last_error(LBM_ECUDA, "MLP upload failed");
    if (rc == LBM_OK) rc = pack_all(n);
    if (rc == LBM_OK && cudaStreamSynchronize(n->stream) != cudaSuccess) rc = set_last_error(LBM_ECUDA, "sync");
    if (rc != LBM_OK) {
        lbm_mlp_destroy(n);
        return rc;
    }
    *out = n;
    return LBM_OK;
}

int lbm_mlp_destroy(lbm_mlp* n)
{
    if (!n) return LBM_OK;
    cudaSetDevice(n->device);
    if (n->stream) cudaStreamSynchronize(n->stream);
    free_train(n);
    cudaFree(n->Xi);
    cudaFree(n->master);
    cudaFree(n->grad);
    cudaFree(n->m);
    cudaFree(n->v);
    for (int l = 0; l < kLayers; ++l) cudaFree(n->W[l]);
    if (n->stream) cudaStreamDestroy(n->stream);
    delete n;
    return LBM_OK;
}

int lbm_mlp_get_params(const lbm_mlp* n, float* out)
{
    if (!n || !out) return set_last_error(LBM_EINVAL, "NULL argument");
    MCK(cudaSetDevice(n->device));
    MCK(cudaMemcpyAsync(out, n->master, sizeof(float) * kNParam, cudaMemcpyDeviceToHost, n->stream));
    MCK(cudaStreamSynchronize(n->stream));
    return LBM_OK;
}

int lbm_mlp_set_params(lbm_mlp* n, const float* in)
{
    if (!n || !in) return set_last_error(LBM_EINVAL, "NULL argument");
    MCK(cudaSetDevice(n->device));
    MCK(cudaMemcpyAsync(n->master, in, sizeof(float) * kNParam, cudaMemcpyHostToDevice, n->stream));
    if (int rc = pack_all(n)) return rc;
    MCK(cudaStreamSynchronize(n->stream));
    return LBM_OK;
}

int lbm_mlp_features(const double* raw, int64_t n, float* out)
{
    if (!raw || !out || n < 0) return set_last_error(LBM_EINVAL, "bad argument");
    for (int64_t i = 0; i < n; ++i)
        mlp_features(raw[5 * i], raw[5 * i + 1], raw[5 * i + 2], raw[5 * i + 3], raw[5 * i + 4], out + 5 * i);
    return LBM_OK;
}

int lbm_mlp_predict(lbm_mlp* n, const float* X, int64_t rows, float* y)
{
    if (!n || !X || !y || rows < 0) return set_last_error(LBM_EINVAL, "bad argument");
    MCK(cudaSetDevice(n->device));
    const int chunk = 1 << 16;
    if (int rc = ensure_infer(n, (int)std::min<int64_t>(chunk, std::max<int64_t>(rows, 1)))) return rc;
    float* yd = n->Xi + (size_t)n->icap * kIn;
    for (int64_t r0 = 0; r0 < rows; r0 += chunk) {
        const int m = (int)std::min<int64_t>(chunk, rows - r0);
        MCK(cudaMemcpyAsync(n->Xi, X + r0 * kIn, sizeof(float) * m * kIn, cudaMemcpyHostToDevice, n->stream));
        if (int rc = forward(n, n->Xi, m, yd)) return rc;
        MCK(cudaMemcpyAsync(y + r0, yd, sizeof(float) * m, cudaMemcpyDeviceToHost, n->stream));
    }
    MCK(cudaStreamSynchronize(n->stream));
    return LBM_OK;
}

// Loss and gradient of one batch (for checks against a reference).
int lbm_mlp_loss_grad(lbm_mlp* n, const float* X, const float* t, int rows, double* loss, float* grad)
{
    if (!n || !X || !t || rows < 1) return set_last_error(LBM_EINVAL, "bad argument");
    MCK(cudaSetDevice(n->device));
    if (int rc = ensure_train(n, rows)) return rc;
    MCK(cudaMemcpyAsync(n->Xt, X, sizeof(float) * rows * (size_t)kIn, cudaMemcpyHostToDevice, n->stream));
    MCK(cudaMemcpyAsync(n->Xt + (size_t)rows * kIn, t, sizeof(float) * rows, cudaMemcpyHostToDevice, n->stream));
    if (int rc = loss_and_grad(n, rows)) return rc;
    double l = 0.0;
    MCK(cudaMemcpyAsync(&l, n->loss + 1, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
    if (grad) MCK(cudaMemcpyAsync(grad, n->grad, sizeof(float) * kNParam, cudaMemcpyDeviceToHost, n->stream));
    MCK(cudaStreamSynchronize(n->stream));
    if (loss) *loss = l;
    return LBM_OK;
}

// Adam on mini-batches of `batch` rows drawn without replacement (SplitMix64
// permutation per epoch).  *final_loss = mean loss of the last epoch.
int lbm_mlp_train(lbm_mlp* n, const float* X, const float* t, int64_t rows, int epochs, double lr, int batch,
                  double* final_loss)
{
    lbm::TraceRange trace("lbm_mlp_train");
    if (!n || !X || !t || rows < 1 || epochs < 0 || !(lr > 0.0) || batch < 16)
        return set_last_error(LBM_EINVAL, "bad argument");
    MCK(cudaSetDevice(n->device));
    if (int rc = ensure_train(n, batch)) return rc;
    std::vector<int64_t> perm(rows);
    for (int64_t i = 0; i < rows; ++i) perm[i] = i;
    uint64_t ctr = n->seed ^ 0xA5A5A5A5u;
    const NetView net = n->view();
    int64_t nb = 0, issued = 0;
    for (int ep = 0; ep < epochs; ++ep) {
        for (int64_t i = rows - 1; i > 0; --i) std::swap(perm[i], perm[splitmix64(ctr++) % (uint64_t)(i + 1)]);
        MCK(cudaMemsetAsync(n->loss, 0, sizeof(double), n->stream));
        nb = 0;
        for (int64_t r0 = 0; r0 + batch <= rows; r0 += batch, ++nb, ++issued) {
            // two pinned copies: the gather of one batch overlaps the step of the one before
            float* xb = n->stage[issued & 1];
            float* yb = xb + (size_t)batch * kIn;
            if (issued >= 2) MCK(cudaEventSynchronize(n->staged[issued & 1]));
            for (int i = 0; i < batch; ++i) {
                const int64_t s = perm[r0 + i];
                std::memcpy(xb + (size_t)i * kIn, X + s * kIn, sizeof(float) * kIn);
                yb[i] = t[s];
            }
            MCK(cudaMemcpyAsync(n->Xt, xb, sizeof(float) * (kIn + 1) * (size_t)batch, cudaMemcpyHostToDevice,
                                n->stream));
            MCK(cudaEventRecord(n->staged[issued & 1], n->stream));
            if (int rc = loss_and_grad(n, batch)) return rc;
            ++n->adam_t;
            const float c1 = 1.f - std::pow(0.9f, (float)n->adam_t), c2 = 1.f - std::pow(0.999f, (float)n->adam_t);
            k_adam<<<blocks(kNParam), 256, 0, n->stream>>>(n->master, n->grad, n->m, n->v, (int)kNParam, (float)lr,
                                                          0.9f, 0.999f, 1e-8f, c1, c2, net);
            MCK(cudaGetLastError());
        }
    }
    double sum = 0.0;
    if (nb) MCK(cudaMemcpyAsync(&sum, n->loss, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
    MCK(cudaStreamSynchronize(n->stream));
    if (final_loss) *final_loss = nb ? sum / nb : 0.0;
    return LBM_OK;
}

int lbm_mlp_save(const lbm_mlp* n, const char* path)
{
    if (!n || !path) return set_last_error(LBM_EINVAL, "NULL argument");
    std::vector<float> p(kNParam);
    if (int rc = lbm_mlp_get_params(n, p.data())) return rc;
    FILE* f = std::fopen(path, "wb");
    if (!f) return set_last_error(LBM_EIO, "cannot open file");
    const uint32_t hdr[2] = {0x4d4c5031u, (uint32_t)kNParam};
    const bool ok = std::fwrite(hdr, sizeof(hdr), 1, f) == 1 && std::fwrite(p.data(), sizeof(float), kNParam, f) == (size_t)kNParam;
    if (std::fclose(f) != 0 || !ok) return set_last_error(LBM_EIO, "write failed");
    return LBM_OK;
}

int lbm_mlp_load(lbm_mlp** out, const char* path)
{
    if (!out || !path) return set_last_error(LBM_EINVAL, "NULL argument");
    FILE* f = std::fopen(path, "rb");
    if (!f) return set_last_error(LBM_EIO, "cannot open file");
    uint32_t hdr[2] = {0, 0};
    std::vector<float> p(kNParam);
    const bool ok = std::fread(hdr, sizeof(hdr), 1, f) == 1 && hdr[0] == 0x4d4c5031u && hdr[1] == (uint32_t)kNParam &&
                    std::fread(p.data(), sizeof(float), kNParam, f) == (size_t)kNParam;
    std::fclose(f);
    if (!ok) return set_last_error(LBM_EIO, "not an MLP file");
    lbm_mlp* n = nullptr;
    if (int rc = lbm_mlp_create(&n, 0)) return rc;
    if (int rc = lbm_mlp_set_params(n, p.data())) {
        lbm_mlp_destroy(n);
        return rc;
    }
    *out = n;
    return LBM_OK;
}

}  // extern "C"

// ---- evaluation of the network on 1-D tables of signed distances ----------------
namespace lbm {

int mlp_device(const lbm_mlp* n) { return n->device; }

cudaError_t mlp_profile_tables(const lbm_mlp* n, double G, double tau, double order, const double* R_dev, double r_in,
                               int ncand, int T, double dmax, float* tables_dev, cudaStream_t s)
{
    PassIn in{};
    in.G = G;
    in.tau = tau;
    in.order = order;
    in.R = R_dev;
    in.r_in = r_in;
    in.T = T;
    in.dmax = dmax;
    const int rows = ncand * T;
    k_mlp_pass<false><<<pass_grid(n, rows), kPassThreads, kPassBytes, s>>>(n->view(), in, rows, tables_dev, TrainBuf{});
    return cudaGetLastError();
}

}  // namespace lbm
