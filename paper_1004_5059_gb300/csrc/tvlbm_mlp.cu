// The closure network on Blackwell tensor cores: inference and training each run as one kernel per
// 128-row tile in which every matrix product is a chain of tcgen05 MMAs (BF16 operands in
// 128-byte-swizzled shared memory, FP32 accumulators in TMEM) and the epilogues between them read
// TMEM row by row and fuse bias, GELU, its derivative, the loss and the bias gradients.
//
// Forward:  Z1 = X W1^T + b1, H1 = g(Z1);  Z2 = H1 W2^T + b2, H2 = g(Z2);  Y = H2 W3^T + b3.
// Backward (L = mean (Y - Y*)^2):  dY = 2 (Y - Y*) / (rows 12);  dZ2 = (dY W3) o g'(Z2);
//   dZ1 = (dZ2 W2) o g'(Z1);  dW3 = dY^T H2, dW2 = dZ2^T H1, dW1 = dZ1^T X (accumulated in TMEM
//   over a CTA's tiles, the CTAs' sums reduced in a fixed order);  db = column sums.
// No operand is ever transposed in memory: a tile stored with rows of 64 entries is a K-major
// operand where the product contracts its columns and an MN-major one where it contracts its rows.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <atomic>
#include <new>

#include "tvlbm.h"
#include "tvlbm_closure.h"
#include "tvlbm_host.h"
#include "tvlbm_kernels.cuh"
#include "tvlbm_mlp.h"
#include "tvlbm_tc.cuh"

using namespace tvlbm;
using namespace tvlbm::tc;

namespace {

constexpr int BM = 128, BK = 64;  // rows of a tile, columns of a 128-byte-swizzled chunk
constexpr int NIN = TVLBM_MLP_IN, NINP = TVLBM_MLP_IN_PAD, NH = TVLBM_MLP_HIDDEN, NOUT = TVLBM_MLP_OUT,
              NOUTP = TVLBM_MLP_OUT_PAD;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NIN, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NOUT * NH, NPARAM = OFF_B3 + NOUT;
static_assert(NPARAM == TVLBM_MLP_PARAMS, "parameter count");

using bf16 = __nv_bfloat16;

// GELU g(z) = z Phi(z), Phi(z) = (1 + erf(z / sqrt 2)) / 2, and g'(z) = Phi(z) + z phi(z).  erf by
// the rational approximation of Abramowitz & Stegun, Handbook of Mathematical Functions, eq.
// 7.1.26 (after Hastings): erf(x) = 1 - (a1 t + ... + a5 t^5) exp(-x^2), t = 1 / (1 + p x), x >= 0,
// |error| <= 1.5e-7, odd in x; the reciprocal and the exponential by the hardware approximations.
// The network stores its activations in BF16 (relative step 2^-8), so the error is invisible.
// E2 = exp(-x^2) = exp(-z^2 / 2) also gives phi(z) = E2 / sqrt(2 pi).
__device__ __forceinline__ float erf_as(float x, float& e2) {
    const float ax = fabsf(x);
    const float t = __fdividef(1.0f, fmaf(0.3275911f, ax, 1.0f));
    const float poly =
        t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.061405429f, -1.453152027f), 1.421413741f), -0.284496736f), 0.254829592f);
    e2 = __expf(-ax * ax);
    return copysignf(fmaf(-poly, e2, 1.0f), x);
}
__device__ __forceinline__ float gelu_f(float z) {
    float e2;
    return 0.5f * z * (1.0f + erf_as(z * 0.70710678118654752f, e2));
}
// Two GELUs in packed FP32 pairs, per lane the operations of gelu_f in its order (a packed
// multiply, add or fused multiply-add rounds each lane as the scalar instruction; the
// reciprocal, the exponential, |x| and the sign stay scalar).  The forward epilogues and
// tvlbm_mlp_activation's g use it.
__device__ __forceinline__ float2 gelu2_f(float2 z) {
    const float2 x = __fmul2_rn(z, make_float2(0.70710678118654752f, 0.70710678118654752f));
    const float2 ax = make_float2(fabsf(x.x), fabsf(x.y));
    const float2 d = __ffma2_rn(make_float2(0.3275911f, 0.3275911f), ax, make_float2(1.0f, 1.0f));
    const float2 t = make_float2(__fdividef(1.0f, d.x), __fdividef(1.0f, d.y));
    float2 q = __ffma2_rn(t, make_float2(1.061405429f, 1.061405429f), make_float2(-1.453152027f, -1.453152027f));
    q = __ffma2_rn(t, q, make_float2(1.421413741f, 1.421413741f));
    q = __ffma2_rn(t, q, make_float2(-0.284496736f, -0.284496736f));
    q = __ffma2_rn(t, q, make_float2(0.254829592f, 0.254829592f));
    const float2 poly = __fmul2_rn(t, q);
    const float2 sq = __fmul2_rn(make_float2(-ax.x, -ax.y), ax);
    const float2 e2 = make_float2(__expf(sq.x), __expf(sq.y));
    const float2 r = __ffma2_rn(make_float2(-poly.x, -poly.y), e2, make_float2(1.0f, 1.0f));
    const float2 er = make_float2(copysignf(r.x, x.x), copysignf(r.y, x.y));
    return __fmul2_rn(__fmul2_rn(make_float2(0.5f, 0.5f), z), __fadd2_rn(make_float2(1.0f, 1.0f), er));
}
// GELU and its derivative of a pair, erf and exponential shared: per lane the operations of gelu_f
// and gelu_grad_f.
__device__ __forceinline__ float2 gelu2_both(float2 z, float2& dg) {
    const float2 x = __fmul2_rn(z, make_float2(0.70710678118654752f, 0.70710678118654752f));
    const float2 ax = make_float2(fabsf(x.x), fabsf(x.y));
    const float2 d = __ffma2_rn(make_float2(0.3275911f, 0.3275911f), ax, make_float2(1.0f, 1.0f));
    const float2 t = make_float2(__fdividef(1.0f, d.x), __fdividef(1.0f, d.y));
    float2 q = __ffma2_rn(t, make_float2(1.061405429f, 1.061405429f), make_float2(-1.453152027f, -1.453152027f));
    q = __ffma2_rn(t, q, make_float2(1.421413741f, 1.421413741f));
    q = __ffma2_rn(t, q, make_float2(-0.284496736f, -0.284496736f));
    q = __ffma2_rn(t, q, make_float2(0.254829592f, 0.254829592f));
    const float2 poly = __fmul2_rn(t, q);
    const float2 sq = __fmul2_rn(make_float2(-ax.x, -ax.y), ax);
    const float2 e2 = make_float2(__expf(sq.x), __expf(sq.y));
    const float2 r = __ffma2_rn(make_float2(-poly.x, -poly.y), e2, make_float2(1.0f, 1.0f));
    const float2 er1 = __fadd2_rn(make_float2(1.0f, 1.0f), make_float2(copysignf(r.x, x.x), copysignf(r.y, x.y)));
    const float2 half = make_float2(0.5f, 0.5f);
    dg = __ffma2_rn(__fmul2_rn(z, make_float2(0.39894228040143268f, 0.39894228040143268f)), e2, __fmul2_rn(half, er1));
    return __fmul2_rn(__fmul2_rn(half, z), er1);
}
__device__ __forceinline__ float gelu_grad_f(float z) {
    float e2;
    const float er = erf_as(z * 0.70710678118654752f, e2);
    return fmaf(z * 0.39894228040143268f, e2, 0.5f * (1.0f + er));
}
__global__ void activation_kernel(const float* __restrict__ z, float* __restrict__ g, float* __restrict__ dg, int n) {
    // pairs of entries, g in the packed form of the forward epilogues (an odd last entry alone)
    for (int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x); i < n; i += 2 * gridDim.x * blockDim.x) {
        if (i + 1 < n) {
            if (g) {
                const float2 r = gelu2_f(make_float2(z[i], z[i + 1]));
                g[i] = r.x;
                g[i + 1] = r.y;
            }
            if (dg) {
                dg[i] = gelu_grad_f(z[i]);
                dg[i + 1] = gelu_grad_f(z[i + 1]);
            }
        } else {
            if (g) g[i] = gelu_f(z[i]);
            if (dg) dg[i] = gelu_grad_f(z[i]);
        }
    }
}
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---- fused inference: the three layers of one 128-row tile in one CTA ---------------------------
// X, W1, W2, W3 arrive by TMA (128-byte swizzle); H1 and H2 never leave shared memory: the
// epilogue threads write them in the same swizzled K-major layout the next MMA reads.  TMEM:
// columns [0, 128) hold layer 1, [128, 256) layer 2, [0, 16) then layer 3.
struct FusedCfg {
    static constexpr int X_OFF = 0, W1_OFF = 16384, W2_OFF = 32768, W3_OFF = 65536, H_OFF = 69632;
    static constexpr int BYTES = H_OFF + 32768;  // 100 KB
    static constexpr int SMEM = BYTES + 1024;
    static constexpr uint32_t TX = 16384 + 16384 + 32768 + 4096;
    static constexpr uint32_t TMEM_COLS = 256;
};

// Row r of a [128][128] BF16 tile stored as two 128-byte-swizzled K-major chunks of 64 columns:
// columns c0 .. c0 + 15 (c0 a multiple of 16) from 16 FP32 values.
__device__ __forceinline__ void store_h_sw128(unsigned char* h, int r, int c0, const float (&v)[16]) {
    const int kc = c0 >> 6, j0 = (c0 & 63) >> 3;  // chunk, first 16-byte unit in the row
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        alignas(16) __nv_bfloat16 b[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) b[q] = __float2bfloat16_rn(v[8 * half + q]);
        const int j = (j0 + half) ^ (r & 7);
        *reinterpret_cast<uint4*>(h + kc * 16384 + r * 128 + j * 16) = *reinterpret_cast<const uint4*>(b);
    }
}

// kFusedGroups warpgroups: warp w reads TMEM lanes 32 (w % 4) .. + 31 (its rows) and takes the
// (w / 4)-th of kFusedGroups column ranges of each hidden layer's epilogue, so every row's 128
// GELUs are split over kFusedGroups threads; the output layer's 16 columns go to the first
// warpgroup.
constexpr int kFusedGroups = 4;
constexpr int kFusedThreads = 128 * kFusedGroups;
static_assert(NH % (16 * kFusedGroups) == 0, "column ranges of whole 16-column loads");
static_assert(NINP == 16 * kFusedGroups, "FEAT: one 16-column input chunk per warpgroup");

// Features 16 G .. 16 G + 15 of cell `cell` (see MlpFeatures); neighbours wrap periodically.
template <int G>
__device__ __forceinline__ void feature_chunk(const MlpFeatures& f, int cell, float (&v)[16]) {
    const int cy = cell / f.nx, cx = cell - cy * f.nx;
    const long long n = (long long)f.nx * f.ny;
    const int xm = cx == 0 ? f.nx - 1 : cx - 1, xp = cx == f.nx - 1 ? 0 : cx + 1;
    const int ym = cy == 0 ? f.ny - 1 : cy - 1, yp = cy == f.ny - 1 ? 0 : cy + 1;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        constexpr int base = 16 * G;
        const int fi = base + e;  // compile time once unrolled
        if (fi >= NIN) {
            v[e] = 0.0f;
            continue;
        }
        const int k = fi / 6, q = fi % 6;
        const int xx = k % 3 == 0 ? xm : (k % 3 == 1 ? cx : xp), yy = k / 3 == 0 ? ym : (k / 3 == 1 ? cy : yp);
        v[e] = (__ldg(f.m6 + q * n + (long long)yy * f.nx + xx) - f.mu[q]) * f.isg[q];
    }
}

// FEAT: the input tile is built by the CTA's threads from the closure's moments (MlpFeatures)
// instead of loaded by TMA; thread (row r, warpgroup g) makes features 16 g .. 16 g + 15 of row
// r with the closure features kernel's arithmetic, so the inputs are the same BF16 values.
template <bool FEAT>
__global__ void __launch_bounds__(kFusedThreads) mlp_fused_forward_kernel(const __grid_constant__ CUtensorMap mx,
                                                                const __grid_constant__ CUtensorMap mw1,
                                                                const __grid_constant__ CUtensorMap mw2,
                                                                const __grid_constant__ CUtensorMap mw3,
                                                                const float* __restrict__ theta, float* __restrict__ y,
                                                                int* status, const MlpFeatures feat) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (saddr(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t load_bar, mma_bar;
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * BM;
    const float* b1 = theta + OFF_B1;
    const float* b2 = theta + OFF_B2;
    const float* b3 = theta + OFF_B3;
    if (tid == 0) {
        bar_init(&load_bar, 1);
        bar_init(&mma_bar, 1);
        bar_init_fence();
    }
    if (warp == 0) tmem_alloc(&tmem_slot, FusedCfg::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    unsigned char* xs = base + FusedCfg::X_OFF;
    unsigned char* w1 = base + FusedCfg::W1_OFF;
    unsigned char* w2 = base + FusedCfg::W2_OFF;
    unsigned char* w3 = base + FusedCfg::W3_OFF;
    unsigned char* hs = base + FusedCfg::H_OFF;
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const int r = (warp & 3) * 32 + lane;  // this thread's row of the tile (= its TMEM lane)
    const int cbeg = (warp >> 2) * (NH / kFusedGroups), cend = cbeg + NH / kFusedGroups;  // its column range

    bool ok = true;
    if (tid == 0) {
        bar_expect_tx(&load_bar, FEAT ? FusedCfg::TX - (uint32_t)(BM * NINP * 2) : FusedCfg::TX);
        if (!FEAT) tma_load_2d(xs, &mx, &load_bar, 0, m0);
        tma_load_2d(w1, &mw1, &load_bar, 0, 0);
        tma_load_2d(w2, &mw2, &load_bar, 0, 0);
        tma_load_2d(w2 + 16384, &mw2, &load_bar, BK, 0);
        tma_load_2d(w3, &mw3, &load_bar, 0, 0);
        tma_load_2d(w3 + 2048, &mw3, &load_bar, BK, 0);
    }
    if constexpr (FEAT) {
        // this thread's 16 input columns 16 g .. 16 g + 15 of row r, each builder with its feature
        // indices known at compile time
        const int g = warp >> 2;
        float v[16];
        switch (g) {
            case 0: feature_chunk<0>(feat, m0 + r, v); break;
            case 1: feature_chunk<1>(feat, m0 + r, v); break;
            case 2: feature_chunk<2>(feat, m0 + r, v); break;
            default: feature_chunk<3>(feat, m0 + r, v); break;
        }
        store_h_sw128(xs, r, 16 * g, v);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> MMA reads
        __syncthreads();
    }
    if (tid == 0) {
        ok = bar_wait(&load_bar, 0);
        if (ok) {
            tc_fence_after();
            const uint32_t idesc = idesc_bf16_f32(BM, NH);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
                mma_bf16(tmem, sw128_desc(saddr(xs) + kk * 32), sw128_desc(saddr(w1) + kk * 32), idesc, kk > 0);
        }
        mma_commit(&mma_bar);
    }
    // layer 1 epilogue: H1 = g(Z1 + b1) into shared memory
    ok = __syncthreads_and((tid != 0 || ok) && bar_wait(&mma_bar, 0)) != 0;
    tc_fence_after();
    if (ok) {
#pragma unroll 1
        for (int c0 = cbeg; c0 < cend; c0 += 16) {
            float v[16];
            __syncwarp();
            tmem_ld16(taddr + (uint32_t)c0, v);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const float2 g = gelu2_f(__fadd2_rn(make_float2(v[k], v[k + 1]), make_float2(b1[c0 + k], b1[c0 + k + 1])));
                v[k] = g.x;
                v[k + 1] = g.y;
            }
            store_h_sw128(hs, r, c0, v);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> MMA reads
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
        if (ok) {
            tc_fence_after();
            const uint32_t idesc = idesc_bf16_f32(BM, NH);
#pragma unroll
            for (int kc = 0; kc < 2; ++kc)
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk)
                    mma_bf16(tmem + NH, sw128_desc(saddr(hs) + kc * 16384 + kk * 32),
                             sw128_desc(saddr(w2) + kc * 16384 + kk * 32), idesc, kc > 0 || kk > 0);
        }
        mma_commit(&mma_bar);
    }
    // layer 2 epilogue: H2 = g(Z2 + b2) over H1 (the MMA that read H1 has completed)
    ok = __syncthreads_and(ok && bar_wait(&mma_bar, 1)) != 0;
    tc_fence_after();
    if (ok) {
#pragma unroll 1
        for (int c0 = cbeg; c0 < cend; c0 += 16) {
            float v[16];
            __syncwarp();
            tmem_ld16(taddr + (uint32_t)(NH + c0), v);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const float2 g = gelu2_f(__fadd2_rn(make_float2(v[k], v[k + 1]), make_float2(b2[c0 + k], b2[c0 + k + 1])));
                v[k] = g.x;
                v[k + 1] = g.y;
            }
            store_h_sw128(hs, r, c0, v);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
        if (ok) {
            tc_fence_after();
            const uint32_t idesc = idesc_bf16_f32(BM, NOUTP);
#pragma unroll
            for (int kc = 0; kc < 2; ++kc)
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk)
                    mma_bf16(tmem, sw128_desc(saddr(hs) + kc * 16384 + kk * 32),
                             sw128_desc(saddr(w3) + kc * 2048 + kk * 32), idesc, kc > 0 || kk > 0);
        }
        mma_commit(&mma_bar);
    }
    ok = __syncthreads_and(ok && bar_wait(&mma_bar, 0)) != 0;
    tc_fence_after();
    if (ok && warp < 4) {
        float v[16];
        __syncwarp();
        tmem_ld16(taddr, v);
        float4* d = reinterpret_cast<float4*>(y + (size_t)(m0 + r) * NOUTP);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = 4 * q + e < NOUT ? v[4 * q + e] + b3[4 * q + e] : 0.0f;
            d[q] = make_float4(o[0], o[1], o[2], o[3]);
        }
    } else if (tid == 0 && status) {
        atomicOr(status, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, FusedCfg::TMEM_COLS);
}

// Sums over the 32 lanes of 32 values a lane: lane c returns the sum of every lane's v[c] (halving
// exchange: 31 shuffles where 32 separate warp sums take 160).  v is overwritten.
__device__ __forceinline__ float column_sums32(float (&v)[32], int lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const float send = up ? v[k] : v[k + o], keep = up ? v[k + o] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0];
}

// ---- training: forward and backward of the 128-row tiles of a CTA ---------------------------------
// Shared memory: the weights (loaded once), the input tile, H1 and H2 (later overwritten by dZ1 and
// dZ2, once the products that read them are done) and dY, all as 64-column chunks with 128-byte
// rows.  TMEM (512 columns): the three weight gradients, accumulated over the CTA's tiles, Y, and
// two 128-column work areas.  g'(Z) stays in registers between the passes (BF16, 16 per layer).
// The products are tiny (0.14 MFLOP a row), so the chain of epilogues bounds it: 18 us for a tile, and
// one CTA per SM runs up to 152 tiles in that time.  A batch of 4096 rows takes 28 us (with the
// gradient reduction and Adam) where thirteen kernels, one product each with its operands and their
// transposes through memory, took 155 us.
struct TrainCfg {
    static constexpr int X_OFF = 0, W1_OFF = 16384, W2_OFF = 32768, W3_OFF = 65536, H1_OFF = 69632, H2_OFF = 102400,
                         DY_OFF = 135168;
    static constexpr int BYTES = DY_OFF + 16384;  // 148 KB
    static constexpr int SMEM = BYTES + 1024;
    static constexpr uint32_t TX_W = 16384 + 32768 + 4096, TX_X = 16384;
    static constexpr uint32_t T_DW2 = 0, T_DW1 = 128, T_DW3 = 192, T_Y = 208, T_A = 256, T_B = 384;
    // a CTA's partial sums, floats: dW1 [128][64], dW2 [128][128], dW3 [16][128], then the bias
    // gradients of the four 32-row groups: db1 [4][128], db2 [4][128], db3 [4][16]
    static constexpr int P_W1 = 0, P_W2 = P_W1 + NH * NINP, P_W3 = P_W2 + NH * NH, P_B1 = P_W3 + NOUTP * NH,
                         P_B2 = P_B1 + 4 * NH, P_B3 = P_B2 + 4 * NH, P_TOTAL = P_B3 + 4 * NOUTP;
};

// K = 16 slices kk of D (+)= A B^T over `steps` slices, operand starts ad / bd advancing by as / bs
// descriptor units (16 bytes) per slice.
__device__ __forceinline__ void mma_chain(uint32_t d, uint64_t ad, uint64_t bd, uint32_t as, uint32_t bs, int steps,
                                          uint32_t idesc, bool accumulate) {
#pragma unroll 8
    for (int k = 0; k < steps; ++k) mma_bf16(d, ad + (uint64_t)k * as, bd + (uint64_t)k * bs, idesc, accumulate || k > 0);
}

__global__ void __launch_bounds__(kFusedThreads, 1) mlp_train_kernel(const __grid_constant__ CUtensorMap mx,
                                                                     const __grid_constant__ CUtensorMap mw1,
                                                                     const __grid_constant__ CUtensorMap mw2,
                                                                     const __grid_constant__ CUtensorMap mw3,
                                                                     const float* __restrict__ theta,
                                                                     const float* __restrict__ ystar, int tiles, float scale,
                                                                     float* __restrict__ part, double* __restrict__ loss_part,
                                                                     int* status) {
    using Cfg = TrainCfg;
    static_assert(kFusedGroups == 4, "32 columns per thread and hidden layer");
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (saddr(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t w_bar, x_bar, mma_bar;
    __shared__ __align__(16) float bias[2 * NH + NOUTP];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_launch_dependents();
    if (tid == 0) {
        bar_init(&w_bar, 1);
        bar_init(&x_bar, 1);
        bar_init(&mma_bar, 1);
        bar_init_fence();
    }
    if (warp == 0) tmem_alloc(&tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();  // the weights (and the partial sums' readers) of the kernels before this one
    const uint32_t tmem = tmem_slot;
    unsigned char *xs = base + Cfg::X_OFF, *w1 = base + Cfg::W1_OFF, *w2 = base + Cfg::W2_OFF, *w3 = base + Cfg::W3_OFF,
                  *h1 = base + Cfg::H1_OFF, *h2 = base + Cfg::H2_OFF, *dys = base + Cfg::DY_OFF;
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const int r = (warp & 3) * 32 + lane;  // this thread's row of the tile (= its TMEM lane)
    const int cbeg = (warp >> 2) * 32;     // its 32 columns of a hidden layer
    // the biases, read past the L1 cache (an earlier kernel on the stream may still have been writing
    // them when this one was launched)
    if (tid < NH) bias[tid] = __ldcg(theta + OFF_B1 + tid);
    else if (tid < 2 * NH) bias[tid] = __ldcg(theta + OFF_B2 + tid - NH);
    else if (tid < 2 * NH + NOUTP) bias[tid] = tid < 2 * NH + NOUT ? __ldcg(theta + OFF_B3 + tid - 2 * NH) : 0.0f;
    const float *b1 = bias + cbeg, *b2 = bias + NH + cbeg, *b3 = bias + 2 * NH;

    if (tid == 0) {
        bar_expect_tx(&w_bar, Cfg::TX_W);
        tma_load_2d(w1, &mw1, &w_bar, 0, 0);
        tma_load_2d(w2, &mw2, &w_bar, 0, 0);
        tma_load_2d(w2 + 16384, &mw2, &w_bar, BK, 0);
        tma_load_2d(w3, &mw3, &w_bar, 0, 0);
        tma_load_2d(w3 + 2048, &mw3, &w_bar, BK, 0);
        bar_expect_tx(&x_bar, Cfg::TX_X);
        tma_load_2d(xs, &mx, &x_bar, 0, (int)blockIdx.x * BM);
    }
    uint32_t ph = 0;  // phase of mma_bar
    bool ok = true;
    // every thread waits for the products committed last; the MMAs' reads of shared memory are done too
    auto products_done = [&]() {
        ok = __syncthreads_and(ok && bar_wait(&mma_bar, ph)) != 0;
        ph ^= 1;
        tc_fence_after();
    };
    // generic writes of this thread -> MMA operands
    auto operands_ready = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    };
    const uint32_t kk = idesc_bf16_f32(BM, NH), kk16 = idesc_bf16_f32(BM, NOUTP);
    constexpr uint32_t A_MN = 1u << 15, B_MN = 1u << 16;
    float db1 = 0.0f, db2 = 0.0f, db3 = 0.0f;  // column sums of this warp's rows: column cbeg + lane (db3: lane)
    double loss = 0.0;
    bool first = true;

#pragma unroll 1
    for (int tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, first = false) {
        const int m0 = tile * BM;
        const uint32_t xph = (uint32_t)((tile - (int)blockIdx.x) / (int)gridDim.x) & 1u;
        float4 ys[3];
        if (warp < 4) {  // the targets, long before they are needed
            const float4* q = reinterpret_cast<const float4*>(ystar + (size_t)(m0 + r) * NOUTP);
#pragma unroll
            for (int k = 0; k < 3; ++k) ys[k] = __ldg(q + k);
        }
        if (tid == 0) {
            ok = (!first || bar_wait(&w_bar, 0)) && bar_wait(&x_bar, xph);
            tc_fence_after();
            if (ok) mma_chain(tmem + Cfg::T_A, sw128_desc(saddr(xs)), sw128_desc(saddr(w1)), 2, 2, BK / 16, kk, false);
            mma_commit(&mma_bar);
        }
        products_done();
        uint32_t g1[16], g2[16];  // g'(Z1), g'(Z2) of this thread's columns, BF16 pairs
        // H = g(Z + b) into h, g'(Z + b) into gp
        auto hidden = [&](uint32_t t0, const float* b, unsigned char* h, uint32_t (&gp)[16]) {
#pragma unroll
            for (int c = 0; c < 32; c += 16) {
                float v[16];
                __syncwarp();
                tmem_ld16(taddr + t0 + (uint32_t)(cbeg + c), v);
#pragma unroll
                for (int k = 0; k < 16; k += 2) {
                    float2 dg;
                    const float2 g = gelu2_both(
                        __fadd2_rn(make_float2(v[k], v[k + 1]), *reinterpret_cast<const float2*>(b + c + k)), dg);
                    v[k] = g.x;
                    v[k + 1] = g.y;
                    const __nv_bfloat162 d2 = __floats2bfloat162_rn(dg.x, dg.y);
                    gp[(c + k) / 2] = *reinterpret_cast<const uint32_t*>(&d2);
                }
                store_h_sw128(h, r, cbeg + c, v);
            }
        };
        if (ok) hidden(Cfg::T_A, b1, h1, g1);
        operands_ready();
        if (tid == 0) {
            if (ok)
#pragma unroll
                for (int kc = 0; kc < 2; ++kc)
                    mma_chain(tmem + Cfg::T_B, sw128_desc(saddr(h1) + kc * 16384), sw128_desc(saddr(w2) + kc * 16384), 2, 2,
                              BK / 16, kk, kc > 0);
            mma_commit(&mma_bar);
        }
        products_done();
        if (ok) hidden(Cfg::T_B, b2, h2, g2);
        operands_ready();
        if (tid == 0) {
            if (ok)
#pragma unroll
                for (int kc = 0; kc < 2; ++kc)
                    mma_chain(tmem + Cfg::T_Y, sw128_desc(saddr(h2) + kc * 16384), sw128_desc(saddr(w3) + kc * 2048), 2, 2,
                              BK / 16, kk16, kc > 0);
            mma_commit(&mma_bar);
        }
        products_done();
        if (ok && warp < 4) {  // the loss, dY (BF16, columns 12 .. 15 zero), db3
            float v[32];
            {
                float y[16];
                __syncwarp();
                tmem_ld16(taddr + Cfg::T_Y, y);
                const float* t = reinterpret_cast<const float*>(ys);
                float sq = 0.0f;
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const float d = k < NOUT ? (y[k] + b3[k]) - t[k < NOUT ? k : 0] : 0.0f;
                    sq = fmaf(d, d, sq);
                    y[k] = scale * d;
                    v[k] = y[k];
                    v[k + 16] = 0.0f;
                }
                store_h_sw128(dys, r, 0, y);
                const float s = warp_sum_f(sq);
                loss += (double)s;
            }
            db3 += column_sums32(v, lane);
        }
        operands_ready();
        if (tid == 0) {
            if (ok) {
                // dH2 = dY W3 (contracts the 16 outputs), dW3^T += H2^T dY (contracts the rows)
                mma_chain(tmem + Cfg::T_A, sw128_desc(saddr(dys)), sw128_mn_desc(saddr(w3), 2048), 0, 0, 1, kk | B_MN, false);
                mma_chain(tmem + Cfg::T_DW3, sw128_mn_desc(saddr(h2), 16384), sw128_mn_desc(saddr(dys), 16384), 128, 128,
                          BM / 16, kk16 | A_MN | B_MN, !first);
            }
            mma_commit(&mma_bar);
        }
        products_done();
        // dZ = dH o g'(Z) into h, its column sums into db
        auto back = [&](uint32_t t0, const uint32_t (&gp)[16], unsigned char* h, float& db) {
            float dz[32];
#pragma unroll
            for (int c = 0; c < 32; c += 16) {
                float v[16];
                __syncwarp();
                tmem_ld16(taddr + t0 + (uint32_t)(cbeg + c), v);
#pragma unroll
                for (int k = 0; k < 16; k += 2) {
                    const __nv_bfloat162 d2 = *reinterpret_cast<const __nv_bfloat162*>(&gp[(c + k) / 2]);
                    v[k] *= __low2float(d2);
                    v[k + 1] *= __high2float(d2);
                    dz[c + k] = v[k];
                    dz[c + k + 1] = v[k + 1];
                }
                store_h_sw128(h, r, cbeg + c, v);
            }
            db += column_sums32(dz, lane);
        };
        if (ok) back(Cfg::T_A, g2, h2, db2);
        operands_ready();
        if (tid == 0) {
            if (ok) {
                // dH1 = dZ2 W2 (contracts layer 2's units), dW2 += dZ2^T H1 (contracts the rows)
#pragma unroll
                for (int kc = 0; kc < 2; ++kc)
                    mma_chain(tmem + Cfg::T_B, sw128_desc(saddr(h2) + kc * 16384),
                              sw128_mn_desc(saddr(w2) + kc * 8192, 16384), 2, 128, BK / 16, kk | B_MN, kc > 0);
                mma_chain(tmem + Cfg::T_DW2, sw128_mn_desc(saddr(h2), 16384), sw128_mn_desc(saddr(h1), 16384), 128, 128,
                          BM / 16, kk | A_MN | B_MN, !first);
            }
            mma_commit(&mma_bar);
        }
        products_done();
        if (ok) back(Cfg::T_B, g1, h1, db1);
        operands_ready();
        if (tid == 0) {
            if (ok)  // dW1 += dZ1^T X
                mma_chain(tmem + Cfg::T_DW1, sw128_mn_desc(saddr(h1), 16384), sw128_mn_desc(saddr(xs), 16384), 128, 128,
                          BM / 16, idesc_bf16_f32(BM, NINP) | A_MN | B_MN, !first);
            mma_commit(&mma_bar);
        }
        products_done();
        if (tid == 0 && ok && tile + (int)gridDim.x < tiles) {
            bar_expect_tx(&x_bar, Cfg::TX_X);
            tma_load_2d(xs, &mx, &x_bar, 0, (tile + (int)gridDim.x) * BM);
        }
    }

    if (ok) {
        float* q = part + (size_t)blockIdx.x * Cfg::P_TOTAL;
        float v[16];
        auto drain = [&](uint32_t t0, float* row) {
            __syncwarp();
            tmem_ld16(taddr + t0, v);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                reinterpret_cast<float4*>(row)[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        };
        drain(Cfg::T_DW2 + cbeg, q + Cfg::P_W2 + r * NH + cbeg);
        drain(Cfg::T_DW2 + cbeg + 16, q + Cfg::P_W2 + r * NH + cbeg + 16);
        drain(Cfg::T_DW1 + cbeg / 2, q + Cfg::P_W1 + r * NINP + cbeg / 2);
        if (warp < 4) {
            __syncwarp();
            tmem_ld16(taddr + Cfg::T_DW3, v);
#pragma unroll
            for (int k = 0; k < NOUTP; ++k) q[Cfg::P_W3 + k * NH + r] = v[k];
            if (lane < NOUTP) q[Cfg::P_B3 + warp * NOUTP + lane] = db3;
            if (lane == 0) loss_part[blockIdx.x * 4 + warp] = loss;
        }
        q[Cfg::P_B1 + (warp & 3) * NH + cbeg + lane] = db1;
        q[Cfg::P_B2 + (warp & 3) * NH + cbeg + lane] = db2;
    } else if (tid == 0) {
        if (status) atomicOr(status, 1);
        // let the loads started so far land before the CTA exits (bounded)
        bar_wait(&w_bar, 0);
        bar_wait(&x_bar, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, 512);
}

// ---- small kernels ---------------------------------------------------------------------------

// grad[i] = the CTAs' partial sums in a fixed order: 64 parameters per block, four threads each
// taking every fourth CTA; the last block sums the loss.
__global__ void __launch_bounds__(256) reduce_gradient_kernel(const float* __restrict__ part,
                                                              const double* __restrict__ loss_part, int ctas,
                                                              float* __restrict__ grad, double* __restrict__ loss) {
    using Cfg = TrainCfg;
    __shared__ float sh[4][64];
    pdl_launch_dependents();
    pdl_wait();
    const int t = threadIdx.x & 63, g = threadIdx.x >> 6;
    if (blockIdx.x == gridDim.x - 1) {
        if (threadIdx.x < 32) {
            double l = 0.0;
            for (int k = threadIdx.x; k < 4 * ctas; k += 32) l += __ldcg(loss_part + k);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
            if (threadIdx.x == 0) *loss = l;
        }
        return;
    }
    const int i = blockIdx.x * 64 + t;
    int off = 0, groups = 1, ld = 0;
    if (i < OFF_B1) off = Cfg::P_W1 + (i / NIN) * NINP + i % NIN;
    else if (i < OFF_W2) off = Cfg::P_B1 + i - OFF_B1, groups = 4, ld = NH;
    else if (i < OFF_B2) off = Cfg::P_W2 + i - OFF_W2;
    else if (i < OFF_W3) off = Cfg::P_B2 + i - OFF_B2, groups = 4, ld = NH;
    else if (i < OFF_B3) off = Cfg::P_W3 + i - OFF_W3;
    else off = Cfg::P_B3 + i - OFF_B3, groups = 4, ld = NOUTP;
    float acc = 0.0f;
    if (i < NPARAM) {
#pragma unroll 8
        for (int c = g; c < ctas; c += 4) acc += __ldcg(part + (size_t)c * Cfg::P_TOTAL + off);
        for (int k = 1; k < groups; ++k)
            for (int c = g; c < ctas; c += 4) acc += __ldcg(part + (size_t)c * Cfg::P_TOTAL + off + k * ld);
    }
    sh[g][t] = acc;
    __syncthreads();
    if (g == 0 && i < NPARAM) grad[i] = (sh[0][t] + sh[1][t]) + (sh[2][t] + sh[3][t]);
}

// The BF16 copy of parameter i in the layout the products read (zero padding where K or N is padded:
// written once, when the network is created).
__device__ __forceinline__ void cast_weight(int i, float v, bf16* w1p, bf16* w2, bf16* w3p) {
    if (i < OFF_B1) w1p[(i / NIN) * NINP + i % NIN] = __float2bfloat16_rn(v);
    else if (i >= OFF_W2 && i < OFF_B2) w2[i - OFF_W2] = __float2bfloat16_rn(v);
    else if (i >= OFF_W3 && i < OFF_B3) w3p[i - OFF_W3] = __float2bfloat16_rn(v);
}

// One Adam step and the BF16 weights with it.
__global__ void __launch_bounds__(256) adam_kernel(float* __restrict__ theta, float* __restrict__ m1, float* __restrict__ m2,
                                                   const float* __restrict__ g, int n, float lr, float b1, float b2,
                                                   float eps, float c1, float c2, bf16* __restrict__ w1p,
                                                   bf16* __restrict__ w2, bf16* __restrict__ w3p) {
    pdl_launch_dependents();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = __ldcg(g + i);
    const float a = b1 * m1[i] + (1.0f - b1) * gi;
    const float b = b2 * m2[i] + (1.0f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    const float t = theta[i] - lr * (a / c1) / (sqrtf(b / c2) + eps);
    theta[i] = t;
    cast_weight(i, t, w1p, w2, w3p);
}

__global__ void cast_weights_kernel(const float* __restrict__ th, bf16* __restrict__ w1p, bf16* __restrict__ w2,
                                    bf16* __restrict__ w3p) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NPARAM) cast_weight(i, th[i], w1p, w2, w3p);
}

}  // namespace

// =============================================================================================
// Host side
// =============================================================================================
struct tvlbm_mlp {
    int device, max_rows;
    cudaStream_t stream;
    unsigned char* mem;
    size_t bytes;
    float *theta, *m1, *m2, *grad, *part;
    double *loss, *loss_part;
    int* status;
    bf16 *w1p, *w2, *w3p;
    float* ybuf;
    int ctas;  // most CTAs of a training pass (one per SM), the partial sums' extent
    int adam_t;
    unsigned long long uid;
    // descriptors of the last inference call (inputs at cached_x, cached_rows rows)
    const void* cached_x;
    int cached_rows;
    alignas(64) CUtensorMap fwd_maps[4];
    char err[256];
};

namespace {

int mfail(tvlbm_mlp* m, int code, const char* fmt, ...) {
    if (m) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(m->err, sizeof(m->err), fmt, ap);
        va_end(ap);
    }
    return code;
}

#define MLP_CUDA(m, call, what)                                                                        \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess) return mfail(m, TVLBM_ECUDA, "%s: %s", what, cudaGetErrorString(e_)); \
    } while (0)

// 2-D BF16 tensor map over a row-major [rows][k_total] matrix with row length ld (elements),
// box 64 x box_rows, 128-byte swizzle.
bool bf16_map(CUtensorMap* map, const void* base, int k_total, int rows, int ld, int box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = host::tensor_map_encoder();
    if (!enc || ((uintptr_t)base & 15) || (ld * 2) % 16) return false;
    cuuint64_t dims[2] = {(cuuint64_t)k_total, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int check_rows(tvlbm_mlp* m, int rows) {
    if (rows <= 0 || rows % BM || rows > m->max_rows)
        return mfail(m, TVLBM_EINVAL, "rows %d must be a positive multiple of 128 and at most %d", rows, m->max_rows);
    return TVLBM_OK;
}

int read_status(tvlbm_mlp* m) {
    int st = 0;
    MLP_CUDA(m, cudaMemcpyAsync(&st, m->status, sizeof(int), cudaMemcpyDeviceToHost, m->stream), "status copy");
    MLP_CUDA(m, cudaStreamSynchronize(m->stream), "synchronize");
    if (st) {
        cudaMemsetAsync(m->status, 0, sizeof(int), m->stream);
        cudaStreamSynchronize(m->stream);
        return mfail(m, TVLBM_ETIMEOUT, "a device-side wait of the network kernels timed out");
    }
    return TVLBM_OK;
}

int refresh_weights(tvlbm_mlp* m) {
    cast_weights_kernel<<<(NPARAM + 255) / 256, 256, 0, m->stream>>>(m->theta, m->w1p, m->w2, m->w3p);
    MLP_CUDA(m, cudaGetLastError(), "cast kernel");
    return TVLBM_OK;
}

}  // namespace

namespace tvlbm {
// Forward pass into y [rows][16] (FP32).  Used by tvlbm_mlp_forward and the closure step.
int mlp_forward_async(tvlbm_mlp* m, const void* x, int rows, float* y) {
    int rc = check_rows(m, rows);
    if (rc) return rc;
    // the weight descriptors never change; the input's are kept for repeated calls on one buffer
    if (m->cached_x != x || m->cached_rows != rows) {
        if (!bf16_map(&m->fwd_maps[0], x, NINP, rows, NINP, BM) ||
            !bf16_map(&m->fwd_maps[1], m->w1p, NINP, NH, NINP, NH) ||
            !bf16_map(&m->fwd_maps[2], m->w2, NH, NH, NH, NH) || !bf16_map(&m->fwd_maps[3], m->w3p, NH, NOUTP, NH, NOUTP)) {
            m->cached_x = nullptr;
            return mfail(m, TVLBM_EINVAL, "TMA descriptor rejected (alignment of x?)");
        }
        m->cached_x = x;
        m->cached_rows = rows;
    }
    const CUtensorMap &mx = m->fwd_maps[0], &mw1 = m->fwd_maps[1], &mw2 = m->fwd_maps[2], &mw3 = m->fwd_maps[3];
    const int tiles = rows / BM;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        MLP_CUDA(m, cudaFuncSetAttribute(mlp_fused_forward_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         FusedCfg::SMEM),
                 "fused forward attribute");
        attr_set[dev] = true;
    }
    MlpFeatures none;
    memset(&none, 0, sizeof(none));
    mlp_fused_forward_kernel<false><<<tiles, kFusedThreads, FusedCfg::SMEM, m->stream>>>(mx, mw1, mw2, mw3, m->theta, y,
                                                                                        m->status, none);
    MLP_CUDA(m, cudaGetLastError(), "fused forward");
    return TVLBM_OK;
}

int mlp_forward_features_async(tvlbm_mlp* m, const MlpFeatures& feat, int rows, float* y) {
    int rc = check_rows(m, rows);
    if (rc) return rc;
    if (!feat.m6 || feat.nx < 1 || feat.ny < 1 || (long long)feat.nx * feat.ny != rows)
        return mfail(m, TVLBM_EINVAL, "feature source does not match the rows");
    // the weight descriptors (the input one is passed along unused)
    CUtensorMap mx, mw1, mw2, mw3;
    memset(&mx, 0, sizeof(mx));
    if (!bf16_map(&mw1, m->w1p, NINP, NH, NINP, NH) || !bf16_map(&mw2, m->w2, NH, NH, NH, NH) ||
        !bf16_map(&mw3, m->w3p, NH, NOUTP, NH, NOUTP))
        return mfail(m, TVLBM_EINVAL, "TMA descriptor rejected");
    const int tiles = rows / BM;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        MLP_CUDA(m, cudaFuncSetAttribute(mlp_fused_forward_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         FusedCfg::SMEM),
                 "fused forward attribute");
        attr_set[dev] = true;
    }
    mlp_fused_forward_kernel<true><<<tiles, kFusedThreads, FusedCfg::SMEM, m->stream>>>(mx, mw1, mw2, mw3, m->theta, y,
                                                                                       m->status, feat);
    MLP_CUDA(m, cudaGetLastError(), "fused forward with features");
    return TVLBM_OK;
}
int mlp_max_rows(const tvlbm_mlp* m) { return m->max_rows; }
float* mlp_ybuf(tvlbm_mlp* m) { return m->ybuf; }
int mlp_set_stream(tvlbm_mlp* m, cudaStream_t s) {
    m->stream = s;
    return TVLBM_OK;
}
int mlp_status(tvlbm_mlp* m) { return read_status(m); }
unsigned long long mlp_uid(const tvlbm_mlp* m) { return m->uid; }
cudaStream_t mlp_stream(const tvlbm_mlp* m) { return m->stream; }
}  // namespace tvlbm

extern "C" {

int tvlbm_mlp_create(int max_rows, tvlbm_mlp** out) {
    if (!out) return TVLBM_EINVAL;
    *out = nullptr;
    if (max_rows <= 0 || max_rows % BM || max_rows > (1 << 26)) return TVLBM_EINVAL;
    tvlbm_mlp* m = new (std::nothrow) tvlbm_mlp();
    if (!m) return TVLBM_ENOMEM;
    memset(m, 0, sizeof(*m));
    cudaGetDevice(&m->device);
    m->max_rows = max_rows;
    static std::atomic<unsigned long long> next_uid{1};
    m->uid = next_uid.fetch_add(1);
    const size_t R = (size_t)max_rows;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device);
    if (sms < 1) sms = 1;
    m->ctas = max_rows / BM < sms ? max_rows / BM : sms;
    // carve one allocation: FP32 block, then BF16 block (every piece 256-byte aligned)
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = host::align_up(off + bytes, 256);
        return o;
    };
    const size_t o_theta = take(NPARAM * 4), o_m1 = take(NPARAM * 4), o_m2 = take(NPARAM * 4), o_grad = take(NPARAM * 4);
    const size_t o_part = take((size_t)m->ctas * TrainCfg::P_TOTAL * 4), o_losses = take((size_t)m->ctas * 4 * 8),
                 o_loss = take(8), o_status = take(4);
    const size_t o_y = take(R * NOUTP * 4);
    const size_t o_w1p = take(NH * NINP * 2), o_w2 = take(NH * NH * 2), o_w3p = take(NOUTP * NH * 2);
    m->bytes = off;
    if (cudaMalloc((void**)&m->mem, off) != cudaSuccess) {
        delete m;
        return TVLBM_ENOMEM;
    }
    unsigned char* b = m->mem;
    m->theta = (float*)(b + o_theta);
    m->m1 = (float*)(b + o_m1);
    m->m2 = (float*)(b + o_m2);
    m->grad = (float*)(b + o_grad);
    m->part = (float*)(b + o_part);
    m->loss = (double*)(b + o_loss);
    m->status = (int*)(b + o_status);
    m->ybuf = (float*)(b + o_y);
    m->loss_part = (double*)(b + o_losses);
    m->w1p = (bf16*)(b + o_w1p);
    m->w2 = (bf16*)(b + o_w2);
    m->w3p = (bf16*)(b + o_w3p);
    // zero everything once: parameters, moments, and the padding of the BF16 weights (never written)
    if (cudaMemset(m->mem, 0, off) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
        cudaFree(m->mem);
        delete m;
        return TVLBM_ECUDA;
    }
    *out = m;
    return TVLBM_OK;
}

int tvlbm_mlp_destroy(tvlbm_mlp* m) {
    if (!m) return TVLBM_OK;
    cudaSetDevice(m->device);
    cudaStreamSynchronize(m->stream);
    cudaFree(m->mem);
    delete m;
    return TVLBM_OK;
}

int tvlbm_mlp_set_stream(tvlbm_mlp* m, void* stream) {
    if (!m) return TVLBM_EINVAL;
    m->stream = (cudaStream_t)stream;
    return TVLBM_OK;
}

int tvlbm_mlp_set_params(tvlbm_mlp* m, const float* params) {
    if (!m || !params) return TVLBM_EINVAL;
    for (int i = 0; i < NPARAM; ++i)
        if (!isfinite(params[i])) return mfail(m, TVLBM_EINVAL, "parameter %d is not finite", i);
    cudaSetDevice(m->device);
    MLP_CUDA(m, cudaMemcpyAsync(m->theta, params, NPARAM * 4, cudaMemcpyHostToDevice, m->stream), "copy params");
    MLP_CUDA(m, cudaMemsetAsync(m->m1, 0, NPARAM * 4, m->stream), "clear moments");
    MLP_CUDA(m, cudaMemsetAsync(m->m2, 0, NPARAM * 4, m->stream), "clear moments");
    m->adam_t = 0;
    const int rc = refresh_weights(m);
    if (rc) return rc;
    MLP_CUDA(m, cudaStreamSynchronize(m->stream), "synchronize");
    return TVLBM_OK;
}

int tvlbm_mlp_get_params(tvlbm_mlp* m, float* params) {
    if (!m || !params) return TVLBM_EINVAL;
    cudaSetDevice(m->device);
    MLP_CUDA(m, cudaMemcpyAsync(params, m->theta, NPARAM * 4, cudaMemcpyDeviceToHost, m->stream), "copy params");
    MLP_CUDA(m, cudaStreamSynchronize(m->stream), "synchronize");
    return TVLBM_OK;
}

int tvlbm_mlp_forward(tvlbm_mlp* m, const void* x, int rows, float* y) {
    if (!m || !x || !y) return TVLBM_EINVAL;
    cudaSetDevice(m->device);
    return mlp_forward_async(m, x, rows, y);
}

int tvlbm_mlp_loss_grad(tvlbm_mlp* m, const void* x, const float* ystar, int rows, double* loss, float* grad) {
    if (!m || !x || !ystar) return TVLBM_EINVAL;
    int rc = check_rows(m, rows);
    if (rc) return rc;
    cudaSetDevice(m->device);
    cudaStream_t s = m->stream;
    const int tiles = rows / BM, ctas = tiles < m->ctas ? tiles : m->ctas;
    CUtensorMap mx, mw1, mw2, mw3;
    if (!bf16_map(&mx, x, NINP, rows, NINP, BM) || !bf16_map(&mw1, m->w1p, NINP, NH, NINP, NH) ||
        !bf16_map(&mw2, m->w2, NH, NH, NH, NH) || !bf16_map(&mw3, m->w3p, NH, NOUTP, NH, NOUTP))
        return mfail(m, TVLBM_EINVAL, "TMA descriptor rejected (alignment of x?)");
    if ((uintptr_t)ystar & 15) return mfail(m, TVLBM_EINVAL, "ystar must be 16-byte aligned");
    static bool attr_set[64] = {};
    if (m->device < 0 || m->device >= 64 || !attr_set[m->device]) {
        MLP_CUDA(m, cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TrainCfg::SMEM),
                 "training kernel attribute");
        if (m->device >= 0 && m->device < 64) attr_set[m->device] = true;
    }
    MLP_CUDA(m, launch_pdl(mlp_train_kernel, dim3(ctas), dim3(kFusedThreads), TrainCfg::SMEM, s, mx, mw1, mw2, mw3,
                           (const float*)m->theta, ystar, tiles, 2.0f / ((float)rows * (float)NOUT), m->part, m->loss_part,
                           m->status),
             "training pass");
    MLP_CUDA(m, launch_pdl(reduce_gradient_kernel, dim3((NPARAM + 63) / 64 + 1), dim3(256), 0, s, (const float*)m->part,
                           (const double*)m->loss_part, ctas, m->grad, m->loss),
             "gradient reduction");
    if (loss || grad) {
        double l = 0.0;
        if (loss) MLP_CUDA(m, cudaMemcpyAsync(&l, m->loss, 8, cudaMemcpyDeviceToHost, s), "copy loss");
        if (grad) MLP_CUDA(m, cudaMemcpyAsync(grad, m->grad, NPARAM * 4, cudaMemcpyDeviceToHost, s), "copy grad");
        rc = read_status(m);
        if (rc) return rc;
        if (loss) *loss = l / ((double)rows * NOUT);
    }
    return TVLBM_OK;
}

int tvlbm_mlp_adam(tvlbm_mlp* m, float lr, float beta1, float beta2, float eps) {
    if (!m || !(lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return mfail(m, TVLBM_EINVAL, "Adam needs lr >= 0, 0 <= beta < 1, eps > 0");
    cudaSetDevice(m->device);
    m->adam_t += 1;
    const float c1 = 1.0f - powf(beta1, (float)m->adam_t), c2 = 1.0f - powf(beta2, (float)m->adam_t);
    MLP_CUDA(m, launch_pdl(adam_kernel, dim3((NPARAM + 255) / 256), dim3(256), 0, m->stream, m->theta, m->m1, m->m2,
                           (const float*)m->grad, NPARAM, lr, beta1, beta2, eps, c1, c2, m->w1p, m->w2, m->w3p),
             "adam kernel");
    return TVLBM_OK;
}

const char* tvlbm_mlp_last_error(const tvlbm_mlp* m) { return m ? m->err : "null network"; }

}  // extern "C"

extern "C" int tvlbm_mlp_activation(const float* z, float* g, float* dg, int n, void* stream) {
    if (!z || n < 0) return TVLBM_EINVAL;
    if (n == 0) return TVLBM_OK;
    const int blocks = (n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024;
    activation_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(z, g, dg, n);
    return cudaGetLastError() == cudaSuccess ? TVLBM_OK : TVLBM_ECUDA;
}
