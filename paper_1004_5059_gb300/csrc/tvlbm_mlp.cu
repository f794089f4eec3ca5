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
// |error| <= 1.5e-7, odd in x; the reciprocal and the exponential (2^(s log2 e)) by the hardware's
// approximations without the handling of subnormal results (1 + p x >= 1; an exp(-x^2) that small adds
// nothing to 1).  The network stores its activations in BF16 (relative step 2^-8), so the error is
// invisible.  E2 = exp(-x^2) = exp(-z^2 / 2) also gives phi(z) = E2 / sqrt(2 pi).
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
constexpr float kLog2e = 1.4426950408889634f;
// For a pair in packed FP32 (a packed multiply, add or fused multiply-add rounds each lane as the scalar
// instruction; the reciprocal, the exponential, |x| and the sign stay scalar; the polynomial's sign is
// in its coefficients): 1 + erf(x), and exp(-x^2).
__device__ __forceinline__ float2 erf2_plus1(float2 x, float2& e2) {
    const float2 ax = make_float2(fabsf(x.x), fabsf(x.y));
    const float2 d = __ffma2_rn(make_float2(0.3275911f, 0.3275911f), ax, make_float2(1.0f, 1.0f));
    const float2 t = make_float2(rcp_approx(d.x), rcp_approx(d.y));
    float2 q = __ffma2_rn(t, make_float2(-1.061405429f, -1.061405429f), make_float2(1.453152027f, 1.453152027f));
    q = __ffma2_rn(t, q, make_float2(-1.421413741f, -1.421413741f));
    q = __ffma2_rn(t, q, make_float2(0.284496736f, 0.284496736f));
    q = __ffma2_rn(t, q, make_float2(-0.254829592f, -0.254829592f));
    const float2 neg_poly = __fmul2_rn(t, q);
    const float2 s = __fmul2_rn(__fmul2_rn(ax, ax), make_float2(-kLog2e, -kLog2e));
    e2 = make_float2(ex2_approx(s.x), ex2_approx(s.y));
    const float2 r = __ffma2_rn(neg_poly, e2, make_float2(1.0f, 1.0f));
    return __fadd2_rn(make_float2(1.0f, 1.0f), make_float2(copysignf(r.x, x.x), copysignf(r.y, x.y)));
}
// Two GELUs (inference).
__device__ __forceinline__ float2 gelu2_f(float2 z) {
    float2 e2;
    const float2 er1 = erf2_plus1(__fmul2_rn(z, make_float2(0.70710678118654752f, 0.70710678118654752f)), e2);
    return __fmul2_rn(__fmul2_rn(make_float2(0.5f, 0.5f), z), er1);
}
// Two GELUs and their derivatives (training): the same g as gelu2_f's.
__device__ __forceinline__ float2 gelu2_both(float2 z, float2& dg) {
    float2 e2;
    const float2 half = make_float2(0.5f, 0.5f);
    const float2 er1 = erf2_plus1(__fmul2_rn(z, make_float2(0.70710678118654752f, 0.70710678118654752f)), e2);
    dg = __ffma2_rn(__fmul2_rn(z, make_float2(0.39894228040143268f, 0.39894228040143268f)), e2, __fmul2_rn(half, er1));
    return __fmul2_rn(__fmul2_rn(half, z), er1);
}
// The kernels' own functions on a caller's entries, in pairs (an odd last entry beside itself): g by the
// forward epilogues', g' by the training epilogues'.
__global__ void activation_kernel(const float* __restrict__ z, float* __restrict__ g, float* __restrict__ dg, int n) {
    for (int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x); i < n; i += 2 * gridDim.x * blockDim.x) {
        const bool two = i + 1 < n;
        const float2 v = make_float2(z[i], z[two ? i + 1 : i]);
        if (g) {
            const float2 r = gelu2_f(v);
            g[i] = r.x;
            if (two) g[i + 1] = r.y;
        }
        if (dg) {
            float2 d;
            gelu2_both(v, d);
            dg[i] = d.x;
            if (two) dg[i + 1] = d.y;
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
// epilogue threads write them in the same swizzled K-major layout the next MMA reads, over X and W1,
// which layer 1 has consumed.  Every layer accumulates in the same 128 TMEM columns (its predecessor's
// have been read by then).  69 KB and 40 registers: three CTAs per SM, so that two tiles' epilogues
// run while a third waits for its products (65 536 rows of features: 21.4 us; 24.5 us with two CTAs, H
// and a second accumulator of their own, and exponentials that handled subnormal results).  Launched
// without programmatic overlap: blocks waiting for the kernel before take the room of its last ones
// (the learned 256 x 256 step 33.9 instead of 32.0 us).
struct FusedCfg {
    static constexpr int X_OFF = 0, W1_OFF = 16384, W2_OFF = 32768, W3_OFF = 65536, H_OFF = 0;
    static constexpr int BYTES = W3_OFF + 4096;
    static constexpr int SMEM = BYTES + 1024;
    static constexpr uint32_t TX = 16384 + 16384 + 32768 + 4096;
    static constexpr uint32_t TMEM_COLS = 128;
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
        v[e] = (*(f.m6 + q * n + (long long)yy * f.nx + xx) - f.mu[q]) * f.isg[q];
    }
}

// FEAT: the input tile is built by the CTA's threads from the closure's moments (MlpFeatures)
// instead of loaded by TMA; thread (row r, warpgroup g) makes features 16 g .. 16 g + 15 of row
// r with the closure features kernel's arithmetic, so the inputs are the same BF16 values.
template <bool FEAT>
__global__ void __launch_bounds__(kFusedThreads, 3) mlp_fused_forward_kernel(const __grid_constant__ CUtensorMap mx,
                                                                const __grid_constant__ CUtensorMap mw1,
                                                                const __grid_constant__ CUtensorMap mw2,
                                                                const __grid_constant__ CUtensorMap mw3,
                                                                const float* __restrict__ theta, float* __restrict__ y,
                                                                int* status, const MlpFeatures feat) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (saddr(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t load_bar, mma_bar, end_bar;
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * BM;
    const float* b1 = theta + OFF_B1;
    const float* b2 = theta + OFF_B2;
    const float* b3 = theta + OFF_B3;
    if (tid == 0) {
        bar_init(&load_bar, 1);
        bar_init(&mma_bar, 1);
        bar_init(&end_bar, 1);
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
    // a hidden layer's epilogue: this thread's columns, the biases four at a time
    auto hidden = [&](const float* bias) {
#pragma unroll 1
        for (int c0 = cbeg; c0 < cend; c0 += 16) {
            float v[16];
            __syncwarp();
            tmem_ld16(taddr + (uint32_t)c0, v);
#pragma unroll
            for (int k = 0; k < 16; k += 4) {
                const float4 bk = *reinterpret_cast<const float4*>(bias + c0 + k);
                const float2 g0 = gelu2_f(__fadd2_rn(make_float2(v[k], v[k + 1]), make_float2(bk.x, bk.y)));
                const float2 g1 = gelu2_f(__fadd2_rn(make_float2(v[k + 2], v[k + 3]), make_float2(bk.z, bk.w)));
                v[k] = g0.x;
                v[k + 1] = g0.y;
                v[k + 2] = g1.x;
                v[k + 3] = g1.y;
            }
            store_h_sw128(hs, r, c0, v);
        }
    };
    if (ok) hidden(b1);
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
                    mma_bf16(tmem, sw128_desc(saddr(hs) + kc * 16384 + kk * 32),
                             sw128_desc(saddr(w2) + kc * 16384 + kk * 32), idesc, kc > 0 || kk > 0);
        }
        mma_commit(&mma_bar);
    }
    // layer 2 epilogue: H2 = g(Z2 + b2) over H1 (the MMA that read H1 has completed)
    ok = __syncthreads_and(ok && bar_wait(&mma_bar, 1)) != 0;
    tc_fence_after();
    if (ok) hidden(b2);
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
            for (int e = 0; e < 4; ++e) o[e] = 4 * q + e < NOUT ? v[4 * q + e] + __ldcg(b3 + 4 * q + e) : 0.0f;
            d[q] = make_float4(o[0], o[1], o[2], o[3]);
        }
    } else if (tid == 0 && !ok) {
        if (status) atomicOr(status, 1);
        // let the loads and products started so far end before the CTA exits (bounded)
        bar_wait(&load_bar, 0);
        mma_commit(&end_bar);
        bar_wait(&end_bar, 0);
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
// The products are tiny (0.14 MFLOP a row), so the chain of epilogues bounds it: 17 us for a tile, and
// one CTA per SM runs up to 152 tiles in that time.  A batch of 4096 rows takes 27 us (with the
// gradient reduction, 5.7 us, and Adam, 3.5) where thirteen kernels, one product each with its operands
// and their transposes through memory, took 155 us.
struct TrainCfg {
    static constexpr int X_OFF = 0, W1_OFF = 16384, W2_OFF = 32768, W3_OFF = 65536, H1_OFF = 69632, H2_OFF = 102400,
                         DY_OFF = 135168;
    static constexpr int BYTES = DY_OFF + 16384;  // 148 KB
    static constexpr int SMEM = BYTES + 1024;
    static constexpr uint32_t TX_W = 16384 + 32768 + 4096, TX_X = 16384;
    static constexpr uint32_t T_DW2 = 0, T_DW1 = 128, T_DW3 = 192, T_Y = 208, T_A = 256, T_B = 384;
    // the second half tile's weight gradients (`halves`, below), in columns that are free by then
    static constexpr uint32_t T_DW2H = T_A, T_DW1H = T_B, T_DW3H = 224;
    // one partial sum of the weight gradients, floats, the hidden unit that owns a TMEM lane running fastest
    // (so that a warp's stores are whole lines): dW1^T [64][128], dW2^T [128][128], dW3 [16][128]; and a
    // CTA's bias gradients of its four 32-row groups: db1 [4][128], db2 [4][128], db3 [4][16]
    static constexpr int P_W1 = 0, P_W2 = P_W1 + NH * NINP, P_W3 = P_W2 + NH * NH, P_SUM = P_W3 + NOUTP * NH;
    static constexpr int P_B1 = 0, P_B2 = P_B1 + 4 * NH, P_B3 = P_B2 + 4 * NH, P_BIAS = P_B3 + 4 * NOUTP;
    // Up to kHalfTiles tiles (8192 rows) every 64 rows give a partial sum of their own, beyond that every
    // CTA's tiles one; the partial sums are added in row order.  (64-row sums added in FP32 are the
    // summation that training runs have been reproduced with.)
    static constexpr int kHalfTiles = 64;
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
                                                                     const float* __restrict__ ystar, int tiles, int halves,
                                                                     float scale, float* __restrict__ part,
                                                                     float* __restrict__ bias_part,
                                                                     double* __restrict__ loss_part, int* status) {
    using Cfg = TrainCfg;
    static_assert(kFusedGroups == 4, "32 columns per thread and hidden layer");
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (saddr(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t w_bar, x_bar, mma_bar, end_bar;
    __shared__ __align__(16) float bias[2 * NH + NOUTP];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_launch_dependents();
    if (tid == 0) {
        bar_init(&w_bar, 1);
        bar_init(&x_bar, 1);
        bar_init(&mma_bar, 1);
        bar_init(&end_bar, 1);
        bar_init_fence();
    }
    pdl_wait();  // the weights (and the partial sums' readers) of the kernels before this one
    // TMEM only once the kernels before this one are complete: a block that held some while waiting for
    // them could keep one of theirs from allocating
    if (warp == 0) tmem_alloc(&tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
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
    uint32_t ph = 0;   // phase of mma_bar
    uint32_t xph = 0;  // phase of x_bar that the last input tile issued completes
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
    // D (+)= A^T B over the tile's 128 rows; with halves (one tile per CTA) rows 64 .. 127 into Dh
    auto rows_product = [&](uint32_t d, uint32_t dh, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
        mma_chain(tmem + d, a, b, 128, 128, BM / 32, idesc, accumulate);
        mma_chain(tmem + (halves ? dh : d), a + 128 * (BM / 32), b + 128 * (BM / 32), 128, 128, BM / 32, idesc, !halves);
    };
    const uint32_t kk = idesc_bf16_f32(BM, NH), kk16 = idesc_bf16_f32(BM, NOUTP);
    constexpr uint32_t A_MN = 1u << 15, B_MN = 1u << 16;
    float db1 = 0.0f, db2 = 0.0f, db3 = 0.0f;  // column sums of this warp's rows: column cbeg + lane (db3: lane)
    double loss = 0.0;
    bool first = true;

#pragma unroll 1
    for (int tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, first = false) {
        const int m0 = tile * BM;
        float4 ys[3];
        if (warp < 4) {  // the targets, long before they are needed
            const float* q = ystar + (size_t)(m0 + r) * NOUTP;
            if ((reinterpret_cast<uintptr_t>(ystar) & 15) == 0) {
#pragma unroll
                for (int k = 0; k < 3; ++k) ys[k] = __ldg(reinterpret_cast<const float4*>(q) + k);
            } else {
#pragma unroll
                for (int k = 0; k < 3; ++k) ys[k] = make_float4(q[4 * k], q[4 * k + 1], q[4 * k + 2], q[4 * k + 3]);
            }
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
                rows_product(Cfg::T_DW3, Cfg::T_DW3H, sw128_mn_desc(saddr(h2), 16384), sw128_mn_desc(saddr(dys), 16384),
                             kk16 | A_MN | B_MN, !first);
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
                rows_product(Cfg::T_DW2, Cfg::T_DW2H, sw128_mn_desc(saddr(h2), 16384), sw128_mn_desc(saddr(h1), 16384),
                             kk | A_MN | B_MN, !first);
            }
            mma_commit(&mma_bar);
        }
        products_done();
        if (ok) back(Cfg::T_B, g1, h1, db1);
        operands_ready();
        if (tid == 0) {
            if (ok)  // dW1 += dZ1^T X
                rows_product(Cfg::T_DW1, Cfg::T_DW1H, sw128_mn_desc(saddr(h1), 16384), sw128_mn_desc(saddr(xs), 16384),
                             idesc_bf16_f32(BM, NINP) | A_MN | B_MN, !first);
            mma_commit(&mma_bar);
        }
        products_done();
        if (tid == 0 && ok && tile + (int)gridDim.x < tiles) {
            bar_expect_tx(&x_bar, Cfg::TX_X);
            tma_load_2d(xs, &mx, &x_bar, 0, (tile + (int)gridDim.x) * BM);
            xph ^= 1;
        }
    }

    if (ok) {
        float v[16];
        auto drain = [&](uint32_t t0, float* q) {  // 16 columns of this thread's lane
            __syncwarp();
            tmem_ld16(taddr + t0, v);
#pragma unroll
            for (int k = 0; k < 16; ++k) q[k * NH + r] = v[k];
        };
        auto sums_out = [&](float* q, uint32_t dw1, uint32_t dw2, uint32_t dw3) {
            drain(dw2 + cbeg, q + Cfg::P_W2 + cbeg * NH);
            drain(dw2 + cbeg + 16, q + Cfg::P_W2 + (cbeg + 16) * NH);
            drain(dw1 + cbeg / 2, q + Cfg::P_W1 + cbeg / 2 * NH);
            if (warp < 4) drain(dw3, q + Cfg::P_W3);
        };
        float* q = part + (size_t)blockIdx.x * (halves ? 2 : 1) * Cfg::P_SUM;
        sums_out(q, Cfg::T_DW1, Cfg::T_DW2, Cfg::T_DW3);
        if (halves) sums_out(q + Cfg::P_SUM, Cfg::T_DW1H, Cfg::T_DW2H, Cfg::T_DW3H);
        float* qb = bias_part + (size_t)blockIdx.x * Cfg::P_BIAS;
        if (warp < 4) {
            if (lane < NOUTP) qb[Cfg::P_B3 + warp * NOUTP + lane] = db3;
            if (lane == 0) loss_part[blockIdx.x * 4 + warp] = loss;
        }
        qb[Cfg::P_B1 + (warp & 3) * NH + cbeg + lane] = db1;
        qb[Cfg::P_B2 + (warp & 3) * NH + cbeg + lane] = db2;
    } else if (tid == 0) {
        if (status) atomicOr(status, 1);
        // let the loads and products started so far end before the CTA exits (bounded)
        bar_wait(&w_bar, 0);
        bar_wait(&x_bar, xph);
        mma_commit(&end_bar);
        bar_wait(&end_bar, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, 512);
}

// ---- small kernels ---------------------------------------------------------------------------

// The gradient: a weight's `sums` partial sums in row order, a bias's sums over the CTAs' row groups;
// one thread per weight, 64 per block so that the blocks spread over the SMs.  The last block sums
// the loss.
__global__ void __launch_bounds__(64) reduce_gradient_kernel(const float* __restrict__ part, const float* __restrict__ bias_part,
                                                             const double* __restrict__ loss_part, int sums, int ctas,
                                                             float* __restrict__ grad, double* __restrict__ loss) {
    using Cfg = TrainCfg;
    pdl_launch_dependents();
    pdl_wait();
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
    // (a warp reads one line per partial sum; blocks beyond the weights' take the biases)
    const int t = blockIdx.x * 64 + threadIdx.x;
    if (t < Cfg::P_SUM) {
        float acc = 0.0f;
#pragma unroll 16
        for (int c = 0; c < sums; ++c) acc += __ldcg(part + (size_t)c * Cfg::P_SUM + t);
        if (t < Cfg::P_W2) {
            const int c = t / NH, r = t % NH;
            if (c < NIN) grad[OFF_W1 + r * NIN + c] = acc;
        } else if (t < Cfg::P_W3) {
            const int c = (t - Cfg::P_W2) / NH, r = (t - Cfg::P_W2) % NH;
            grad[OFF_W2 + r * NH + c] = acc;
        } else if (t - Cfg::P_W3 < NOUT * NH) {
            grad[OFF_W3 + t - Cfg::P_W3] = acc;
        }
        return;
    }
    // a bias per warp, its lanes sharing the CTAs' row groups, in compensated FP32 (each addition's
    // rounding error is kept by the two-sum identity; FP64 would take 64 cycles a warp instruction).
    // The last bit of a bias flips a BF16 rounding now and then, and a training run amplifies that (4096
    // rows, 16 iterations: gradients up to 3e-4 apart, as two runs with atomic sums were); plain sums
    // in row order lie further from either.
    const int k = (t - Cfg::P_SUM) >> 5, lane = threadIdx.x & 31;  // b1, b2, b3
    if (k >= 2 * NH + NOUT) return;
    const int boff = k < NH ? Cfg::P_B1 + k : k < 2 * NH ? Cfg::P_B2 + k - NH : Cfg::P_B3 + k - 2 * NH;
    const int ld = k < 2 * NH ? NH : NOUTP;
    float a = 0.0f, err = 0.0f;
    const auto add = [&](float v) {
        const float sum = __fadd_rn(a, v), av = __fadd_rn(sum, -a);
        err = __fadd_rn(err, __fadd_rn(__fadd_rn(a, -__fadd_rn(sum, -av)), __fadd_rn(v, -av)));
        a = sum;
    };
#pragma unroll 4
    for (int c = lane; c < 4 * ctas; c += 32) add(__ldcg(bias_part + (size_t)(c >> 2) * Cfg::P_BIAS + boff + (c & 3) * ld));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float other = __shfl_down_sync(0xffffffffu, a, o);
        err = __fadd_rn(err, __shfl_down_sync(0xffffffffu, err, o));
        add(other);
    }
    if (lane == 0) grad[k < NH ? OFF_B1 + k : k < 2 * NH ? OFF_B2 + k - NH : OFF_B3 + k - 2 * NH] = __fadd_rn(a, err);
}
constexpr int kReduceBlocks = TrainCfg::P_SUM / 64 + (2 * NH + NOUT + 1) / 2 + 1;
static_assert(TrainCfg::P_SUM % 64 == 0, "whole blocks of weights");

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
    float *theta, *m1, *m2, *grad, *part, *bias_part;
    double *loss, *loss_part;
    int* status;
    bf16 *w1p, *w2, *w3p;
    float* ybuf;
    int ctas;  // most CTAs of a training pass (one per SM)
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
    MLP_CUDA(m, launch_as(false, mlp_fused_forward_kernel<false>, dim3(tiles), dim3(kFusedThreads), FusedCfg::SMEM, m->stream, mx,
                           mw1, mw2, mw3, (const float*)m->theta, y, m->status, none),
             "fused forward");
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
    MLP_CUDA(m, launch_as(false, mlp_fused_forward_kernel<true>, dim3(tiles), dim3(kFusedThreads), FusedCfg::SMEM, m->stream, mx,
                           mw1, mw2, mw3, (const float*)m->theta, y, m->status, feat),
             "fused forward with features");
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
    const int half_tiles = max_rows / BM < TrainCfg::kHalfTiles ? max_rows / BM : TrainCfg::kHalfTiles;
    const size_t sums = m->ctas > 2 * half_tiles ? m->ctas : 2 * half_tiles;  // partial sums of a pass
    const size_t o_part = take(sums * TrainCfg::P_SUM * 4), o_bias = take((size_t)m->ctas * TrainCfg::P_BIAS * 4),
                 o_losses = take((size_t)m->ctas * 4 * 8), o_loss = take(8), o_status = take(4);
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
    m->bias_part = (float*)(b + o_bias);
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
    const int halves = tiles <= TrainCfg::kHalfTiles && tiles <= m->ctas ? 1 : 0;  // (one tile per CTA)
    CUtensorMap mx, mw1, mw2, mw3;
    if (!bf16_map(&mx, x, NINP, rows, NINP, BM) || !bf16_map(&mw1, m->w1p, NINP, NH, NINP, NH) ||
        !bf16_map(&mw2, m->w2, NH, NH, NH, NH) || !bf16_map(&mw3, m->w3p, NH, NOUTP, NH, NOUTP))
        return mfail(m, TVLBM_EINVAL, "TMA descriptor rejected (alignment of x?)");
    static bool attr_set[64] = {};
    if (m->device < 0 || m->device >= 64 || !attr_set[m->device]) {
        MLP_CUDA(m, cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TrainCfg::SMEM),
                 "training kernel attribute");
        if (m->device >= 0 && m->device < 64) attr_set[m->device] = true;
    }
    MLP_CUDA(m, launch_pdl(mlp_train_kernel, dim3(ctas), dim3(kFusedThreads), TrainCfg::SMEM, s, mx, mw1, mw2, mw3,
                           (const float*)m->theta, ystar, tiles, halves, 2.0f / ((float)rows * (float)NOUT), m->part,
                           m->bias_part, m->loss_part, m->status),
             "training pass");
    MLP_CUDA(m, launch_pdl(reduce_gradient_kernel, dim3(kReduceBlocks), dim3(64), 0, s, (const float*)m->part,
                           (const float*)m->bias_part, (const double*)m->loss_part, halves ? 2 * tiles : ctas, ctas, m->grad,
                           m->loss),
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
