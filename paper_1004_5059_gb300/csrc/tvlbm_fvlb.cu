// The paper's own evolution scheme (Sec. "The TVLBM Evolution scheme", Eq. FVLB) on the unit
// grid: an explicit Euler step f(t + dt) = f + dt (Omega_bar - c . grad f) with the second-order
// stencils over the eight neighbours P1..P8 of P0 (east, north, west, south, north-east,
// north-west, south-west, south-east):
//   d_x f ~ 3/8 (f1 - f3) + 1/16 (f5 - f6 - f7 + f8),  d_y f ~ 3/8 (f2 - f4) + 1/16 (f5 + f6 - f7 - f8),
//   Omega_bar ~ 9/16 Omega(0) + 3/32 (Omega(1..4)) + 1/64 (Omega(5..8)),
// and the collision term of Eq. OMEGAFVLB: BGK plus the Prandtl-number term
// (1 / tau_g) f_eq / (rho T^2) Pi : (c - u)(c - u), applied without its components along the
// collision invariants (an exact Maxwellian has none; a truncated equilibrium leaves a residue).
// FP32: one fused kernel per step (fv_fused_kernel: warps march over strips of columns, the collision
// term in registers), or, as the two-kernel form, the collision term of every cell (stored with the
// periodic frame images in a population-sized buffer) and then the update, which reads both fields
// at the 3 x 3 cells.  Both give the same populations.  FP64 runs two kernels in either form.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "tvlbm.h"
#include "tvlbm_ctx.h"
#include "tvlbm_kernels.cuh"
#include "tvlbm_tiled.cuh"

using namespace tvlbm;

namespace {

// The scheme's constants in both precisions (a double constant in FP32 code costs a conversion on
// the FP64 pipe: 64 cycles per warp instruction on sm_103a).
template <class R>
struct FvConst {
    R it, itg;          // (dt / 64) / tau and (dt / 64) / tau_g
    R dt16;             // dt / 16
    R g00, g03, g33;    // inverse Gram matrix of the collision invariants (1, c_x, c_y, |c|^2) in
    R g11, g22;         //   sum_l w_l g_l h_l; by the set's mirror symmetry only 1 and |c|^2 couple
};
struct FvParams {
    FvConst<float> f;
    FvConst<double> d;
    int prandtl;
    int pscale;         // relaxation times divided by the local pressure: tau -> tau / p, p = rho T
    int walls;          // channel: wall nodes on the first and last rows
    const double* ysc;  // per row the y factor of its stencil [ny] (see fv_march), or null for unit spacing
};
template <class R>
__device__ __forceinline__ const FvConst<R>& fv_const(const FvParams& p) {
    if constexpr (std::is_same<R, double>::value) return p.d; else return p.f;
}

// Wall imposition parameters: wall velocity and temperature per side, the Newton-Raphson mode.
struct WallParams {
    double u[2], T[2];
    // sum over the outgoing y-nodes of w_j E_jb, w_j |x_j| E_jb and w_j x_j^2 E_jb for b = 0, 2, 4
    // (E_jb = He_b(x_j) / b!; the same for both walls)
    double k0[3], kn[3], k2[3];
    int exact, iters;
    double* eq;  // [2][nx][2] wall equilibria (u_eq, T_eq), warm start of the next imposition
};

// Two populations side by side, the velocities (i, j) and (i, N1 - 1 - j) mirrored in y: packed
// FP32 instructions (each lane rounded as the scalar one), or two FP64 ones.  The rounding is
// spelled out (no contraction), so that every kernel that runs this arithmetic gets the same bits.
template <class R>
struct Pair {
    R x, y;
};
__device__ __forceinline__ Pair<float> fma2(Pair<float> a, Pair<float> b, Pair<float> c) {
    const float2 r = __ffma2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y), make_float2(c.x, c.y));
    return {r.x, r.y};
}
__device__ __forceinline__ Pair<float> add2(Pair<float> a, Pair<float> b) {
    const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    return {r.x, r.y};
}
__device__ __forceinline__ Pair<float> mul2(Pair<float> a, Pair<float> b) {
    // as PTX: the compiler may contract the intrinsic's product with a following sum
    Pair<float> d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ Pair<double> fma2(Pair<double> a, Pair<double> b, Pair<double> c) {
    return {fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}
__device__ __forceinline__ Pair<double> add2(Pair<double> a, Pair<double> b) {
    return {__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y)};
}
__device__ __forceinline__ Pair<double> mul2(Pair<double> a, Pair<double> b) {
    return {__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)};
}
__device__ __forceinline__ Pair<float> sub2(Pair<float> a, Pair<float> b) {
    const float2 r = f2sub(make_float2(a.x, a.y), make_float2(b.x, b.y));
    return {r.x, r.y};
}
template <class R> __device__ __forceinline__ Pair<R> bc(R v) { return {v, v}; }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }

// Pairs of a velocity set: HP y-groups of N1 pairs; for an odd node count the last group's mirror
// is itself and its y lane holds nothing (zero weight, zero value).
template <int N1> constexpr int fv_hp() { return (N1 + 1) / 2; }
template <int N1> __host__ __device__ constexpr bool fv_single(int g) { return 2 * g == N1 - 1; }

// Sums over i of one y-group: v, x_i v, x_i^2 v.
template <int N1, class R>
__device__ __forceinline__ void fv_group_sums(const Pair<R> (&v)[N1], const KParams& p, Pair<R>& r, Pair<R>& rx, Pair<R>& rxx) {
    r = v[0];
    rx = mul2(bc<R>(kx<R>(p, 0)), v[0]);
    rxx = mul2(bc<R>(kx2<R>(p, 0)), v[0]);
#pragma unroll
    for (int i = 1; i < N1; ++i) {
        r = add2(r, v[i]);
        rx = fma2(bc<R>(kx<R>(p, i)), v[i], rx);
        rxx = fma2(bc<R>(kx2<R>(p, i)), v[i], rxx);
    }
}

// Collision term of Eq. OMEGAFVLB at one cell from its populations s, times dt / 64 (the weight of
// a corner cell in the 9-point average and the Euler step): BGK, plus with tau_g the Prandtl term
// (1 / tau_g) f_eq / (rho T^2) Pi : (c - u)(c - u) less its components along the collision invariants.
// The work per population is what bounds both precisions (FP32: issue slots; FP64: 64 cycles per
// warp instruction), hence the pairs, the separable sums and the closed forms:
//  * Pi is traceless and the equilibrium's second moments are exact for every set, so Pi_xx = -Pi_yy
//    = (sum f (c_x^2 - c_y^2) - rho (u_x^2 - u_y^2)) / 2 and Pi_xy = sum f c_x c_y - rho u_x u_y;
//  * moments of f_eq up to order N are those of the Maxwellian, for which the Prandtl term carries
//    no invariant.  What a set truncated at order N = 3 leaves is the fourth-order part of the
//    energy, sum |c|^2 f_eq Pi : (c - u)(c - u) = -rho (Pi_xx (h_4x - h_4y) + 2 Pi_xy (h_3x h_1y +
//    h_1x h_3y)), h_n the Hermite factors of u and T; N = 5 leaves nothing; N = 2 also misses the
//    third order, and there the moments are summed.
template <int N1, class R>
__device__ __forceinline__ void fv_omega_cell(const Pair<R> (&s)[fv_hp<N1>()][N1], const KParams& p, const FvParams& fp,
                                              Pair<R> (&w)[fv_hp<N1>()][N1]) {
    constexpr int HP = fv_hp<N1>(), N = N1 - 1;
    const FvConst<R>& fc = fv_const<R>(fp);
    R rho = 0, jx = 0, jy = 0, exx = 0, eyy = 0, exy = 0;
#pragma unroll
    for (int g = 0; g < HP; ++g) {
        Pair<R> r, rx, rxx;
        fv_group_sums<N1, R>(s[g], p, r, rx, rxx);
        const R yj = kx<R>(p, g), rs = add_(r.x, r.y);
        rho = add_(rho, rs);
        jx = add_(jx, add_(rx.x, rx.y));
        jy = fma(yj, add_(r.x, -r.y), jy);
        exy = fma(yj, add_(rx.x, -rx.y), exy);
        eyy = fma(kx2<R>(p, g), rs, eyy);
        exx = add_(exx, add_(rxx.x, rxx.y));
    }
    const R inv = R(1) / rho;
    const R ux = mul_(jx, inv), uy = mul_(jy, inv);
    const R T = mul_(R(0.5), fma(add_(exx, eyy), inv, -fma(ux, ux, mul_(uy, uy))));
    const R th = add_(T, R(-1));
    R hx[N + 1], hy[N + 1];
    hx[0] = R(1);
    hy[0] = R(1);
    hx[1] = ux;
    hy[1] = uy;
#pragma unroll
    for (int n = 1; n < N; ++n) {
        const R nt = n == 1 ? th : mul_(R(n), th);
        hx[n + 1] = n == 1 ? fma(ux, ux, th) : fma(ux, hx[n], mul_(nt, hx[n - 1]));
        hy[n + 1] = n == 1 ? fma(uy, uy, th) : fma(uy, hy[n], mul_(nt, hy[n - 1]));
    }
    // f_eq = w rho (1 + SX_i + P_jN + sum_a X_ia P_j,N-a)  (see cell_equilibrium)
    R X[N1][N], SX[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) {
        SX[i] = R(1);
#pragma unroll
        for (int a = 1; a <= N; ++a) {
            if (a < N) {
                X[i][a] = mul_(hx[a], kE<R>(p, i, a));
                SX[i] = add_(SX[i], X[i][a]);
            } else {
                SX[i] = fma(hx[a], kE<R>(p, i, a), SX[i]);
            }
        }
    }
    const R ps = fp.pscale ? mul_(rho, T) : R(1);
    const R it = mul_(fc.it, ps);
    // o = f_eq (it + qx_i + qy_j + c_i dy_j) - it f - w (ex_i + ey_j)
    R qx[N1], cxy[N1], ex[N1], ayy = 0, b3 = 0;
    if (fp.prandtl) {
        const R pxx = mul_(R(0.5), fma(-rho, fma(ux, ux, -mul_(uy, uy)), add_(exx, -eyy)));
        const R pxy = fma(-rho, mul_(ux, uy), exy);
        const R sc = mul_(mul_(fc.itg, ps), mul_(inv, R(1) / mul_(T, T)));
        const R axx = mul_(sc, pxx), axy = mul_(mul_(R(2), sc), pxy);
        ayy = -axx;
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            const R dx = add_(kx<R>(p, i), -ux);
            qx[i] = fma(axx, mul_(dx, dx), it);
            cxy[i] = mul_(axy, dx);
        }
        if constexpr (N == 3) {
            const R h4x = fma(ux, hx[3], mul_(mul_(R(3), th), hx[2])), h4y = fma(uy, hy[3], mul_(mul_(R(3), th), hy[2]));
            const R m3 = mul_(-rho, fma(axx, add_(h4x, -h4y), mul_(axy, fma(hx[3], uy, mul_(ux, hy[3])))));
            const R b0 = mul_(fc.g03, m3);
            b3 = mul_(fc.g33, m3);
#pragma unroll
            for (int i = 0; i < N1; ++i) ex[i] = fma(b3, kx2<R>(p, i), b0);
        }
    }
    R m0 = 0, m1 = 0, m2 = 0, m3 = 0;  // N = 2
#pragma unroll
    for (int g = 0; g < HP; ++g) {
        Pair<R> P[N + 1];
        P[0] = bc<R>(R(0));
#pragma unroll
        for (int a = 1; a <= N; ++a) P[a] = fma2(bc<R>(hy[a]), Pair<R>{kE<R>(p, g, a), kE<R>(p, N1 - 1 - g, a)}, P[a - 1]);
        const R wj = kw<R>(p, g);
        const R wjr = mul_(wj, fp.prandtl ? rho : mul_(rho, it));
        const Pair<R> W = {wjr, fv_single<N1>(g) ? R(0) : wjr};
        const Pair<R> dy = {add_(kx<R>(p, g), -uy), add_(-kx<R>(p, g), -uy)};
        const Pair<R> dy2 = mul2(dy, dy);
        const R ey = mul_(b3, kx2<R>(p, g));
        Pair<R> raw[N1];
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            Pair<R> phi = add2(bc<R>(SX[i]), P[N]);
#pragma unroll
            for (int a = 1; a < N; ++a) phi = fma2(bc<R>(X[i][a]), P[N - a], phi);
            const Pair<R> eq = mul2(mul2(bc<R>(kw<R>(p, i)), W), phi);  // f_eq (without the Prandtl term: it f_eq)
            if (fp.prandtl) {
                const Pair<R> q = fma2(bc<R>(cxy[i]), dy, fma2(bc<R>(ayy), dy2, bc<R>(qx[i])));
                if constexpr (N == 3) {
                    const R wl = mul_(wj, -kw<R>(p, i));
                    w[g][i] = fma2(eq, q, fma2(bc<R>(-it), s[g][i], bc<R>(mul_(wl, add_(ex[i], ey)))));
                } else {
                    w[g][i] = fma2(eq, q, mul2(bc<R>(-it), s[g][i]));
                    if constexpr (N == 2) raw[i] = mul2(eq, add2(q, bc<R>(-it)));
                }
            } else {
                w[g][i] = fma2(bc<R>(-it), s[g][i], eq);
            }
        }
        if constexpr (N == 2) {
            if (fp.prandtl) {
                Pair<R> r, rx, rxx;
                fv_group_sums<N1, R>(raw, p, r, rx, rxx);
                const R rs = add_(r.x, r.y);
                m0 = add_(m0, rs);
                m1 = add_(m1, add_(rx.x, rx.y));
                m2 = fma(kx<R>(p, g), add_(r.x, -r.y), m2);
                m3 = fma(kx2<R>(p, g), rs, add_(m3, add_(rxx.x, rxx.y)));
            }
        }
    }
    if constexpr (N == 2) {
        if (fp.prandtl) {
            const R c0 = fma(fc.g00, m0, mul_(fc.g03, m3)), c3 = fma(fc.g03, m0, mul_(fc.g33, m3));
            const R c1 = mul_(fc.g11, m1), c2 = mul_(fc.g22, m2);
#pragma unroll
            for (int i = 0; i < N1; ++i) ex[i] = fma(kx<R>(p, i), fma(c3, kx<R>(p, i), c1), c0);
#pragma unroll
            for (int g = 0; g < HP; ++g) {
                const R yj = kx<R>(p, g), wj = kw<R>(p, g), y2 = mul_(c3, kx2<R>(p, g));
                const Pair<R> ey = {fma(c2, yj, y2), fma(-c2, yj, y2)};
#pragma unroll
                for (int i = 0; i < N1; ++i) {
                    const R wl = mul_(wj, -kw<R>(p, i));
                    w[g][i] = fma2(Pair<R>{wl, fv_single<N1>(g) ? R(0) : wl}, add2(bc<R>(ex[i]), ey), w[g][i]);
                }
            }
        }
    }
}

// ---- the update of Eq. FVLB, row by row --------------------------------------------------------
// With dxr = f_E - f_W, sm = 6 f_0 + f_E + f_W and om = 6 o_0 + o_E + o_W per row (o the collision
// term times dt / 64), both 9-point stencils are separable: the row at the cell's own height gives
// f_0 + 6 A, A = om - (c_x dt / 16) dxr, and the rows below and above give A -+ k sm with
// k = c_y dt ysc / 16.  The increments are summed first and f_0 is added last (read once more), so
// that a step rounds once relative to f.  A wall node of a channel takes the one-sided stencils of Eq. FVLB2 for the
// populations arriving at the wall (c . n <= 0; the leaving ones keep their imposed values): twice
// A of its neighbour row, and k (sm_neighbour - sm_own).
// The y factor per row: 2 / (dy_y + dy_{y-1}) inside, 2 / dy at a wall node; without a table 1, 2.
__device__ __forceinline__ int fv_wall_of(const KParams& p, const FvParams& fp, int y) {
    return fp.walls ? (y == 0 ? 1 : (y == p.ny - 1 ? 2 : 0)) : 0;
}
template <class R>
__device__ __forceinline__ R fv_kfac(const FvParams& fp, int y, int wall) {  // dt ysc / 16 of target row y
    const R d = fv_const<R>(fp).dt16;
    return mul_(d, fp.ysc ? (R)__ldg(fp.ysc + y) : (wall ? R(2) : R(1)));
}

// March of one column segment over output rows [y0, y1): rows from one below to one above are
// taken in turn, each once, its contributions to the rows around it carried in registers.
// PN pairs per thread (a whole cell: g = 0 .. HP - 1, i = 0 .. N1 - 1; the index functions ig, gg
// give them).  src.row(y) moves to a row, src.get(q, ...) supplies a pair's values at the column
// and beside it, src.own(q, y) the one at the column of row y; put(y, out) takes a finished row.  WALLS:
// the domain may be a channel.  Both FP32 forms run this one function, so they give the same bits (FP64
// runs fv_update64_kernel in either form).
template <int N1, int PN, class R, bool WALLS, class IG, class GG, class Src, class Put>
__device__ __forceinline__ void fv_march(const KParams& p, const FvParams& fp, int y0, int y1, const IG& ig, const GG& gg,
                                         Src& src, const Put& put) {
    Pair<R> own[PN];  // f_0 of the row whose output is pending
    Pair<R> pend[PN], Lp[PN];
    const int ra = WALLS && fp.walls ? max(y0 - 1, 0) : y0 - 1, rb = WALLS && fp.walls ? min(y1, p.ny - 1) : y1;
    const R dt16 = fv_const<R>(fp).dt16;
#pragma unroll
    for (int q = 0; q < PN; ++q) Lp[q] = pend[q] = bc<R>(R(0));
#pragma unroll 1
    for (int r = ra; r <= rb; ++r) {
        src.row(r);
        const int wu = WALLS && r > ra ? fv_wall_of(p, fp, r - 1) : 0;               // the row below (its upper neighbour is r)
        const int wl = WALLS && (r + 1 < p.ny || !fp.walls) ? fv_wall_of(p, fp, r + 1) : 0;  // the row above
        const int wo = WALLS ? fv_wall_of(p, fp, r) : 0;
        const bool ysc = WALLS && (fp.ysc != nullptr || fp.walls);
        R kU = dt16, kL = dt16;
        if (ysc) {
            if (r > ra) kU = fv_kfac<R>(fp, r - 1, wu);
            if (r < rb) kL = fv_kfac<R>(fp, r + 1, wl);
        }
        Pair<R> out[PN];
        if (wu | wl | wo) {  // next to or at a wall node
            const R kO = wo ? fv_kfac<R>(fp, r, wo) : R(0);
#pragma unroll
            for (int q = 0; q < PN; ++q) {
                const R cx = kx<R>(p, ig(q)), yj = kx<R>(p, gg(q));
                const Pair<R> cy = {yj, -yj};
                Pair<R> f0, fE, fW, o0, oE, oW;
                src.get(q, f0, fE, fW, o0, oE, oW);
                const Pair<R> dxr = sub2(fE, fW), sm = fma2(bc<R>(R(6)), f0, add2(fE, fW));
                const Pair<R> A = fma2(bc<R>(mul_(cx, -dt16)), dxr, fma2(bc<R>(R(6)), o0, add2(oE, oW)));
                const Pair<R> B = mul2(bc<R>(R(6)), A);
                const Pair<R> A2 = add2(A, A);
                const Pair<R> U = fma2(mul2(cy, bc<R>(-kU)), sm, wu ? A2 : A);
                const Pair<R> L = fma2(mul2(cy, bc<R>(kL)), sm, wl ? A2 : A);
                Pair<R> o = add2(pend[q], U);
                if (wu) {  // leaving populations (c . n > 0) keep their imposed values
                    const R sg = wu == 1 ? R(1) : R(-1);
                    if (mul_(sg, cy.x) > R(0)) o.x = R(0);
                    if (mul_(sg, cy.y) > R(0)) o.y = R(0);
                }
                out[q] = o;
                Pair<R> b = B;
                if (wo) {
                    const R sg = wo == 1 ? R(1) : R(-1);
                    b = fma2(mul2(cy, bc<R>(mul_(sg, kO))), sm, wo == 2 ? fma2(bc<R>(R(6)), A, Lp[q]) : B);
                    if (mul_(sg, cy.x) > R(0)) b.x = R(0);
                    if (mul_(sg, cy.y) > R(0)) b.y = R(0);
                } else if (r > ra) {
                    b = fma2(bc<R>(R(6)), A, Lp[q]);
                }
                pend[q] = b;
                Lp[q] = L;
            }
        } else {
#pragma unroll
            for (int q = 0; q < PN; ++q) {
                const R cx = kx<R>(p, ig(q)), yj = kx<R>(p, gg(q));
                const Pair<R> cy = {yj, -yj};
                Pair<R> f0, fE, fW, o0, oE, oW;
                src.get(q, f0, fE, fW, o0, oE, oW);
                const Pair<R> dxr = sub2(fE, fW), sm = fma2(bc<R>(R(6)), f0, add2(fE, fW));
                const Pair<R> A = fma2(bc<R>(mul_(cx, -dt16)), dxr, fma2(bc<R>(R(6)), o0, add2(oE, oW)));
                out[q] = add2(pend[q], fma2(mul2(cy, bc<R>(-kU)), sm, A));
                pend[q] = fma2(bc<R>(R(6)), A, Lp[q]);
                Lp[q] = fma2(mul2(cy, bc<R>(kL)), sm, A);
            }
        }
        if (r > ra && r - 1 >= y0) {
#pragma unroll
            for (int q = 0; q < PN; ++q) {
                if constexpr (Src::kCarry) out[q] = add2(own[q], out[q]);
                else out[q] = add2(src.own(q, r - 1), out[q]);
            }
            put(r - 1, out);
        }
        if constexpr (Src::kCarry) {
#pragma unroll
            for (int q = 0; q < PN; ++q) own[q] = src.cur(q);
        }
    }
    if (WALLS && fp.walls && y1 == p.ny) {
#pragma unroll
        for (int q = 0; q < PN; ++q) pend[q] = add2(src.cur(q), pend[q]);
        put(p.ny - 1, pend);
    }
}

// ---- two-kernel form -----------------------------------------------------------------------------
template <int N1, class C>
__device__ __forceinline__ void fv_load_cell(const typename C::T* fb, long long plane, Pair<typename C::R> (&s)[fv_hp<N1>()][N1]) {
    using R = typename C::R;
#pragma unroll
    for (int g = 0; g < fv_hp<N1>(); ++g)
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            s[g][i].x = C::ld(fb + (long long)(i + N1 * g) * plane);
            s[g][i].y = fv_single<N1>(g) ? R(0) : (R)C::ld(fb + (long long)(i + N1 * (N1 - 1 - g)) * plane);
        }
}
template <int N1, class R>
__device__ __forceinline__ void fv_unpair(const Pair<R> (&v)[fv_hp<N1>()][N1], R (&s)[N1 * N1]) {
#pragma unroll
    for (int g = 0; g < fv_hp<N1>(); ++g)
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            s[i + N1 * g] = v[g][i].x;
            if (!fv_single<N1>(g)) s[i + N1 * (N1 - 1 - g)] = v[g][i].y;
        }
}

// The collision term of every cell, with its frame images: one warp per 32 columns and row.  In FP64 a warp
// is alone in its block, so that small grids (a channel of 64 x 61 nodes) spread over as many SM
// partitions as they can; in FP32 four make a block, since starting a block takes about 1.1 ns, more than
// a warp of so little work leaves (see launch_fv).
template <int N1, class C>
__global__ void __launch_bounds__(128) fv_omega_kernel(const typename C::T* __restrict__ f, typename C::T* __restrict__ om,
                                                      const KParams p, const FvParams fp) {
    using R = typename C::R;
    pdl_launch_dependents();
    pdl_wait();
    const int gx = (p.nx + 31) / 32, by = blockIdx.x / gx, x = (blockIdx.x - by * gx) * 32 + threadIdx.x;
    const int y = by * blockDim.y + threadIdx.y;
    if (x >= p.nx || y >= p.ny) return;
    Pair<R> s[fv_hp<N1>()][N1], w[fv_hp<N1>()][N1];
    fv_load_cell<N1, C>(f + sidx(p, 0, x, y), p.plane, s);
    fv_omega_cell<N1, R>(s, p, fp, w);
    R o[N1 * N1];
    fv_unpair<N1, R>(w, o);
    store_collided<N1, C>(om, geom_of(p), x, y, o);
}

// Row source of the update: a pair of velocities of both fields in memory (two: false for a y-node
// without a mirror, whose second lane of the pair is not used).
template <class C>
struct FvGlobalSrc {
    using R = typename C::R;
    static constexpr bool kCarry = true;
    const typename C::T *fa, *fb, *oa, *ob;  // the column's elements of row 0
    long long pitch, at;
    bool two;
    Pair<R> f0, fE, fW, o0, oE, oW;
    __device__ __forceinline__ void row(int r) {
        at = r * pitch;
        f0.x = C::ld(fa + at);
        fE.x = C::ld(fa + at + 1);
        fW.x = C::ld(fa + at - 1);
        o0.x = C::ld(oa + at);
        oE.x = C::ld(oa + at + 1);
        oW.x = C::ld(oa + at - 1);
        if (two) {
            f0.y = C::ld(fb + at);
            fE.y = C::ld(fb + at + 1);
            fW.y = C::ld(fb + at - 1);
            o0.y = C::ld(ob + at);
            oE.y = C::ld(ob + at + 1);
            oW.y = C::ld(ob + at - 1);
        }
    }
    __device__ __forceinline__ Pair<R> cur(int) const { return f0; }
    __device__ __forceinline__ Pair<R> own(int, int) const { return f0; }  // (carried by the march)
    __device__ __forceinline__ void get(int, Pair<R>& f, Pair<R>& e, Pair<R>& w, Pair<R>& o, Pair<R>& p, Pair<R>& q) const {
        f = f0;
        e = fE;
        w = fW;
        o = o0;
        p = oE;
        q = oW;
    }
};

// The update from both fields in memory: one thread per (column, pair of velocities), marching over
// `seg` rows; the warps of a block take segments one above the other.  A periodic domain has its own
// instantiation: the tests for wall rows were a third of a row's instructions (512 x 512 D2Q9 15.5 us against 12.6),
// and a warp away from the edges stores without looking for images (11.6).
template <int N1, class C, bool WALLS>
__global__ void __launch_bounds__(128) fv_update_kernel(const typename C::T* __restrict__ f,
                                                       const typename C::T* __restrict__ om,
                                                       typename C::T* __restrict__ fout, const KParams p,
                                                       const FvParams fp, int seg) {
    using R = typename C::R;
    pdl_launch_dependents();
    pdl_wait();
    const int gx = (p.nx + 31) / 32, by = blockIdx.x / gx, x = (blockIdx.x - by * gx) * 32 + threadIdx.x;
    const int y0 = (by * blockDim.y + threadIdx.y) * seg, y1 = min(y0 + seg, p.ny);
    if (x >= p.nx || y0 >= p.ny) return;
    const int g = blockIdx.y / N1, i = blockIdx.y - g * N1;
    const bool single = 2 * g == N1 - 1;
    const int la = i + N1 * g, lb = single ? la : i + N1 * (N1 - 1 - g);
    Geom geo = geom_of(p);
    geo.walls = WALLS;
    FvGlobalSrc<C> src{f + sidx(p, la, x, 0), f + sidx(p, lb, x, 0), om + sidx(p, la, x, 0), om + sidx(p, lb, x, 0),
                       (long long)p.pitch, 0, !single};
    src.f0 = src.fE = src.fW = src.o0 = src.oE = src.oW = Pair<R>{R(0), R(0)};
    typename C::T *pa = fout + sidx(p, la, x, 0), *pb = fout + sidx(p, lb, x, 0);
    const int xw = x - (int)threadIdx.x;
    const bool inner = xw >= FILL && xw + 31 < p.nx - FILL;  // the whole warp
    const auto put = [&](int y, const Pair<R>(&out)[1]) {
        if (inner && (WALLS || (y >= FILL && y < p.ny - FILL))) {
            stg(pa + (long long)y * p.pitch, C::enc(out[0].x));
            if (!single) stg(pb + (long long)y * p.pitch, C::enc(out[0].y));
            return;
        }
        store_with_images(fout, geo, (long long)la * p.plane, x, y, C::enc(out[0].x));
        if (!single) store_with_images(fout, geo, (long long)lb * p.plane, x, y, C::enc(out[0].y));
    };
    fv_march<N1, 1, R, WALLS>(p, fp, y0, y1, [&](int) { return i; }, [&](int) { return g; }, src, put);
}

// ---- fused form ------------------------------------------------------------------------------------
// One kernel per step: a warp owns a strip of 30 output columns (lanes 0 and 31 hold the columns
// beside it; a row of 31 or 32 columns is periodic within its warp: 31 x 1000 D2Q16 8.4 us per step with
// two blocks of shared memory side by side, 13.5 with two strips here, 8.1 within the warp) and marches
// over a segment of rows: it loads a row's populations, computes the collision term of its 32 cells in
// registers, takes the east and west neighbours' values by warp
// shuffles and carries the row's contributions to the next rows (fv_march).  The collision term
// never leaves the registers: Q values read and Q written per cell update, 4 shuffles per velocity
// and cell where a block with both fields in shared memory read 18 values, 1.07 x (seg + 2) / seg
// collision terms per output cell.  D2Q16 at 1024 x 1024 with the Prandtl term: 50 us per step (91 us
// with a 32 x 16 block of both fields in shared memory, 1 873 instructions per cell, 35 us of it on
// the FP64 pipe converting double parameters); bound by the FP32 pipe and issue, 20 us of memory
// traffic underneath.
template <int N1, class C>
constexpr int fv_fused_minb() {  // resident CTAs: 16 warps per SM (D2Q36: 8, 250 registers); a fifth
    return 4;                     // for D2Q9 spills at 96 registers (41 against 39 us)
}
template <int N1>
constexpr int fv_fused_warps() {  // warps per CTA; two for D2Q36, whose rings are 14 KB each
    return N1 == 6 ? 2 : 4;
}
__device__ __forceinline__ Pair<float> shfl_e(Pair<float> v) {
    return {__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1)};
}
__device__ __forceinline__ Pair<float> shfl_w(Pair<float> v) {
    return {__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1)};
}
__device__ __forceinline__ Pair<float> shfl_from(Pair<float> v, int lane) {
    return {__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane)};
}

// Row source of the fused form: the lane's cell in registers, its neighbours by shuffles.  Rows come
// through a ring of three slots in shared memory that each lane fills for itself (asynchronous copies,
// no barrier: a lane reads only what it copied): the next row is in flight while this one is computed,
// which registers had no room for, and the row before it is still there when its output is completed,
// so its f_0 needs no registers either and D2Q16 fits four CTAs.  Against loads into registers at the
// head of each row, us per step at 1024 x 1024: D2Q9 44 -> 39, D2Q16 57.5 -> 50, D2Q36 134 -> 112; 64 x 61:
// 6.6 -> 6.0, 6.3 -> 6.4, 9.0 -> 10.1.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
template <int N1, class C, bool WHOLE>
struct FvStripSrc {
    using R = typename C::R;
    static constexpr bool kCarry = false;
    static constexpr int SLOT = N1 * N1 * 32;  // elements of a warp's row
    const typename C::T* f;  // the column's element of row 0 in plane 0
    const KParams& p;
    const FvParams& fp;
    R* ring;  // [3][Q][32], at this lane
    int east, west;  // WHOLE: the lanes that hold the columns beside this one
    int next, last, slot;  // the row whose copy is started next, the last one; the current row's slot
    Pair<R> s[fv_hp<N1>()][N1], o[fv_hp<N1>()][N1];
    __device__ __forceinline__ void start(int sl) {
        if (next <= last) {
            const typename C::T* b = f + (long long)next * p.pitch;
#pragma unroll
            for (int l = 0; l < N1 * N1; ++l) {
                cp_async4(ring + sl * SLOT + l * 32, b);
                b += p.plane;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++next;
    }
    __device__ __forceinline__ void begin(int first, int last_) {
        next = first;
        last = last_;
        slot = 2;
        start(0);
    }
    __device__ __forceinline__ Pair<R> at(const R* b, int q) const {
        const int i = q % N1, g = q / N1;
        return {b[(i + N1 * g) * 32], fv_single<N1>(g) ? R(0) : b[(i + N1 * (N1 - 1 - g)) * 32]};
    }
    __device__ __forceinline__ Pair<R> cur(int q) const { return s[q / N1][q % N1]; }
    __device__ __forceinline__ Pair<R> own(int q, int) const { return at(ring + (slot == 0 ? 2 : slot - 1) * SLOT, q); }
    __device__ __forceinline__ void row(int) {
        slot = slot == 2 ? 0 : slot + 1;
        start(slot == 2 ? 0 : slot + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        const R* b = ring + slot * SLOT;
#pragma unroll
        for (int g = 0; g < fv_hp<N1>(); ++g)
#pragma unroll
            for (int i = 0; i < N1; ++i) s[g][i] = at(b, g * N1 + i);
        fv_omega_cell<N1, R>(s, p, fp, o);
    }
    __device__ __forceinline__ void get(int q, Pair<R>& f0, Pair<R>& fE, Pair<R>& fW, Pair<R>& o0, Pair<R>& oE,
                                        Pair<R>& oW) const {
        f0 = s[q / N1][q % N1];
        o0 = o[q / N1][q % N1];
        fE = WHOLE ? shfl_from(f0, east) : shfl_e(f0);
        fW = WHOLE ? shfl_from(f0, west) : shfl_w(f0);
        oE = WHOLE ? shfl_from(o0, east) : shfl_e(o0);
        oW = WHOLE ? shfl_from(o0, west) : shfl_w(o0);
    }
};

// WHOLE: rows of 31 or 32 columns, the periodic row within the warp.
template <int N1, class C, bool WHOLE>
__global__ void __launch_bounds__(fv_fused_warps<N1>() * 32, fv_fused_minb<N1, C>())
    fv_fused_kernel(const typename C::T* __restrict__ f, typename C::T* __restrict__ fout, const KParams p,
                    const FvParams fp, int strips, int seg) {
    using R = typename C::R;
    constexpr int HP = fv_hp<N1>(), PN = HP * N1;
    pdl_launch_dependents();
    pdl_wait();
    const int w = blockIdx.x * fv_fused_warps<N1>() + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int strip = w % strips, y0 = (w / strips) * seg;
    if (y0 >= p.ny) return;  // whole warps
    const int y1 = min(y0 + seg, p.ny);
    const int x = WHOLE ? lane : strip * 30 + lane - 1;
    const int xl = min(x, p.nx);  // columns beyond the frame column nx belong to no output
    const bool mine = x < p.nx && (WHOLE || (lane >= 1 && lane <= 30));
    const int east = lane == p.nx - 1 ? 0 : min(lane + 1, 31), west = lane == 0 ? p.nx - 1 : lane - 1;
    const Geom geo = geom_of(p);
    using Src = FvStripSrc<N1, C, WHOLE>;
    __shared__ R ring[fv_fused_warps<N1>()][3 * Src::SLOT];
    Src src{f + sidx(p, 0, xl, 0), p, fp, &ring[threadIdx.x >> 5][lane], east, west};
    src.begin(fp.walls ? max(y0 - 1, 0) : y0 - 1, fp.walls ? min(y1, p.ny - 1) : y1);
    const auto put = [&](int y, const Pair<R>(&out)[PN]) {
        if (!mine) return;
        R s[N1 * N1];
#pragma unroll
        for (int g = 0; g < HP; ++g)
#pragma unroll
            for (int i = 0; i < N1; ++i) {
                s[i + N1 * g] = out[g * N1 + i].x;
                if (!fv_single<N1>(g)) s[i + N1 * (N1 - 1 - g)] = out[g * N1 + i].y;
            }
        store_collided<N1, C>(fout, geo, x, y, s);
    };
    fv_march<N1, PN, R, true>(p, fp, y0, y1, [](int q) { return q % N1; }, [](int q) { return q / N1; }, src, put);
}

// ---- wall imposition ---------------------------------------------------------------------------------
// Before a step: the leaving populations of every wall node (c . n > 0, n into the fluid)
// become A f_eq(u_eq, T_eq) with A = sum_{c.n<=0} |c.n| f / sum_{c.n>0} |c.n| f_eq (Eq.
// IMPOSITION); in the exact mode (u_eq, T_eq) follows the Newton-Raphson of App. B so that the
// node's velocity and temperature are the wall's.  One thread per (column, wall); FP64.
// A warp instruction of FP64 takes 64 cycles of its SM partition, so the iteration works on
// sums and not on populations: for the equilibrium f_eq_ij = w_i w_j sum_{a+b<=N} h_a(u) E_ia
// h_b(0) E_jb the sums over the leaving velocities follow from the quadrature along x (sum w E_a =
// [a=0], sum w x E_a = [a=1], sum w x^2 E_a = [a=0] + [a=2]) and three host tables along y (the odd
// h_b vanish at u_y = 0); their derivatives are exact, h_a' = a h_{a-1} in u and a (a - 1) / 2 h_{a-2}
// in T.  One iteration is then about 30 FP64 instructions and one division, where five equilibria
// with central differences took about 1 500 (64 columns, 6 iterations: 16 against 229 us).  One warp
// per block: the columns spread over the SMs.
// Velocity and temperature of the wall equilibrium of one wall node from the moments of the
// populations that stay (mass, x-momentum, energy, flux onto the wall); st: the node's warm start (the
// caller writes the result back).
template <int N1>
__device__ __forceinline__ void wall_equilibrium(const WallParams& wp, int side, const double* st, double in0, double inx,
                                                 double in2, double inc, double& ue, double& Te) {
    constexpr int N = N1 - 1;
    const double uw = wp.u[side], Tw = wp.T[side];
    ue = uw;
    Te = Tw;
    if (wp.exact) {
        ue = st[0];
        Te = st[1];
        const double g1 = uw * in0 - inx, cw = 2.0 * Tw + uw * uw, g2 = cw * in0 - in2;
        for (int it = 0; it < wp.iters; ++it) {
            const double th = Te - 1.0;
            // sums over b = 0, 2, 4 with h_0 = 1, h_2 = th, h_4 = 3 th^2, truncated at a + b <= N
            double S = fma(th, wp.kn[1], wp.kn[0]), s0 = fma(th, wp.k0[1], wp.k0[0]), q2 = fma(th, wp.k2[1], wp.k2[0]);
            double dS = wp.kn[1], ds0 = wp.k0[1], dq2 = wp.k2[1];
            if constexpr (N >= 4) {
                const double h4 = 3.0 * th * th, d4 = 6.0 * th;
                S = fma(h4, wp.kn[2], S);
                s0 = fma(h4, wp.k0[2], s0);
                q2 = fma(h4, wp.k2[2], q2);
                dS = fma(d4, wp.kn[2], dS);
                ds0 = fma(d4, wp.k0[2], ds0);
                dq2 = fma(d4, wp.k2[2], dq2);
            }
            // b <= N - 1 (with h_1(u)) and b <= N - 2 (with h_2(u))
            const double s1 = N == 2 ? wp.k0[0] : s0, ds1 = N == 2 ? 0.0 : ds0;
            const double sb = N <= 3 ? wp.k0[0] : fma(th, wp.k0[1], wp.k0[0]), dsb = N <= 3 ? 0.0 : wp.k0[1];
            const double h2 = fma(ue, ue, th);
            const double sx = ue * s1, s2 = fma(h2, sb, s0 + q2);
            // S-fold derivatives of the node's moments; S does not depend on u
            const double A = s1 * S, B = fma(ue * ds1, S, -(dS * sx));
            const double Cc = 2.0 * ue * sb * S, D = fma(fma(h2, dsb, sb + ds0 + dq2), S, -(dS * s2));
            const double F1 = fma(S, g1, inc * fma(uw, s0, -sx)), F2 = fma(S, g2, inc * fma(cw, s0, -s2));
            const double pref = S / (fma(A, D, -(B * Cc)) * inc);
            ue = fma(pref, fma(D, F1, -(B * F2)), ue);
            Te = fma(pref, fma(A, F2, -(Cc * F1)), Te);
        }
    }
}

// The leaving populations A f_eq(1, u_eq, T_eq) of a wall node, one y-node at a time.
template <int N1>
struct WallFactors {
    static constexpr int N = N1 - 1;
    double hx[N + 1], hy[N + 1], amp;
    __device__ __forceinline__ void set(const WallParams& wp, double ue, double Te, double inc) {
        const double th = Te - 1.0;
        hx[0] = hy[0] = 1.0;
        hx[1] = ue;
        hy[1] = 0.0;
#pragma unroll
        for (int n = 1; n < N; ++n) {
            hx[n + 1] = fma(ue, hx[n], n * th * hx[n - 1]);
            hy[n + 1] = (n & 1) ? n * th * hy[n - 1] : 0.0;
        }
        double S = 0.0;
#pragma unroll
        for (int b = 0; b <= N; b += 2) S = fma(hy[b], wp.kn[b / 2], S);
        amp = inc / S;
    }
    __device__ __forceinline__ void row(const KParams& p, int j, double (&v)[N1]) const {
        double G[N + 1], acc = 0.0;  // h_a sum_{b <= N - a} h_b E_jb
#pragma unroll
        for (int b = 0; b <= N; ++b) {
            if ((b & 1) == 0) acc = fma(hy[b], p.Ed[j][b], acc);
            G[N - b] = acc * hx[N - b];
        }
        const double wj = p.wd[j] * amp;
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            v[i] = G[0];
#pragma unroll
            for (int a = 1; a <= N; ++a) v[i] = fma(G[a], p.Ed[i][a], v[i]);
            v[i] *= p.wd[i] * wj;
        }
    }
};

template <int N1, class C>
__global__ void __launch_bounds__(32) fv_impose_kernel(typename C::T* __restrict__ f, const KParams p, const WallParams wp) {
    constexpr int N = N1 - 1, H = N1 / 2;
    pdl_launch_dependents();
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * p.nx) return;
    const int side = t / p.nx, x = t - side * p.nx;
    const int y = side == 0 ? 0 : p.ny - 1;
    // moments of the populations that stay: mass, x-momentum, energy, flux onto the wall
    double in0 = 0.0, inx = 0.0, in2 = 0.0, inc = 0.0;
#pragma unroll
    for (int jj = 0; jj < N1 - H; ++jj) {
        const int j = side == 0 ? jj : N1 - 1 - jj;  // c . n <= 0
        double r = 0.0, rx = 0.0, rxx = 0.0;
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            const double v = (double)C::ld(f + sidx(p, i + N1 * j, x, y));
            r += v;
            rx = fma(p.xd[i], v, rx);
            rxx = fma(p.x2d[i], v, rxx);
        }
        const double yj = p.xd[j];
        in0 += r;
        inx += rx;
        in2 += fma(p.x2d[j], r, rxx);
        inc = fma(fabs(yj), r, inc);
    }
    double ue, Te;
    double* st = wp.eq + (side * p.nx + x) * 2;
    wall_equilibrium<N1>(wp, side, st, in0, inx, in2, inc, ue, Te);
    if (wp.exact) {
        st[0] = ue;
        st[1] = Te;
    }
    WallFactors<N1> wf;
    wf.set(wp, ue, Te, inc);
    Geom g = geom_of(p);
    g.walls = 1;
#pragma unroll
    for (int jj = 0; jj < H; ++jj) {
        const int j = side == 0 ? N1 - 1 - jj : jj;  // c . n > 0
        double v[N1];
        wf.row(p, j, v);
#pragma unroll
        for (int i = 0; i < N1; ++i)
            store_with_images(f, g, (long long)(i + N1 * j) * p.plane, x, y, C::enc((typename C::R)v[i]));
    }
}

// ---- FP64 ------------------------------------------------------------------------------------------
// One warp instruction of FP64 takes 64 cycles of its SM partition whatever its active lanes, and the
// chip has 608 partitions: a 64 x 61 channel, one cell per lane, keeps 122 of them busy.  So on small
// grids four lanes share a cell of D2Q16, each with one y-node: the moments meet in two shuffle
// rounds, the shared scalars are computed by all four (about 95 FP64 instructions per warp instead
// of 215; 18.7 us against 16.1 + 10.4 us for the wall imposition and one lane per cell).  A wall row first
// imposes its leaving populations (as fv_impose_kernel), while the other rows' warps are already computing.
// The collision term is fv_omega_cell's with the sums in another order, so FP64 populations differ in
// their last bits between grids of up to 64 cells per SM and larger ones (one lane per cell there: D2Q9 and D2Q36
// on every grid).
__device__ __forceinline__ double quad_sum(double v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
__global__ void __launch_bounds__(32) fv_omega_lanes_kernel(double* __restrict__ f, double* __restrict__ om,
                                                            const KParams p, const FvParams fp, const WallParams wp) {
    constexpr int N1 = 4;
    pdl_launch_dependents();
    pdl_wait();
    const int gx = (p.nx + 7) / 8, y = blockIdx.x / gx, lane = threadIdx.x, j = lane & 3;
    const int x = (blockIdx.x - y * gx) * 8 + (lane >> 2), xl = min(x, p.nx - 1);
    const Geom geo = geom_of(p);
    const double xj = p.xd[j], xj2 = p.x2d[j];
    double v[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = f[sidx(p, i + N1 * j, xl, y)];
    const auto sums = [&](double& r, double& rx, double& rxx) {
        r = (v[0] + v[1]) + (v[2] + v[3]);
        rx = p.xd[0] * v[0];
        rxx = p.x2d[0] * v[0];
#pragma unroll
        for (int i = 1; i < N1; ++i) {
            rx = fma(p.xd[i], v[i], rx);
            rxx = fma(p.x2d[i], v[i], rxx);
        }
    };
    double r, rx, rxx;
    const int wall = fv_wall_of(p, fp, y);
    if (wall) {  // the whole warp
        const bool leaves = (wall == 1 ? xj : -xj) > 0.0;
        sums(r, rx, rxx);
        if (leaves) r = rx = rxx = 0.0;
        const double in0 = quad_sum(r), inx = quad_sum(rx), in2 = quad_sum(fma(xj2, r, rxx)), inc = quad_sum(fabs(xj) * r);
        double ue, Te;
        double* st = wp.eq + ((wall - 1) * p.nx + xl) * 2;
        wall_equilibrium<N1>(wp, wall - 1, st, in0, inx, in2, inc, ue, Te);
        __syncwarp();  // every lane has read the warm start
        if (wp.exact && j == 0 && x < p.nx) {
            st[0] = ue;
            st[1] = Te;
        }
        WallFactors<N1> wf;
        wf.set(wp, ue, Te, inc);
        double out[N1];
        wf.row(p, j, out);
        if (leaves) {
#pragma unroll
            for (int i = 0; i < N1; ++i) {
                v[i] = out[i];
                if (x < p.nx) store_with_images(f, geo, (long long)(i + N1 * j) * p.plane, x, y, out[i]);
            }
        }
        __syncwarp();
    }
    sums(r, rx, rxx);
    const double rho = quad_sum(r), jx = quad_sum(rx), jy = quad_sum(xj * r), eyy = quad_sum(xj2 * r), exx = quad_sum(rxx);
    const double inv = 1.0 / rho, ux = jx * inv, uy = jy * inv;
    const double T = 0.5 * fma(exx + eyy, inv, -fma(ux, ux, uy * uy)), th = T - 1.0;
    const double hx2 = fma(ux, ux, th), hy2 = fma(uy, uy, th), th2 = 2.0 * th;
    const double hx3 = fma(ux, hx2, th2 * ux), hy3 = fma(uy, hy2, th2 * uy);
    const double P1 = uy * p.Ed[j][1], P2 = fma(hy2, p.Ed[j][2], P1), P3 = fma(hy3, p.Ed[j][3], P2);
    const double ps = fp.pscale ? rho * T : 1.0, it = fp.d.it * ps;
    double qy = 0.0, axx = 0.0, cj = 0.0, b3 = 0.0, eyj = 0.0;
    if (fp.prandtl) {
        const double exy = quad_sum(xj * rx);
        const double pxx = 0.5 * fma(-rho, fma(ux, ux, -(uy * uy)), exx - eyy), pxy = fma(-rho, ux * uy, exy);
        const double sc = fp.d.itg * ps * inv / (T * T);
        axx = sc * pxx;
        const double axy = 2.0 * sc * pxy, dy = xj - uy;
        qy = fma(-axx, dy * dy, it);
        cj = axy * dy;
        const double h4x = fma(ux, hx3, 3.0 * th * hx2), h4y = fma(uy, hy3, 3.0 * th * hy2);
        const double m3 = -rho * fma(axx, h4x - h4y, axy * fma(hx3, uy, ux * hy3));
        b3 = fp.d.g33 * m3;
        eyj = fma(b3, xj2, fp.d.g03 * m3);
    }
    const double W = p.wd[j] * (fp.prandtl ? rho : rho * it);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
        const double X1 = ux * p.Ed[i][1], X2 = hx2 * p.Ed[i][2], SX = fma(hx3, p.Ed[i][3], (1.0 + X1) + X2);
        const double phi = fma(X1, P2, fma(X2, P1, SX + P3));
        const double eq = p.wd[i] * W * phi;
        double o;
        if (fp.prandtl) {
            const double dx = p.xd[i] - ux, q = fma(cj, dx, fma(axx, dx * dx, qy));
            o = fma(eq, q, fma(-it, v[i], -(p.wd[i] * p.wd[j]) * fma(b3, p.x2d[i], eyj)));
        } else {
            o = fma(-it, v[i], eq);
        }
        if (x < p.nx) store_with_images(om, geo, (long long)(i + N1 * j) * p.plane, x, y, o);
    }
}

// The update in FP64: one thread per cell and velocity, every load of its two 3 x 3 neighbourhoods in
// flight together, the stencils' coefficients paired over opposite neighbours (19 FP64 instructions;
// the row march spends 12 per row and row visited: 6.2 against 9.9 us on the 64 x 61 channel).
template <int N1>
__global__ void __launch_bounds__(32) fv_update64_kernel(const double* __restrict__ f, const double* __restrict__ om,
                                                         double* __restrict__ fout, const KParams p, const FvParams fp) {
    pdl_launch_dependents();
    pdl_wait();
    const int gx = (p.nx + 31) / 32, y = blockIdx.x / gx, x = (blockIdx.x - y * gx) * 32 + threadIdx.x;
    if (x >= p.nx) return;
    const int l = blockIdx.y, j = l / N1, i = l - j * N1, wall = fv_wall_of(p, fp, y);
    const double *a = f + sidx(p, l, x, y), *o = om + sidx(p, l, x, y);
    const double cxd = p.xd[i] * fp.d.dt16, k = p.xd[j] * fv_kfac<double>(fp, y, wall);
    double out;
    if (!wall) {
        const double *aN = a + p.pitch, *aS = a - p.pitch, *oN = o + p.pitch, *oS = o - p.pitch;
        const double f0 = __ldg(a), fE = __ldg(a + 1), fW = __ldg(a - 1), fN = __ldg(aN), fS = __ldg(aS);
        const double fNE = __ldg(aN + 1), fNW = __ldg(aN - 1), fSE = __ldg(aS + 1), fSW = __ldg(aS - 1);
        const double o0 = __ldg(o), oE = __ldg(o + 1), oW = __ldg(o - 1), o1 = __ldg(oN), o2 = __ldg(oS);
        const double oNE = __ldg(oN + 1), oNW = __ldg(oN - 1), oSE = __ldg(oS + 1), oSW = __ldg(oS - 1);
        const double d = fNE - fSW, q = fSE - fNW;
        const double gx16 = fma(6.0, fE - fW, d + q), gy16 = fma(6.0, fN - fS, d - q);
        const double ob = fma(36.0, o0, fma(6.0, (oE + oW) + (o1 + o2), (oNE + oSW) + (oNW + oSE)));
        out = f0 + fma(-cxd, gx16, fma(-k, gy16, ob));
    } else {
        const double sg = wall == 1 ? 1.0 : -1.0;
        out = __ldg(a);
        if (!(sg * p.xd[j] > 0.0)) {  // arriving: one-sided stencils into the fluid (Eq. FVLB2)
            const long long in = wall == 1 ? p.pitch : -(long long)p.pitch;
            const double *aI = a + in, *oI = o + in;
            const double fE = __ldg(a + 1), fW = __ldg(a - 1), fI = __ldg(aI), fIE = __ldg(aI + 1), fIW = __ldg(aI - 1);
            const double gx16 = fma(6.0, fE - fW, 2.0 * (fIE - fIW));
            const double gy16 = fma(6.0, fI - out, (fIE + fIW) - (fE + fW));
            const double oc = fma(6.0, __ldg(o), __ldg(o + 1) + __ldg(o - 1)), oi = fma(6.0, __ldg(oI), __ldg(oI + 1) + __ldg(oI - 1));
            out += fma(-cxd, gx16, fma(-sg * k, gy16, fma(6.0, oc, 2.0 * oi)));
        }
    }
    store_with_images(fout, geom_of(p), (long long)l * p.plane, x, y, out);
}

template <int N1, class C>
cudaError_t launch_fv(const void* f, void* om, void* fout, const KParams& p, const FvParams& fp, const WallParams& wp,
                      bool split, cudaStream_t s) {
    using T = typename C::T;
    cudaError_t e = cudaSuccess;
    const long long gx = (p.nx + 31) / 32;
    const int sms = sm_count();
    // FP64 runs the collision term and the update as two kernels in either form: its time is FP64
    // instructions, and the two kernels compute every collision term once (the march of the fused
    // form recomputes those of its ring)
    if constexpr (sizeof(typename C::R) == 8) {
        // (plain launches: the blocks of a kernel launched early are placed around those still resident
        // and share partitions -- the 64 x 61 channel took 37 us per step against 25 us)
        bool lanes = false;
        // four lanes per cell take 95 FP64 instructions where one lane takes 215, and fill the
        // chip's 4 x SMs partitions with a quarter of the cells
        if constexpr (N1 == 4) lanes = (long long)p.nx * p.ny <= 64LL * sms;
        if (lanes) {
            if constexpr (N1 == 4)
                e = launch_as(false, fv_omega_lanes_kernel, dim3((unsigned)((p.nx + 7) / 8 * p.ny)), dim3(32), 0, s, (T*)f,
                               (T*)om, p, fp, wp);
        } else {
            if (fp.walls) e = launch_as(false, fv_impose_kernel<N1, C>, dim3((2 * p.nx + 31) / 32), dim3(32), 0, s, (T*)f, p, wp);
            if (e != cudaSuccess) return e;
            e = launch_as(false, fv_omega_kernel<N1, C>, dim3((unsigned)(gx * p.ny)), dim3(32), 0, s, (const T*)f, (T*)om, p, fp);
        }
        if (e != cudaSuccess) return e;
        return launch_as(false, fv_update64_kernel<N1>, dim3((unsigned)(gx * p.ny), N1 * N1), dim3(32), 0, s, (const T*)f,
                          (const T*)om, (T*)fout, p, fp);
    } else {
        constexpr int W = fv_fused_warps<N1>();
        const long long warps = (long long)W * fv_fused_minb<N1, C>() * sms;  // resident warps of the fused form
        const int strips = p.nx <= 32 ? 1 : (p.nx + 29) / 30;
        if (fp.walls) {
            // The imposition is FP64: its blocks, launched early, are placed around those of the step before and share
            // SM partitions, so it overlaps where it has few blocks and that step leaves the chip room.  us per step
            // overlapping and not, fused: D2Q16 16 x 200 22.7 and 24.8, 256 x 200 24.4 and 27.0, 1000 x 100 27.0 and
            // 29.0, 500 x 500 32.2 and 33.5; D2Q9 500 x 1000 50 and 39; D2Q16 2000 x 30 31 and 27, 8192 x 32 106 and 35, 1024 x
            // 1024 139 and 69; D2Q36 256 x 200 37.6 and 39.3, 1000 x 30 37.0 and 39.2, 128 x 4000 103 and 95, 500 x 500 74 and
            // 58.  Two kernels, whose blocks are more: D2Q16 64 x 64 20.9 and 22.8, 64 x 4000 43.1 and 45.3, 128 x 16
            // 20.8 and 22.6, 100 x 200 24.6 and 24.0, 256 x 200 30.3 and 27.0, 500 x 16 33.1 and 22.9
            const int blocks = (2 * p.nx + 31) / 32;
            const bool room = 2 * blocks <= sms && (long long)blocks * strips * p.ny <= (N1 < 6 ? 300000 : 65000);
            const bool few = blocks <= 4 || (blocks <= 8 && p.ny <= 64);
            e = launch_as(split ? few : room, fv_impose_kernel<N1, C>, dim3(blocks), dim3(32), 0, s, (T*)f, p, wp);
        }
        if (e != cudaSuccess) return e;
        if (split) {
            // four warps to a block in both kernels: one-warp blocks are paced by their starts (1024 x 1024 D2Q9 without
            // the Prandtl term 92 us per step with them, 69 with four; 128 x 128 D2Q16 9.6 and 8.5)
            e = launch_pdl(fv_omega_kernel<N1, C>, dim3((unsigned)(gx * ((p.ny + 3) / 4))), dim3(32, 4), 0, s, (const T*)f,
                           (T*)om, p, fp);
            if (e != cudaSuccess) return e;
            // rows per thread: what gives 32 warps per SM, up to 6 (the rows above and below a
            // segment are taken again; D2Q9 FP32 per step, 8 rows always against this: 64 x 61 13.3 and 6.3 us,
            // 300 x 200 12.7 and 8.3; 512 x 512 17.0 with 8, 15.7 with 6, 17.5 with 2)
            const long long pairs = fv_hp<N1>() * N1;
            int seg = (int)((gx * p.ny * pairs + 32LL * sms - 1) / (32LL * sms));
            seg = seg < 1 ? 1 : (seg > 6 ? 6 : seg);
            const int segs = (p.ny + seg - 1) / seg;
            return launch_pdl(fp.walls ? fv_update_kernel<N1, C, true> : fv_update_kernel<N1, C, false>,
                              dim3((unsigned)(gx * ((segs + 3) / 4)), fv_hp<N1>() * N1),
                              dim3(32, 4), 0, s, (const T*)f, (const T*)om, (T*)fout, p, fp, seg);
        }
        // rows per warp: what fills the resident warps once, up to 32 (a small grid is bound by the latency
        // of the rows a warp visits and takes one row: 60 x 20 D2Q16 6.3 us against 12.1 with four)
        long long seg = ((long long)strips * p.ny + warps - 1) / warps;
        seg = seg < 1 ? 1 : (seg > 32 ? 32 : seg);
        const long long n = strips * ((p.ny + seg - 1) / seg);
        // (rows of up to 30 columns are one strip as they are, 5 % faster by the immediate shuffles)
        return launch_pdl(p.nx == 31 || p.nx == 32 ? fv_fused_kernel<N1, C, true> : fv_fused_kernel<N1, C, false>,
                          dim3((unsigned)((n + W - 1) / W)), dim3(W * 32), 0, s, (const T*)f,
                          (T*)fout, p, fp, strips, (int)seg);
    }
}

template <int N1>
cudaError_t launch_fv_storage(int storage, const void* f, void* om, void* fout, const KParams& p, const FvParams& fp,
                              const WallParams& wp, bool split, cudaStream_t s) {
    return storage == TVLBM_FP64 ? launch_fv<N1, CodecF64>(f, om, fout, p, fp, wp, split, s)
                                 : launch_fv<N1, CodecF32>(f, om, fout, p, fp, wp, split, s);
}

// Inverse of the 4 x 4 Gram matrix of (1, c_x, c_y, |c|^2) under the set's weights (Gauss-Jordan).
bool gram_inverse(const host::Rule& r, double out[4][4]) {
    double G[4][8];
    memset(G, 0, sizeof(G));
    for (int j = 0; j < r.n; ++j)
        for (int i = 0; i < r.n; ++i) {
            const double w = r.w[i] * r.w[j], cx = r.x[i], cy = r.x[j];
            const double phi[4] = {1.0, cx, cy, cx * cx + cy * cy};
            for (int a = 0; a < 4; ++a)
                for (int b = 0; b < 4; ++b) G[a][b] += w * phi[a] * phi[b];
        }
    for (int a = 0; a < 4; ++a) G[a][4 + a] = 1.0;
    for (int c = 0; c < 4; ++c) {
        int piv = c;
        for (int a = c + 1; a < 4; ++a)
            if (fabs(G[a][c]) > fabs(G[piv][c])) piv = a;
        if (fabs(G[piv][c]) < 1e-14) return false;
        for (int b = 0; b < 8; ++b) {
            const double t = G[c][b];
            G[c][b] = G[piv][b];
            G[piv][b] = t;
        }
        const double d = G[c][c];
        for (int b = 0; b < 8; ++b) G[c][b] /= d;
        for (int a = 0; a < 4; ++a)
            if (a != c) {
                const double m = G[a][c];
                for (int b = 0; b < 8; ++b) G[a][b] -= m * G[c][b];
            }
    }
    for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b) out[a][b] = G[a][4 + b];
    return true;
}

}  // namespace

int fvlb_steps(tvlbm_ctx* c, int n) {
    FvParams fp;
    memset(&fp, 0, sizeof(fp));
    double ginv[4][4];
    if (!gram_inverse(c->rule, ginv)) {
        snprintf(c->err, sizeof(c->err), "singular invariant Gram matrix");
        return TVLBM_EINVAL;
    }
    fp.prandtl = isfinite(c->tau_g) ? 1 : 0;
    fp.d.it = c->dt / 64.0 / c->tau;
    fp.d.itg = fp.prandtl ? c->dt / 64.0 / c->tau_g : 0.0;
    fp.d.dt16 = c->dt / 16.0;
    fp.d.g00 = ginv[0][0];
    fp.d.g03 = ginv[0][3];
    fp.d.g33 = ginv[3][3];
    fp.d.g11 = ginv[1][1];
    fp.d.g22 = ginv[2][2];
    fp.f = {(float)fp.d.it, (float)fp.d.itg, (float)fp.d.dt16, (float)fp.d.g00, (float)fp.d.g03,
            (float)fp.d.g33, (float)fp.d.g11, (float)fp.d.g22};
    fp.pscale = c->fv_pscale;
    fp.walls = c->kp.walls ? 1 : 0;
    fp.ysc = c->fv_ysc;
    WallParams wp;
    memset(&wp, 0, sizeof(wp));
    if (fp.walls) {
        if (!c->fv_wall_eq) {
            snprintf(c->err, sizeof(c->err), "channel: call tvlbm_set_fv_walls first");
            return TVLBM_EINVAL;
        }
        wp.u[0] = c->bc.u_lo;
        wp.T[0] = c->bc.T_lo;
        wp.u[1] = c->bc.u_hi;
        wp.T[1] = c->bc.T_hi;
        wp.exact = c->fv_exact;
        wp.iters = c->fv_nr_iters;
        wp.eq = c->fv_wall_eq;
        const host::Rule& r = c->rule;
        for (int j = 0; j < r.n; ++j)
            for (int b = 0; b < r.n && r.x[j] > 0.0; b += 2) {
                const double e = r.w[j] * host::hermite_over_fact(b, r.x[j]);
                wp.k0[b / 2] += e;
                wp.kn[b / 2] += e * r.x[j];
                wp.k2[b / 2] += e * r.x[j] * r.x[j];
            }
    }
    for (int t = 0; t < n; ++t) {
        void* f = c->mem + c->L.off_f[c->cur];
        void* fout = c->mem + c->L.off_f[1 - c->cur];
        cudaError_t e;
        switch (c->n1) {
            case 3: e = launch_fv_storage<3>(c->storage, f, c->fv_omega, fout, c->kp, fp, wp, c->fv_split != 0, c->stream); break;
            case 4: e = launch_fv_storage<4>(c->storage, f, c->fv_omega, fout, c->kp, fp, wp, c->fv_split != 0, c->stream); break;
            default: e = launch_fv_storage<6>(c->storage, f, c->fv_omega, fout, c->kp, fp, wp, c->fv_split != 0, c->stream); break;
        }
        if (e != cudaSuccess) {
            snprintf(c->err, sizeof(c->err), "finite-volume kernels: %s", cudaGetErrorString(e));
            return TVLBM_ECUDA;
        }
        c->cur ^= 1;
    }
    return TVLBM_OK;
}

extern "C" int tvlbm_set_scheme(tvlbm_ctx* c, int scheme, double tau_g) {
    if (!c) return TVLBM_EINVAL;
    if (scheme == TVLBM_SCHEME_VOLUMETRIC) {
        c->scheme = scheme;
        c->tau_g = INFINITY;
        return TVLBM_OK;
    }
    if (scheme != TVLBM_SCHEME_FVLB) {
        snprintf(c->err, sizeof(c->err), "unknown scheme %d", scheme);
        return TVLBM_EINVAL;
    }
    if (c->mesh_mem) {
        snprintf(c->err, sizeof(c->err), "the finite-volume scheme takes its mesh from tvlbm_set_fv_walls");
        return TVLBM_EINVAL;
    }
    if ((c->storage != TVLBM_FP64 && c->storage != TVLBM_FP32) || isnan(tau_g) || tau_g == 0.0 || !isfinite(c->tau)) {
        snprintf(c->err, sizeof(c->err), "the finite-volume scheme needs FP64 or FP32 storage, finite tau and tau_g != 0");
        return TVLBM_EINVAL;
    }
    cudaSetDevice(c->device);
    if (!c->fv_omega) {
        void* p = nullptr;
        if (cudaMalloc(&p, c->L.buf_bytes) != cudaSuccess) return TVLBM_ENOMEM;
        if (cudaMemset(p, 0, c->L.buf_bytes) != cudaSuccess) {
            cudaFree(p);
            return TVLBM_ECUDA;
        }
        c->fv_omega = p;
    }
    c->scheme = scheme;
    c->tau_g = tau_g;
    return TVLBM_OK;
}

extern "C" int tvlbm_set_fv_pressure_scaling(tvlbm_ctx* c, int enable) {
    if (!c) return TVLBM_EINVAL;
    if (c->scheme != TVLBM_SCHEME_FVLB) {
        snprintf(c->err, sizeof(c->err), "pressure scaling applies to the finite-volume scheme");
        return TVLBM_EINVAL;
    }
    c->fv_pscale = enable ? 1 : 0;
    return TVLBM_OK;
}

extern "C" int tvlbm_set_fv_fused(tvlbm_ctx* c, int fused) {
    if (!c) return TVLBM_EINVAL;
    c->fv_split = fused ? 0 : 1;
    return TVLBM_OK;
}

extern "C" int tvlbm_set_fv_walls(tvlbm_ctx* c, int exact, int nr_iters, const double* y_nodes) {
    if (!c) return TVLBM_EINVAL;
    if (!c->kp.walls || c->scheme != TVLBM_SCHEME_FVLB || (exact && nr_iters < 1) || nr_iters > 1000) {
        snprintf(c->err, sizeof(c->err), "needs a channel context in the finite-volume scheme and 1..1000 iterations");
        return TVLBM_EINVAL;
    }
    double* ysc = nullptr;  // the y factor of every row's stencil (see fv_march)
    if (y_nodes) {
        ysc = new double[c->ny];
        double below = 0.0;
        for (int j = 0; j < c->ny; ++j) {
            const double above = j + 1 < c->ny ? y_nodes[j + 1] - y_nodes[j] : below;
            if (!(above > 0.0) || !isfinite(above)) {
                delete[] ysc;
                snprintf(c->err, sizeof(c->err), "y_nodes must be finite and increasing");
                return TVLBM_EINVAL;
            }
            ysc[j] = 2.0 / (j == 0 || j + 1 == c->ny ? above : above + below);
            below = above;
        }
    }
    cudaSetDevice(c->device);
    if (!c->fv_wall_eq && cudaMalloc((void**)&c->fv_wall_eq, sizeof(double) * 4 * c->nx) != cudaSuccess) {
        delete[] ysc;
        return TVLBM_ENOMEM;
    }
    // warm start of the Newton-Raphson: the walls' own velocity and temperature
    double* eq = new double[4 * c->nx];
    for (int x = 0; x < c->nx; ++x) {
        eq[2 * x] = c->bc.u_lo;
        eq[2 * x + 1] = c->bc.T_lo;
        eq[2 * (c->nx + x)] = c->bc.u_hi;
        eq[2 * (c->nx + x) + 1] = c->bc.T_hi;
    }
    cudaError_t e = cudaMemcpy(c->fv_wall_eq, eq, sizeof(double) * 4 * c->nx, cudaMemcpyHostToDevice);
    delete[] eq;
    if (e == cudaSuccess && ysc) {
        if (!c->fv_ysc) e = cudaMalloc((void**)&c->fv_ysc, sizeof(double) * c->ny);
        if (e == cudaSuccess) e = cudaMemcpy(c->fv_ysc, ysc, sizeof(double) * c->ny, cudaMemcpyHostToDevice);
    } else if (e == cudaSuccess && c->fv_ysc) {
        cudaFree(c->fv_ysc);
        c->fv_ysc = nullptr;
    }
    delete[] ysc;
    if (e != cudaSuccess) {
        snprintf(c->err, sizeof(c->err), "CUDA: %s", cudaGetErrorString(e));
        return TVLBM_ECUDA;
    }
    c->fv_exact = exact ? 1 : 0;
    c->fv_nr_iters = exact ? nr_iters : 0;
    return TVLBM_OK;
}
