"""The finite-volume kernels at the edges of their work split, against the FP64 oracle and
against each other: strips of 30 columns and row segments of the fused form (FP32), channels with
wall nodes in it, four lanes or one lane per cell (FP64, on either side of 64 cells per SM)."""
import numpy as np
import pytest

from math import factorial

from oracle import fvlb

pytestmark = pytest.mark.gpu

WALLS = (0.02, 1.0, -0.03, 1.05)


@pytest.fixture(scope="module")
def tv():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1004_5059_gb300 as tv
    return tv


def fields(nx, ny):
    yy = np.linspace(0, 1, ny).reshape(-1, 1) * np.ones((1, nx))
    xx = np.linspace(0, 1, nx, endpoint=False).reshape(1, -1) * np.ones((ny, 1))
    return (1.0 + 0.01 * np.cos(2 * np.pi * xx) * yy, 0.03 * np.sin(3 * yy) + 0.01 * np.sin(2 * np.pi * xx),
            0.005 * np.sin(np.pi * yy) * np.cos(2 * np.pi * xx), 1.0 + 0.02 * yy)


class ExactDerivatives(fvlb.FVLBChannel):
    """The oracle's channel with the wall equilibrium's derivatives in closed form (h_a' = a h_{a-1}
    in u, a (a - 1) / 2 h_{a-2} in T) instead of its central differences, whose own error on D2Q36
    reaches 5e-13 of a population."""

    def impose(self):
        cx, cy, w, N = self.vs["cx"], self.vs["cy"], self.vs["w"], self.vs["n"] - 1

        def hermite(x, th):  # h_n(x): x h_{n-1} + (n-1) th h_{n-2}
            h = [np.ones_like(x), x]
            for k in range(1, N):
                h.append(x * h[k] + k * th * h[k - 1])
            return h
        E, F = hermite(cx, -1.0), hermite(cy, -1.0)
        K = [(a, b, w * E[a] * F[b] / (factorial(a) * factorial(b))) for a in range(N + 1) for b in range(N + 1 - a)]
        c2 = cx * cx + cy * cy
        for side, j in ((0, 0), (1, self.ny - 1)):
            cn = cy if side == 0 else -cy
            out = cn > 0
            uw, Tw = self.walls[2 * side], self.walls[2 * side + 1]
            for x in range(self.nx):
                f = self.f[:, j, x]
                inc = np.sum(np.abs(cn[~out]) * f[~out])
                ue, Te = self.wall_eq[side][x] if self.exact else (uw, Tw)
                for it in range(self.nr_iters + 1):
                    hx, hy = hermite(np.float64(ue), Te - 1.0), hermite(np.float64(0.0), Te - 1.0)
                    feq = sum(k * hx[a] * hy[b] for a, b, k in K)
                    S = np.sum(cn[out] * feq[out])
                    f[out] = inc / S * feq[out]
                    if it == self.nr_iters or not self.exact:
                        break
                    du = sum(k * a * hx[a - 1] * hy[b] for a, b, k in K if a)
                    dT = sum(k * (a * (a - 1) / 2 * hx[a - 2] * hy[b] if a > 1 else 0.0) for a, b, k in K) + sum(
                        k * (b * (b - 1) / 2 * hx[a] * hy[b - 2] if b > 1 else 0.0) for a, b, k in K)
                    rho = f.sum()
                    F1 = rho * uw - np.sum(f * cx)
                    F2 = 2.0 * rho * Tw + rho * uw * uw - np.sum(f * c2)
                    coef = [np.sum(g[out] * d[out]) - np.sum(cn[out] * d[out]) * np.sum(g[out] * feq[out]) / S
                            for g, d in ((cx, du), (cx, dT), (c2, du), (c2, dT))]
                    A, B, C, D = coef
                    pref = S / ((A * D - B * C) * inc)
                    ue += pref * (D * F1 - B * F2)
                    Te += pref * (A * F2 - C * F1)
                if self.exact:
                    self.wall_eq[side][x] = [ue, Te]


def make(tv, nx, ny, velset, storage, walls, tau_g, fused=True, exact=True, y=None, pscale=False):
    sim = tv.Simulation(nx, ny, velset, tau=0.5, dt=0.01, walls=WALLS if walls else None, storage=storage)
    sim.set_scheme("fvlb", tau_g)
    if walls:
        sim.set_fv_walls(exact=exact, nr_iters=12, y_nodes=y)
    sim.set_fv_pressure_scaling(pscale)
    sim.set_fv_fused(fused)
    sim.init_moments(*fields(nx, ny))
    return sim


@pytest.mark.parametrize("velset", ["D2Q9", "D2Q16", "D2Q36"])
@pytest.mark.parametrize("nx,ny,walls", [(1, 9, True), (30, 13, True), (31, 40, True), (61, 133, True), (1, 3, False),
                                         (30, 4, False), (91, 70, False)])
def test_fp32_fused_equals_two_kernels(tv, velset, nx, ny, walls):
    y = fvlb.tanh_nodes(ny, ny / 2.0, 1.5) if walls and ny != 40 else None
    out = []
    for fused in (True, False):
        sim = make(tv, nx, ny, velset, "fp32", walls, 2.0, fused=fused, y=y, pscale=nx == 61)
        sim.step(9)
        out.append(sim.populations_f64())
        sim.close()
    assert np.all(np.isfinite(out[0]))
    assert np.array_equal(out[0], out[1])


# FP32: the populations are rounded once per step (relative 6e-8, and as much again for the
# increments' own rounding): 9 steps stay within 9 x 2 x 6e-8 = 1.1e-6 of the oracle, relative to
# each velocity's largest population.  FP64: the same count with 1.1e-16, with a factor 100 for the
# wall iteration's division of small differences (against exact derivatives).
@pytest.mark.parametrize("storage,tol", [("fp32", 1.1e-6), ("fp64", 2e-13)])
@pytest.mark.parametrize("velset,tau_g", [("D2Q9", np.inf), ("D2Q16", 2.0), ("D2Q16", np.inf), ("D2Q36", -1.0)])
@pytest.mark.parametrize("nx,ny,walls,exact", [(31, 13, True, True), (29, 11, True, False), (33, 37, False, False)])
def test_matches_oracle(tv, storage, tol, velset, tau_g, nx, ny, walls, exact):
    if velset != "D2Q16" and np.isfinite(tau_g):
        tau_g = np.inf  # the oracle's Prandtl term is defined on the D2Q16 basis
    y = fvlb.tanh_nodes(ny, 6.0, 1.2)
    sim = make(tv, nx, ny, velset, storage, walls, tau_g, exact=exact, y=y if walls else None)
    if walls:
        ref = ExactDerivatives(nx, ny, y, WALLS, velset, tau=0.5, tau_g=tau_g, dt=0.01, exact=exact, nr_iters=12)
    else:
        ref = fvlb.FVLB(nx, ny, velset, tau=0.5, tau_g=tau_g, dt=0.01)
    ref.init_moments(*fields(nx, ny))
    sim.step(9)
    ref.step(9)
    err = np.max(np.abs(sim.populations_f64() - ref.f), axis=(1, 2)) / np.max(np.abs(ref.f), axis=(1, 2))
    assert np.max(err) <= tol, err
    sim.close()


@pytest.mark.parametrize("nx,ny", [(64, 152), (64, 153), (130, 75)])
def test_fp64_lane_split_matches_oracle(tv, nx, ny):
    """9 728 cells (four lanes per cell on 152 SMs) and just above (one lane per cell)."""
    sim = make(tv, nx, ny, "D2Q16", "fp64", False, 2.0)
    ref = fvlb.FVLB(nx, ny, "D2Q16", tau=0.5, tau_g=2.0, dt=0.01)
    ref.init_moments(*fields(nx, ny))
    sim.step(3)
    ref.step(3)
    assert np.max(np.abs(sim.populations_f64() - ref.f)) <= 2e-13 * np.max(np.abs(ref.f))
    sim.close()
