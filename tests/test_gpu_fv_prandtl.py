"""The finite-volume scheme's Prandtl term in its closed form, for every velocity set, against the oracle
with the term's components along the collision invariants removed by their Gram matrix (on D2Q16 that is
the oracle's own projection): periodic and channel, FP32 fused and in two kernels, FP64."""
import numpy as np
import pytest

from oracle import fvlb
from test_gpu_fv_forms import WALLS, ExactDerivatives, fields, make, tv  # noqa: F401


class Gram:
    def prandtl_term(self, f, feq):
        cx, cy, w = (self.vs[k].reshape(-1, 1, 1) for k in ("cx", "cy", "w"))
        rho, ux, uy, T = self._eq.moments(f)
        dx, dy = cx - ux, cy - uy
        neq = f - feq
        pxx, pxy, pyy = ((neq * a).sum(axis=0) for a in (dx * dx, dx * dy, dy * dy))
        raw = feq / (rho * T * T) * (pxx * dx * dx + 2.0 * pxy * dx * dy + pyy * dy * dy) / self.tau_g
        phi = np.stack([np.ones_like(cx), cx, cy, cx * cx + cy * cy])[..., 0, 0]
        G = np.einsum("l,al,bl->ab", self.vs["w"], phi, phi)
        b = np.einsum("ab,bl,lyx->ayx", np.linalg.inv(G), phi, raw)
        return raw - w * np.einsum("al,ayx->lyx", phi, b)


class Periodic(Gram, fvlb.FVLB):
    pass


class Channel(Gram, ExactDerivatives):
    pass


def test_the_reference_is_the_oracles_on_d2q16():
    nx, ny = 9, 7
    a, b = Periodic(nx, ny, "D2Q16", tau_g=2.0), fvlb.FVLB(nx, ny, "D2Q16", tau_g=2.0)
    for o in (a, b):
        o.init_moments(*fields(nx, ny))
        o.step(3)
    assert np.max(np.abs(a.f - b.f)) <= 1e-15


# FP32: 9 steps, each rounding a population (relative 6e-8) and its increment (as much again).  FP64: the
# same count with 1.1e-16 and a factor 100 for the differences of nearly equal moments (and, in the channel,
# for the wall iteration's).
@pytest.mark.gpu
@pytest.mark.parametrize("storage,fused,tol", [("fp32", True, 1.1e-6), ("fp32", False, 1.1e-6), ("fp64", True, 2e-13)])
@pytest.mark.parametrize("velset", ["D2Q9", "D2Q16", "D2Q36"])
@pytest.mark.parametrize("nx,ny,walls,tau_g,pscale", [(33, 37, False, 2.0, False), (33, 37, False, -1.0, True),
                                                      (31, 13, True, 2.0, True), (130, 77, False, 1.5, False)])
def test_matches_oracle(tv, storage, fused, tol, velset, nx, ny, walls, tau_g, pscale):  # noqa: F811
    y = fvlb.tanh_nodes(ny, 6.0, 1.2)
    sim = make(tv, nx, ny, velset, storage, walls, tau_g, fused=fused, y=y if walls else None, pscale=pscale)
    if walls:
        ref = Channel(nx, ny, y, WALLS, velset, tau=0.5, tau_g=tau_g, dt=0.01, exact=True, nr_iters=12, pressure_scaled=pscale)
    else:
        ref = Periodic(nx, ny, velset, tau=0.5, tau_g=tau_g, dt=0.01, pressure_scaled=pscale)
    ref.init_moments(*fields(nx, ny))
    sim.step(9)
    ref.step(9)
    err = np.max(np.abs(sim.populations_f64() - ref.f), axis=(1, 2)) / np.max(np.abs(ref.f), axis=(1, 2))
    assert np.max(err) <= tol, err
    sim.close()
