"""Finite-volume rows of a few columns (of 31 and 32: the periodic row within a warp) and the blocks of the two-kernel
form: the fused and the two-kernel form give the same populations bit for bit, and those of the oracle."""
import numpy as np
import pytest

from oracle import fvlb
from test_gpu_fv_forms import fields, make, tv  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("velset", ["D2Q9", "D2Q16", "D2Q36"])
@pytest.mark.parametrize("nx,ny,walls", [(1, 5, False), (2, 13, True), (29, 9, False), (31, 7, False), (32, 40, True),
                                         (32, 133, False), (33, 21, False), (97, 611, False), (40, 1300, True)])
def test_fused_equals_two_kernels(tv, velset, nx, ny, walls):  # noqa: F811
    out = []
    for fused in (True, False):
        sim = make(tv, nx, ny, velset, "fp32", walls, 2.0, fused=fused)
        sim.step(5)
        out.append(sim.populations_f64())
        sim.close()
    assert np.all(np.isfinite(out[0]))
    assert np.array_equal(out[0], out[1])


# 6e-8 for the step's rounding of a population and as much for its increment's, five steps
@pytest.mark.parametrize("nx", [1, 2, 31, 32, 33])
@pytest.mark.parametrize("fused", [True, False])
def test_narrow_rows_match_oracle(tv, nx, fused):  # noqa: F811
    ny = 23
    sim = make(tv, nx, ny, "D2Q16", "fp32", False, 2.0, fused=fused)
    ref = fvlb.FVLB(nx, ny, "D2Q16", tau=0.5, tau_g=2.0, dt=0.01)
    ref.init_moments(*fields(nx, ny))
    sim.step(5)
    ref.step(5)
    err = np.max(np.abs(sim.populations_f64() - ref.f), axis=(1, 2)) / np.max(np.abs(ref.f), axis=(1, 2))
    assert np.max(err) <= 5 * 2 * 6e-8, err
    sim.close()
