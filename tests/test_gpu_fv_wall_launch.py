"""Finite-volume channels on both sides of the lines where the wall imposition is launched early: the fused
and the two-kernel form, which draw them differently, give the same populations bit for bit."""
import numpy as np
import pytest

from test_gpu_fv_forms import make, tv  # noqa: F401


# two kernels: 4 and 5 blocks of 16 columns, 8 of them up to and beyond 64 rows; fused: 76 and 77 blocks, and
# blocks x strips of 30 columns x rows up to 300 000 (D2Q36: 65 000)
@pytest.mark.gpu
@pytest.mark.parametrize("velset,nx,ny", [
    ("D2Q9", 64, 70), ("D2Q9", 65, 70), ("D2Q16", 128, 64), ("D2Q16", 128, 65), ("D2Q16", 129, 16), ("D2Q16", 1216, 20),
    ("D2Q16", 1217, 20), ("D2Q9", 1200, 100), ("D2Q9", 1200, 101), ("D2Q36", 256, 451), ("D2Q36", 256, 452)])
def test_both_sides_of_the_wall_lines(tv, velset, nx, ny):  # noqa: F811
    out = []
    for fused in (True, False):
        sim = make(tv, nx, ny, velset, "fp32", True, 2.0, fused=fused)
        sim.step(5)
        out.append(sim.populations_f64())
        sim.close()
    assert np.all(np.isfinite(out[0]))
    assert np.array_equal(out[0], out[1])
