"""The mesh sweep's FP32 instantiations (mirror velocities in packed pairs) against the FP64 oracle: every
set, list lengths of 2 to 4 and the general loop, columns at the edges of its 31-column warps; and
domains taller than the grid's y extent."""
import numpy as np
import pytest

import workloads
from oracle.mesh import MeshOracle
from test_gpu_mesh import WALLS, _pattern, pair, tv  # noqa: F401
from workloads import random_faces, tanh_faces

pytestmark = pytest.mark.gpu

MESHES = {2: random_faces(21, 4, 0.9, 1.1), 3: random_faces(21, 4), 4: _pattern([2.0, 0.5, 0.5, 0.5], 21),
          8: _pattern([3.0, 0.25, 0.25, 0.25, 0.25, 0.25, 0.25], 21)}


# A step rounds the stored value (relative 6e-8) and, in the gather, the collision and the walls' sums, about
# as much again for each of a velocity's two interpolations and its relaxation: 4 x 6e-8 per step, of the
# largest stored value of its kind (raw populations: of the velocity's largest population; deviations: of the
# deviations' largest, which the rest value multiplies back).  Ten steps.
@pytest.mark.parametrize("velset", ["D2Q9", "D2Q16", "D2Q36"])
@pytest.mark.parametrize("storage", ["fp32", "fp32_dev"])
@pytest.mark.parametrize("entries", [2, 3, 4, 8])
@pytest.mark.parametrize("walls", [None, WALLS])
def test_fp32_matches_oracle(tv, velset, storage, entries, walls):  # noqa: F811
    for nx in (1, 30, 31, 32, 62, 63) if entries == 3 else (29,):
        sim, ref = pair(tv, nx, MESHES[entries], velset, storage, walls)
        sim.step(10)
        ref.step(10)
        got = sim.populations_f64()
        err = np.max(np.abs(got - ref.f), axis=(1, 2)) / np.max(np.abs(ref.f), axis=(1, 2))
        assert np.max(err) <= 10 * 4 * 6e-8, (nx, err)
        sim.close()


# Rows repeat with a period, so a tall domain repeats a short one.  Its faces lie at larger numbers, whose
# last bit (270 000 x 1.1e-16) may move a weight by 6e-11: far below the FP32 weights' own rounding,
# which it can flip (6e-8 of a value per interpolation, four steps).
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp32_dev"])
@pytest.mark.parametrize("heights", [[1.0, 0.75, 1.25, 1.0], [2.0, 0.5, 0.5, 0.5]])
def test_taller_than_the_grid(tv, storage, heights):  # noqa: F811
    out = []
    for ny in (9000, 270000):
        sim = tv.Simulation(2, ny, "D2Q9", tau=0.8, dt=0.5, storage=storage)
        sim.set_y_faces(_pattern(heights, ny))
        y = np.arange(ny) % 9000 / 9000.0
        f = [np.repeat(a[:, None], 2, axis=1) for a in (1 + 0.02 * np.sin(2 * np.pi * y), 0.03 * np.cos(2 * np.pi * y),
                                                        0.02 * np.sin(4 * np.pi * y), 1 + 0.02 * np.cos(2 * np.pi * y))]
        sim.init_moments(*f)
        sim.step(4)
        out.append(sim.populations_f64())
        sim.close()
    tol = 4 * 4 * 6e-8 if storage != "fp64" else 1e-9
    for k in range(30):
        part = out[1][:, 9000 * k:9000 * (k + 1)]
        assert np.max(np.abs(part - out[0])) <= tol * np.max(np.abs(out[0])), k


# widths at which 32 columns to a warp, each lane combining both of its columns, take the place of 31
@pytest.mark.parametrize("velset,storage,tol", [("D2Q9", "fp64", 1e-12), ("D2Q16", "fp64", 1e-12), ("D2Q36", "fp64", 1e-12),
                                                ("D2Q9", "fp32", 10 * 4 * 6e-8), ("D2Q9", "fp32_dev", 10 * 4 * 6e-8)])
@pytest.mark.parametrize("entries", [2, 3, 4, 8])
def test_both_columns_by_one_lane(tv, velset, storage, tol, entries):  # noqa: F811
    for nx in (31, 32, 33, 64, 65, 96):
        sim, ref = pair(tv, nx, MESHES[entries], velset, storage, WALLS if nx % 2 else None)
        sim.step(10)
        ref.step(10)
        got = sim.populations_f64()
        err = np.max(np.abs(got - ref.f), axis=(1, 2)) / np.max(np.abs(ref.f), axis=(1, 2))
        assert np.max(err) <= tol, (nx, err)
        sim.close()
