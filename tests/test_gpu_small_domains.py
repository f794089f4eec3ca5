"""Domains that the tiled form runs without tiles (one cell per thread, or lanes sharing an FP64 cell)
against the strip form and against tiles: the same populations bit for bit, on both sides of the
lines between the kernels, ragged against their blocks, periodic and with walls, with and without a
per-row reference."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

WALLS = (0.02, 1.0, -0.03, 1.05)


@pytest.fixture(scope="module")
def tv():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1004_5059_gb300 as tv
    return tv


def run(tv, nx, ny, velset, storage, form, walls, rows, steps, graphs=True):
    sim = tv.Simulation(nx, ny, velset, tau=0.8, walls=walls, storage=storage, form=form, graphs=graphs)
    if rows:
        sim.set_reference_rows(0.0, 0.0, np.linspace(1.0, 1.05, ny))
    sim.init_moments(*workloads.random_smooth(nx, ny, seed=nx + ny, amp_u=0.04, amp_T=0.03))
    sim.step(steps)
    out = sim.raw_populations()
    sim.close()
    return out.view(np.uint16) if storage == "bf16_dev" else out


@pytest.mark.parametrize("velset", ["D2Q9", "D2Q16", "D2Q36"])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp32_dev", "fp16_dev", "bf16_dev"])
@pytest.mark.parametrize("nx,ny,walls", [(1, 1, None), (3, 5, None), (33, 9, WALLS), (65, 37, None), (130, 41, WALLS)])
def test_tiled_equals_strip_on_small_domains(tv, velset, storage, nx, ny, walls):
    a = run(tv, nx, ny, velset, storage, "tiled", walls, False, 35)
    b = run(tv, nx, ny, velset, storage, "strip", walls, False, 35, graphs=False)
    assert np.all(np.isfinite(a.astype(np.float64)))
    assert np.array_equal(a, b)
    if walls and storage.endswith("_dev"):
        a = run(tv, nx, ny, velset, storage, "tiled", walls, True, 35)
        b = run(tv, nx, ny, velset, storage, "strip", walls, True, 35)
        assert np.array_equal(a, b)


# either side of: 64 and 600 FP64 cells per SM (152 SMs); 12 M populations in 4-byte storage, 8 M in 2-byte
@pytest.mark.parametrize("velset,storage,nx,ny", [
    ("D2Q16", "fp64", 128, 76), ("D2Q16", "fp64", 128, 77), ("D2Q36", "fp64", 64, 76), ("D2Q36", "fp64", 64, 77),
    ("D2Q9", "fp64", 304, 300), ("D2Q9", "fp64", 304, 301), ("D2Q16", "fp32", 1000, 750), ("D2Q16", "fp32_dev", 1000, 751),
    ("D2Q36", "fp16_dev", 500, 444), ("D2Q36", "bf16_dev", 500, 445), ("D2Q9", "fp32", 1, 70000)])
def test_lines_between_the_kernels(tv, velset, storage, nx, ny):
    a = run(tv, nx, ny, velset, storage, "tiled", None, False, 4)
    b = run(tv, nx, ny, velset, storage, "strip", None, False, 4)
    assert np.array_equal(a, b)


# the 31 columns that a warp of the shuffled gather takes
@pytest.mark.parametrize("velset,storage,rows", [("D2Q16", "fp32", False), ("D2Q16", "fp16_dev", True),
                                                 ("D2Q36", "fp32_dev", True), ("D2Q36", "bf16_dev", False)])
@pytest.mark.parametrize("nx", [30, 31, 32, 61, 62, 63, 94])
def test_columns_of_the_shuffled_gather(tv, velset, storage, rows, nx):
    ny = (250000 if velset == "D2Q16" else 64000) // nx + 1  # the smallest that takes it
    a = run(tv, nx, ny, velset, storage, "plain", WALLS, rows, 6)
    b = run(tv, nx, ny, velset, storage, "strip", WALLS, rows, 6)
    assert np.all(np.isfinite(a.astype(np.float64)))
    assert np.array_equal(a, b)


# either side of: 15 M populations (30 M: D2Q36 in 2-byte storage) for the tiled form; 250 000 and 64 000
# cells, both buffers of 125 MB for the shuffled gather
@pytest.mark.parametrize("velset,storage,nx,ny,form", [
    ("D2Q16", "fp32", 1000, 937, "tiled"), ("D2Q16", "fp32", 1000, 938, "tiled"), ("D2Q16", "fp16_dev", 1000, 937, "tiled"),
    ("D2Q16", "fp16_dev", 1000, 938, "tiled"), ("D2Q36", "fp16_dev", 1000, 833, "tiled"), ("D2Q36", "fp16_dev", 1000, 834, "tiled"),
    ("D2Q16", "fp32_dev", 1000, 976, "plain"), ("D2Q16", "fp32_dev", 1000, 977, "plain"),
    ("D2Q16", "bf16_dev", 500, 499, "plain"), ("D2Q16", "bf16_dev", 500, 500, "tiled"), ("D2Q36", "fp32", 256, 249, "tiled"),
    ("D2Q36", "fp32", 256, 250, "tiled")])
def test_lines_of_the_shuffled_gather(tv, velset, storage, nx, ny, form):
    a = run(tv, nx, ny, velset, storage, form, None, False, 4)
    b = run(tv, nx, ny, velset, storage, "strip", None, False, 4)
    assert np.array_equal(a, b)
