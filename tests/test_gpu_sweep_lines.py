"""The lines between the untiled, shuffled and tiled sweeps on narrow, tall and ragged domains: on both
sides of each the same populations as the strip form, bit for bit; and, without a GPU, where the
tiled form runs tiles."""
import numpy as np
import pytest

import workloads

WALLS = (0.02, 1.0, -0.03, 1.05)


@pytest.fixture(scope="module")
def tv():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1004_5059_gb300 as tv
    return tv


def run(tv, nx, ny, velset, storage, form, walls, rows, steps=4):
    sim = tv.Simulation(nx, ny, velset, tau=0.8, walls=walls, storage=storage, form=form)
    if rows:
        sim.set_reference_rows(0.0, 0.0, np.linspace(1.0, 1.05, ny))
    sim.init_moments(*workloads.random_smooth(nx, ny, seed=nx + ny, amp_u=0.04, amp_T=0.03))
    sim.step(steps)
    out = sim.raw_populations()
    sim.close()
    return out.view(np.uint16) if storage == "bf16_dev" else out


# sizes around the lines: 8000, 4000 and 2000 warps of 31 columns; 31 columns to a warp against 32 (one warp in
# eight, one in three more); 16 and 8 columns; both buffers of 200, 130, 100 and 97 MB; 15.6, 9, 32, 19, 10, 8 and 7 M
# populations, or those that whole warps cover; blocks of eight rows from 0.4 to 1, from 1.5 to 4 per SM
@pytest.mark.gpu
@pytest.mark.parametrize("velset,storage,sizes", [
    ("D2Q16", "fp32", [(1, 3999), (1, 4000), (31, 4001), (32, 4001), (64, 2100), (224, 600), (256, 500), (32, 12000)]),
    ("D2Q16", "fp16_dev", [(16, 30000), (16, 31000), (8, 40000), (9, 40000), (32, 15600), (32, 15700), (96, 1500)]),
    ("D2Q36", "fp32_dev", [(64, 500), (64, 640), (30, 1999), (30, 2000), (62, 3000), (64, 3000), (64, 3100), (17, 17000)]),
    ("D2Q36", "bf16_dev", [(96, 700), (128, 2000), (128, 4200), (64, 2500), (33, 5000), (64, 7500), (32, 14000)]),
    ("D2Q16", "fp16_dev", [(1, 7999), (8, 8000), (9, 4000)]), ("D2Q36", "fp32", [(40, 8192), (31, 8192), (30, 243), (30, 249)]),
    ("D2Q9", "fp32", [(64, 900), (64, 920), (200, 150), (300, 200), (64, 2432), (64, 2433), (1, 50000), (32, 54000)]),
    ("D2Q9", "fp16_dev", [(16, 31000), (16, 32000), (1000, 970), (1000, 980)])])
def test_both_sides_of_the_lines(tv, velset, storage, sizes):
    for k, (nx, ny) in enumerate(sizes):
        walls = WALLS if k % 2 else None
        rows = bool(walls) and storage.endswith("_dev")
        want = run(tv, nx, ny, velset, storage, "strip", walls, rows)
        assert np.all(np.isfinite(want.astype(np.float64)))
        for form in ("tiled", "plain"):
            assert np.array_equal(run(tv, nx, ny, velset, storage, form, walls, rows), want), (nx, ny, form)


# (without tiles, with tiles): what each was measured at stands beside the rule
@pytest.mark.parametrize("velset,storage,without,with_", [
    ("D2Q16", "fp32", (64, 6000), (32, 12100)), ("D2Q16", "fp32", (960, 960), (1024, 1024)),
    ("D2Q16", "fp16_dev", (64, 6000), (64, 8192)), ("D2Q16", "fp16_dev", (16, 16384), (16, 32768)),
    ("D2Q16", "bf16_dev", (1, 60000), (16, 32768)), ("D2Q36", "fp32", (64, 2048), (64, 4096)),
    ("D2Q36", "fp32_dev", (8, 20000), (31, 8192)), ("D2Q36", "fp16_dev", (128, 4096), (96, 6000)),
    ("D2Q36", "fp16_dev", (1000, 840), (2048, 512)), ("D2Q9", "fp16_dev", (1000, 950), (16, 32768)),
    ("D2Q16", "fp32_dev", (16, 32768), (32, 32768)), ("D2Q36", "fp32", (48, 8192), (48, 9100)),
    ("D2Q36", "fp32_dev", (16, 13000), (16, 16384)), ("D2Q36", "bf16_dev", (8, 30000), (64, 8192)),
    ("D2Q9", "fp32", (1300, 1300), (2000, 1000))])
def test_where_the_tiles_begin(velset, storage, without, with_):
    import paper_1004_5059_gb300 as tv
    v, s = tv.VELSETS[velset], tv.STORAGES[storage]
    assert not tv.tvlbm_tiled_form_tiles(*without, v, s), without
    assert tv.tvlbm_tiled_form_tiles(*with_, v, s), with_
