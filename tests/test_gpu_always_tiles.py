"""The tiled kernel on domains that the tiled form otherwise runs without tiles (tvlbm_set_always_tiles):
every tile configuration against the oracle in FP64, and against the one-cell-per-thread and strip
kernels bit for bit, with walls, a per-row reference, other time steps, ragged and tiny domains.
Tolerances of the FP64 comparison: those of test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads

WALLS = (0.02, 1.0, -0.03, 1.05)


@pytest.fixture(scope="module")
def tv():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1004_5059_gb300 as tv
    return tv


def make(tv, nx, ny, velset, storage, form, tile=0, walls=None, dt=1.0, rows=False, graphs=True, tau=0.9):
    sim = tv.Simulation(nx, ny, velset, tau=tau, dt=dt, walls=walls, storage=storage, form=form, graphs=graphs)
    if form == "tiled":
        sim.set_tile(tile)
        sim.set_always_tiles()
        assert sim.runs_tiles()
    if rows:
        sim.set_reference_rows(0.01, 0.0, np.linspace(1.0, 1.05, ny))
    sim.init_moments(*workloads.random_smooth(nx, ny, seed=nx + ny, amp_u=0.04, amp_T=0.03))
    return sim


def raw(sim, storage):
    out = sim.raw_populations()
    sim.close()
    return out.view(np.uint16) if storage == "bf16_dev" else out


@pytest.mark.gpu
@pytest.mark.parametrize("tile", [0, 1, 2, 3])
@pytest.mark.parametrize("velset,nx,ny,walls,dt", [
    ("D2Q9", 33, 35, None, 1.0), ("D2Q16", 37, 29, None, 1.0), ("D2Q36", 45, 23, None, 0.6), ("D2Q16", 1, 12, None, 1.2),
    ("D2Q36", 3, 5, None, 1.0), ("D2Q9", 65, 41, WALLS, 1.0), ("D2Q16", 29, 21, WALLS, 0.37), ("D2Q36", 29, 21, WALLS, 1.0)])
def test_fp64_tiles_match_oracle(tv, tile, velset, nx, ny, walls, dt):
    sim = make(tv, nx, ny, velset, "fp64", "tiled", tile, walls, dt)
    ref = oracle.Oracle(nx, ny, velset, tau=0.9, dt=dt, walls=walls)
    ref.init_moments(*workloads.random_smooth(nx, ny, seed=nx + ny, amp_u=0.04, amp_T=0.03))
    sim.step(30)
    ref.run(30)
    got = sim.populations_f64()
    assert np.max(np.abs(got - ref.f)) < 1e-11 * np.max(np.abs(ref.f))
    sim.close()


@pytest.mark.gpu
@pytest.mark.parametrize("tile", [0, 1, 2, 3])
@pytest.mark.parametrize("velset", ["D2Q9", "D2Q16", "D2Q36"])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp32_dev", "fp16_dev", "bf16_dev"])
def test_tiles_equal_the_other_kernels(tv, tile, velset, storage):
    for nx, ny, walls, dt, rows in ((1, 1, None, 1.0, False), (70, 33, None, 0.8, False), (130, 41, WALLS, 1.0, False),
                                    (65, 37, WALLS, 0.8, True), (64, 64, None, 1.0, False)):
        if rows and not storage.endswith("_dev"):
            continue
        want = make(tv, nx, ny, velset, storage, "strip", walls=walls, dt=dt, rows=rows, graphs=False)
        plain = make(tv, nx, ny, velset, storage, "plain", walls=walls, dt=dt, rows=rows, graphs=False)
        sim = make(tv, nx, ny, velset, storage, "tiled", tile, walls, dt, rows)
        for s in (want, plain, sim):
            s.step(35)  # one captured graph and three single steps
        want, plain, sim = raw(want, storage), raw(plain, storage), raw(sim, storage)
        assert np.all(np.isfinite(want.astype(np.float64)))
        assert np.array_equal(sim, want) and np.array_equal(sim, plain), (nx, ny, walls, dt, rows)


@pytest.mark.gpu
def test_switching_between_steps(tv):
    """The switch takes effect at the next step, captured graphs included, and changes no population."""
    a = make(tv, 100, 75, "D2Q16", "fp32", "strip")
    b = tv.Simulation(100, 75, "D2Q16", tau=0.9, storage="fp32")
    b.init_moments(*workloads.random_smooth(100, 75, seed=175, amp_u=0.04, amp_T=0.03))
    assert not b.runs_tiles()
    for on in (False, True, True, False):
        b.set_always_tiles(on)
        assert b.runs_tiles() == on
        a.step(40)
        b.step(40)
    assert np.array_equal(raw(a, "fp32"), raw(b, "fp32"))
    big = tv.Simulation(1200, 1100, "D2Q16", storage="fp32")
    assert big.runs_tiles()
    big.set_form("plain")
    assert not big.runs_tiles()
    big.close()


def test_rule_without_a_context():
    import paper_1004_5059_gb300 as tv
    tiles = lambda nx, ny, v, s: tv.tvlbm_tiled_form_tiles(nx, ny, tv.VELSETS[v], tv.STORAGES[s])
    for v in tv.VELSETS:
        for s in tv.STORAGES:
            assert tiles(4096, 4096, v, s) and not tiles(40, 30, v, s)
    assert tiles(304, 301, "D2Q16", "fp64") and not tiles(304, 299, "D2Q16", "fp64")  # 600 cells per SM
    for args in ((0, 8, 16, 1), (8, 8, 17, 1), (8, 8, 16, 9)):
        with pytest.raises(tv.TvlbmError) as e:
            tv.tvlbm_tiled_form_tiles(*args)
        assert e.value.code == tv.TVLBM_EINVAL
