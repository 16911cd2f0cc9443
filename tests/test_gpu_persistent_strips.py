"""The persistent plan where the last strip is 2 to 4 columns wide (widths just above a
whole number of strips), so that an item's neighbours lie beyond that strip too: bit
for bit the per-step paired plan, as in test_gpu_persistent.py, for the mode itself and
for LBM_PIPELINE_AUTO, which takes it for one domain."""
import numpy as np
import pytest

from paper_1902_08933_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1902_08933_gb300 import build, lbm
    build.build()
    return lbm


def run(L, cfg, form, mode, tile=0):
    with L.Simulation([cfg], form, phi0=[wl.initial_phi(cfg)]) as sim:
        L.lbm_set_pipeline(sim.ctx, getattr(L, "LBM_PIPELINE_" + mode))
        L.lbm_set_launch(sim.ctx, tile, 0)
        for n in (3, 40):
            sim.step(n)
        launches = L.lbm_step_launch_count(sim.ctx)
        return sim.populations(0), launches


@pytest.mark.parametrize("form", ["f32_c", "f32_h16"])
@pytest.mark.parametrize("nx,ny,mode,tile", [(66, 300, "PERSISTENT", 64), (258, 200, "PERSISTENT", 256),
                                             (260, 200, "PERSISTENT", 128), (1026, 1100, "AUTO", 0),
                                             (5122, 300, "AUTO", 0)])
def test_narrow_last_strip(L, form, nx, ny, mode, tile):
    for walls in (0, 1):
        R = min(nx, ny) / 8.0
        cfg = dict(wl.rising_bubble(nx=nx, ny=ny, R=R, cy=3 * R, W=4.0, Re=8.0), walls_y=walls)
        cfg["init"] = dict(cfg["init"], cx=nx - 4.0)   # across the seam
        ref, _ = run(L, cfg, form, "PAIRS", tile)
        got, launches = run(L, cfg, form, mode, tile)
        assert launches == 2   # a launch for each call: the several-step kernel ran
        for a, b in zip(got, ref):
            assert np.array_equal(a, b), (nx, walls)
