"""The tile plan (LBM_PIPELINE_AUTO, domains too small to fill the GPU with row
marches): tiles of at most 128 cells or pairs of cells, several steps in one
cooperative launch. It runs the row marches' arithmetic cell by cell, so the
populations must equal those of the march kernels (forced by asking for a run
length) bit for bit; the march kernels are held to the oracle in
test_gpu_parity.py. Sizes: the smallest grids, one more and one less than a
tile's edge in x and y, ragged parts in both, several rounds of items a block,
several instances, periodic and walled, more than the 256 steps of a launch."""
import numpy as np
import pytest

from paper_1902_08933_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

FORMS = ["f64", "f32", "f32_c", "f32_cc", "f32_g16", "f32_h16"]


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1902_08933_gb300 import build, lbm
    build.build()
    return lbm


def sized(nx, ny, walls, seed=3):
    """A noisy mixture with gravity and unequal viscosities (every term of the
    step at work) of any size."""
    c = wl.spinodal()
    c.update(nx=nx, ny=ny, walls_y=walls, nu_B=0.05, gravity=1e-6, surface_force=walls, force_x=1e-7)
    c["init"] = dict(kind="noise", seed=seed, mean=0.5, amp=0.05)
    return c


def run(L, cfgs, form, steps, rows):
    with L.Simulation(cfgs, form, phi0=[wl.initial_phi(c) for c in cfgs]) as sim:
        L.lbm_set_launch(sim.ctx, 0, rows)   # 0: the tile plan; else row marches
        n0 = L.lbm_step_launch_count(sim.ctx)
        for n in steps:
            sim.step(n)
        launches = L.lbm_step_launch_count(sim.ctx) - n0
        return [sim.populations(k) for k in range(len(cfgs))], launches


def check(L, cfgs, form, steps, launches):
    got, n = run(L, cfgs, form, steps, 0)
    assert n == launches
    ref, _ = run(L, cfgs, form, steps, 8)
    for k, (a, b) in enumerate(zip(got, ref)):
        for x, y in zip(a, b):
            assert np.array_equal(x, y), (form, cfgs[k]["nx"], cfgs[k]["ny"])


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("walls", [0, 1])
def test_tiles_equal_marches(L, form, walls):
    for nx, ny in ((3, 3), (4, 3), (7, 5), (15, 4), (16, 4), (18, 9), (31, 8), (32, 33), (34, 65), (130, 37)):
        check(L, [sized(nx, ny, walls)], form, (1, 2, 9), 3)


@pytest.mark.parametrize("form", FORMS)
def test_tiles_several_rounds_and_launches(L, form):
    # more items than resident blocks; 300 steps are two launches
    for nx, ny in ((520, 301), (401, 297)):
        check(L, [sized(nx, ny, 1)], form, (6,), 1)
    check(L, [sized(24, 17, 0)], form, (300, 1), 3)


@pytest.mark.parametrize("form", FORMS)
def test_tiles_several_instances(L, form):
    sizes = ((20, 12, 0), (64, 50, 1), (34, 3, 0)) if form != "f64" else ((20, 12, 0), (33, 50, 1), (7, 3, 0))
    check(L, [sized(nx, ny, w, seed=k) for k, (nx, ny, w) in enumerate(sizes)], form, (3, 20), 2)
