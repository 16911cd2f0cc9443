"""Graph replay against direct launches for the plans that run a launch a step, each
pinned by its load path or run length (by default most domains run several steps a
launch, without graphs): one launch class for every load path, several classes as
graph branches, and the D3Q15 step. 161 steps from an odd start: two whole replays of
64 steps (fewer per replay with several classes) and a rest of direct launches."""
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


def cases(classes):
    cfgs = [wl.static_droplet(n=64, R=15)]
    if classes > 1:
        cfgs += [wl.rising_bubble(nx=160, ny=48, R=10, cy=18, W=4.0, Re=10.0), wl.static_droplet(n=33, R=8)]
    return cfgs


@pytest.mark.parametrize("form,mode,rows,classes", [
    ("f64", "PLAIN", 0, 1), ("f64", "AUTO", 8, 3), ("f32_c", "PAIRS", 0, 1), ("f32_c", "AUTO", 8, 3),
    ("f32", "ASYNC", 0, 1), ("f32", "TMA", 0, 1), ("f32_h16", "PAIRS", 0, 1), ("f32_g16", "PLAIN", 0, 1)])
def test_graph_replay_matches_direct_launches(L, form, mode, rows, classes):
    cfgs = cases(classes)
    phis = [wl.initial_phi(c) for c in cfgs]
    out = []
    for graphs in (True, False):
        with L.Simulation(cfgs, form, phi0=phis) as sim:
            L.lbm_set_pipeline(sim.ctx, getattr(L, "LBM_PIPELINE_" + mode))
            L.lbm_set_launch(sim.ctx, 0, rows)
            L.lbm_set_graphs(sim.ctx, graphs)
            per_step = L.lbm_launches_per_step(sim.ctx)
            assert per_step == classes if classes == 1 else per_step >= 2
            for n in (1, 157, 3):
                sim.step(n)
            assert L.lbm_step_launch_count(sim.ctx) == 161 * per_step   # a launch a step and class
            out.append([sim.populations(k) for k in range(len(cfgs))])
    for a, b in zip(*out):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("form", ["f64", "f32_c"])
def test_graph_replay_matches_direct_launches_d3(L, form):
    cfg = wl.rising_bubble3(nx=16, ny=24, nz=16, R=5.0, cy=8.0, Re=5.0)
    out = []
    for graphs in (True, False):
        with L.Simulation([cfg], form, phi0=[wl.initial_phi(cfg)]) as sim:
            L.lbm_set_graphs(sim.ctx, graphs)
            for n in (1, 157, 3):
                sim.step(n)
            out.append(sim.populations(0))
    for x, y in zip(*out):
        assert np.array_equal(x, y)
