"""lbm_step and lbm_sp_step captured into a caller's CUDA graph, for every plan that
runs several steps a launch (cooperative launches behind a reset of their counters)
and a launch a step: replays continue the run bit for bit as direct calls do."""
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


def contexts():
    even = wl.rising_bubble(nx=48, ny=40, R=8.0, cy=14.0, Re=5.0)
    big = wl.rising_bubble(nx=1024, ny=1024, R=100.0, cy=300.0)
    return {"tile_f32_c": ("f32_c", [even], "AUTO"), "tile_f64": ("f64", [even], "AUTO"),
            "persistent": ("f32_c", [big], "AUTO"), "batched": ("f32", [big, even], "AUTO"),
            "pairs": ("f32_c", [even], "PAIRS")}


def captured(stream, calls, replays):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        calls()
    for _ in range(replays):
        g.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("name", list(contexts()))
def test_step_in_a_callers_graph(L, name):
    import torch
    form, cfgs, mode = contexts()[name]
    phis = [wl.initial_phi(c) for c in cfgs]
    stream = torch.cuda.Stream()
    with L.Simulation(cfgs, form, phi0=phis) as ref, \
            L.Simulation(cfgs, form, stream=stream.cuda_stream, phi0=phis) as sim:
        for s in (ref, sim):
            L.lbm_set_pipeline(s.ctx, getattr(L, "LBM_PIPELINE_" + mode))
            s.step(3)
            s.sync()
        captured(stream, lambda: (sim.step(6), sim.step(1), sim.step(1)), 3)   # replays start from the same parity
        ref.step(24)
        for k in range(len(cfgs)):
            for a, b in zip(sim.populations(k), ref.populations(k)):
                np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("nx,ny", [(64, 50), (63, 50), (2048, 256)])   # tiles: pairs, one cell; a launch a step
@pytest.mark.parametrize("model,scheme", [(1, 0), (0, 1)])
def test_single_phase_step_in_a_callers_graph(L, nx, ny, model, scheme):
    import torch
    x, y = np.arange(nx) / nx, np.arange(ny)[:, None] / ny
    S = 1e-4 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    cfg = dict(nx=nx, ny=ny, nu=0.1, model=model, scheme=scheme)
    stream = torch.cuda.Stream()
    with L.SourceFlow(cfg, "f32", source=S) as ref, L.SourceFlow(cfg, "f32", stream=stream.cuda_stream, source=S) as sim:
        captured(stream, lambda: (sim.step(6), sim.step(1), sim.step(1)), 3)
        ref.step(24)
        np.testing.assert_array_equal(sim.populations(), ref.populations())
