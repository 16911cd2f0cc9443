"""The single-phase step kernels at the edges of their launch shapes: tiles (small
domains, several steps a launch), row marches (strips of at most 126 units: cells,
or pairs in FP32 with nx even; runs in both directions; one strip of few columns)
and Remark 3's one unit a thread, against the FP64 oracles with the bars of
test_gpu_sp.py. The grids are at least one unit more and less than a strip, a tile
and a run, walled and periodic."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MODELS = {"remark3": (0, 0), "remark1": (1, 0), "remark2": (2, 0), "remark4": (0, 1)}
# tiles (smallest grids, ragged tiles), marches (a single narrow strip; one strip and
# one unit more, odd and even; several strips with ragged runs)
SIZES = [(3, 3), (4, 3), (5, 7), (33, 9), (34, 17), (130, 40), (6, 6200), (126, 2100), (252, 1500), (254, 1501),
         (1102, 331), (1101, 203)]


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1902_08933_gb300 import build, lbm
    build.build()
    return lbm


def rel(a, b):
    den = np.max(np.abs(b))
    return float(np.max(np.abs(a - b)) / (den if den > 0 else 1.0))


def reference(orc, model, cfg, S, n):
    P = orc.sp_params(cfg)
    if model == "remark3":
        g = orc.sp_init(P)
        orc.sp_step(P, S, g, n)
        return g, orc.sp_fields(P, S, g)
    if model == "remark1":
        g = orc.sp1_init(P, 1.0)
        orc.sp1_step(P, S, g, n)
        return g, orc.sp1_fields(P, S, g)
    if model == "remark2":
        g = orc.sp2_init(P)
        orc.sp2_step(P, S, g, n)
        return g, orc.sp2_fields(P, S, g)
    g, G = orc.sp4_init(P, S)
    orc.sp4_step(P, S, g, G, n)
    return g, orc.sp4_fields(P, S, g)


@pytest.mark.parametrize("model", list(MODELS))
@pytest.mark.parametrize("walls", [0, 1])
def test_shapes_match_oracle(L, orc, model, walls):
    for nx, ny in SIZES:
        cfg = dict(nx=nx, ny=ny, walls_y=walls, nu=0.07, xi=0.02, force_x=2e-6, force_y=-1e-6, p0=0.4)
        if model == "remark4":
            cfg.update(drag_lin=0.01, drag_quad=0.4)
        x, y = np.arange(nx) / nx, np.arange(ny)[:, None] / ny
        S = 1e-4 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y) + 2e-5 * np.cos(2 * np.pi * (x + 3 * y))
        steps = (3, 8)
        g, ref = reference(orc, model, cfg, S, sum(steps))
        gpu = dict(cfg, model=MODELS[model][0], scheme=MODELS[model][1])
        for form in ("f64", "f32"):
            with L.SourceFlow(gpu, form, source=S) as sim:
                for n in steps:
                    sim.step(n)
                got, gg = sim.fields(), sim.populations()
            if form == "f64":
                assert rel(gg, g) < 1e-12, (nx, ny)
            # the oracles of Remarks 1 and 2 sum absolute populations: see test_gpu_sp.py
            bar = 1e-4 if form == "f32" else (1e-10 if model in ("remark1", "remark2") else 1e-12)
            for k in ("ux", "uy"):
                assert rel(got[k], ref[k]) < bar, (nx, ny, form, k, rel(got[k], ref[k]))
