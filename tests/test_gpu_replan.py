"""A context whose plan changes between calls: what one plan keeps for itself (the
persistent plan's neighbours, counters and monitor buffers) serves no other plan.
Monitored steps under LBM_PIPELINE_AUTO (one FP32 domain: the persistent plan), then
every step monitored under another mode, against a context that ran the paired plan
throughout: the state bit for bit (the plans share the cell arithmetic), the records
with the bars of test_gpu_persistent.py."""
import ctypes

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


@pytest.mark.parametrize("first,second", [("AUTO", "BATCHED"), ("PERSISTENT", "BATCHED"), ("BATCHED", "AUTO"),
                                          ("AUTO", "PLAIN"), ("BATCHED", "PERSISTENT")])
def test_every_step_record_after_a_change_of_plan(L, first, second):
    import torch
    cfg = wl.rising_bubble(nx=256, ny=144, R=18, cy=48, W=4.0, Re=8.0)
    phi0 = wl.initial_phi(cfg)
    size, n = ctypes.sizeof(L.lbm_monitor), 9
    out = {}
    for name, modes in (("ref", ("PAIRS", "PAIRS")), ("got", (first, second))):
        buf = torch.zeros(2 * n * size, dtype=torch.uint8).pin_memory()
        with L.Simulation([cfg], "f32_c", phi0=[phi0]) as sim:
            L.lbm_set_monitor(sim.ctx, True)
            for k, mode in enumerate(modes):
                L.lbm_set_pipeline(sim.ctx, getattr(L, "LBM_PIPELINE_" + mode))
                L.lbm_step_monitored_all(sim.ctx, n, buf.data_ptr() + k * n * size)
                sim.step(3)
            sim.sync()
            out[name] = (sim.populations(0), [L.lbm_monitor.from_address(buf.data_ptr() + k * size) for k in range(2 * n)],
                         buf)
    if "PLAIN" not in (first, second):   # (the one-cell kernel is another compilation of the arithmetic)
        for a, b in zip(out["got"][0], out["ref"][0]):
            assert np.array_equal(a, b)
    for r, q in zip(out["got"][1], out["ref"][1]):
        assert r.time == q.time and r.nonfinite == 0 and r.device_status == 0
        assert abs(r.sum_phi - q.sum_phi) <= cfg["nx"] * cfg["ny"] * 2.0 ** -24
        assert abs(r.kinetic_energy - q.kinetic_energy) <= 1e-4 * q.kinetic_energy
        assert abs(r.max_u - q.max_u) <= 1e-4 * q.max_u
