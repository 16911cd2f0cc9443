"""The bounded waits of every launch that runs several steps, made to run out
(lbm_inject_step_wait_timeout, lbm_sp_inject_wait_timeout): the launch gives up and
returns, LBM_ETIMEOUT is reported, and after lbm_load / lbm_sp_init the run continues
exactly as an undisturbed one. Nothing faults or hangs: each wait ends after the given
number of rounds. Also launches back to back (more steps than the 256 of one)."""
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
    odd = wl.rising_bubble(nx=49, ny=41, R=8.0, cy=14.0, Re=5.0)
    big = wl.rising_bubble(nx=1024, ny=1024, R=100.0, cy=300.0)
    # tiles: pairs, one cell in FP32 and FP64, several instances; then a domain of the
    # persistent plan, and instances of the batched launch
    return {"tile_f32_c": ("f32_c", [even]), "tile_f32_odd": ("f32", [odd]), "tile_f64": ("f64", [even]),
            "tile_instances": ("f32_h16", [even, wl.static_droplet(n=32, R=8.0), even]),
            "persistent": ("f32_c", [big]), "batched": ("f32", [big, even])}


@pytest.mark.parametrize("name", list(contexts()))
def test_step_wait_runs_out_and_the_checkpoint_recovers(L, tmp_path, name):
    form, cfgs = contexts()[name]
    phis = [wl.initial_phi(c) for c in cfgs]
    ckpt = str(tmp_path / "state.bin")
    with L.Simulation(cfgs, form, phi0=phis) as ref, L.Simulation(cfgs, form, phi0=phis) as sim:
        ref.step(30)
        sim.step(10)
        L.lbm_save(sim.ctx, ckpt)
        sim.step(7)
        for bad in (0, (1 << 21) + 1):
            with pytest.raises(L.LbmError) as e:
                L.lbm_inject_step_wait_timeout(sim.ctx, bad)
            assert e.value.status == L.LBM_EINVAL
        L.lbm_inject_step_wait_timeout(sim.ctx, 1 << 12)
        for read in (sim.sync, lambda: sim.fields(0, ("phi",)), lambda: sim.diagnostics(0)):
            with pytest.raises(L.LbmError) as e:
                read()
            assert e.value.status == L.LBM_ETIMEOUT
        L.lbm_load(sim.ctx, ckpt)
        sim.step(20)
        for k in range(len(cfgs)):
            for a, b in zip(sim.populations(k), ref.populations(k)):
                np.testing.assert_array_equal(a, b)


def test_step_wait_hook_needs_a_launch_of_several_steps(L):
    cfg = wl.rising_bubble(nx=48, ny=40, R=8.0, cy=14.0, Re=5.0)
    with L.Simulation([cfg], "f32_c", phi0=[wl.initial_phi(cfg)]) as sim:
        L.lbm_set_pipeline(sim.ctx, L.LBM_PIPELINE_PAIRS)
        with pytest.raises(L.LbmError) as e:
            L.lbm_inject_step_wait_timeout(sim.ctx, 100)
        assert e.value.status == L.LBM_ESTATE
        sim.step(3)
        sim.sync()


def _source(nx, ny):
    x, y = np.arange(nx) / nx, np.arange(ny)[:, None] / ny
    return 1e-4 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)


@pytest.mark.parametrize("model,scheme", [(0, 0), (1, 0), (2, 0), (0, 1)])
@pytest.mark.parametrize("form,nx", [("f32", 64), ("f32", 63), ("f64", 64)])
def test_single_phase_wait_runs_out_and_init_recovers(L, model, scheme, form, nx):
    cfg = dict(nx=nx, ny=50, nu=0.1, model=model, scheme=scheme)
    S = _source(nx, 50)
    with L.SourceFlow(cfg, form, source=S) as sim, L.SourceFlow(cfg, form, source=S) as ref:
        ref.step(600)                     # launches of 256, 256 and 88 steps
        sim.step(5)
        for bad in (0, (1 << 21) + 1):
            with pytest.raises(L.LbmError) as e:
                L.lbm_sp_inject_wait_timeout(sim.ctx, bad)
            assert e.value.status == L.LBM_EINVAL
        L.lbm_sp_inject_wait_timeout(sim.ctx, 1 << 12)
        for read in (sim.fields, sim.populations):
            with pytest.raises(L.LbmError) as e:
                read()
            assert e.value.status == L.LBM_ETIMEOUT
        sim.init(S)
        for _ in range(600):              # one step a launch: no waits
            sim.step(1)
        np.testing.assert_array_equal(sim.populations(), ref.populations())
        assert np.isfinite(ref.populations()).all()


def test_single_phase_hook_needs_tiles(L):
    cfg = dict(nx=2048, ny=512, nu=0.1, model=1)
    with L.SourceFlow(cfg, "f32", source=_source(2048, 512)) as sim:
        with pytest.raises(L.LbmError) as e:
            L.lbm_sp_inject_wait_timeout(sim.ctx, 100)
        assert e.value.status == L.LBM_ESTATE
        sim.step(3)
        sim.fields()
