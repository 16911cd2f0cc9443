"""Field read-back of small domains (one launch over tiles of 16 x 8 cells) against
the three passes that larger ones take. A domain and the same one repeated m times
in x until it takes the passes hold the same populations cell by cell (the steps'
arithmetic does not depend on a cell's place; m odd keeps the parity of nx, which
chooses between one and two cells a thread), so the fields must be equal bit for
bit; P, whose expression the compiler may contract differently in the two kernels,
within 1e-13 of its largest value (about 450 roundings of it). Sizes: the smallest,
one less than, equal to and one more than a tile's edge, several tiles with ragged
parts, periodic and walled."""
import numpy as np
import pytest

from paper_1902_08933_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CELLS = 1 << 19   # more cells than any domain read back over tiles


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1902_08933_gb300 import build, lbm
    build.build()
    return lbm


@pytest.mark.parametrize("form", ["f64", "f32", "f32_c", "f32_cc", "f32_g16", "f32_h16"])
@pytest.mark.parametrize("nx,ny,walls", [(3, 3, 0), (4, 3, 1), (15, 7, 1), (16, 8, 0), (17, 9, 1), (33, 16, 0),
                                         (130, 37, 1)])
def test_tile_read_back_equals_the_passes(L, form, nx, ny, walls):
    c = wl.spinodal()
    c.update(nx=nx, ny=ny, walls_y=walls, nu_B=0.05, gravity=1e-6, surface_force=walls, force_x=1e-7)
    c["init"] = dict(kind="noise", seed=5, mean=0.5, amp=0.05)
    phi0 = wl.initial_phi(c)
    m = CELLS // (nx * ny) | 1
    m += 2 * (m * nx * ny <= CELLS)
    big = dict(c, nx=m * nx)
    with L.Simulation(c, form, phi0=[phi0]) as small, L.Simulation(big, form, phi0=[np.tile(phi0, (1, m))]) as large:
        small.step(3)
        large.step(3)
        a, b = small.fields(0), large.fields(0)
        for name in ("phi", "ux", "uy", "p", "rho", "mu"):
            assert np.array_equal(np.tile(a[name], (1, m)), b[name]), name
        assert np.max(np.abs(np.tile(a["P"], (1, m)) - b["P"])) <= 1e-13 * np.max(np.abs(b["P"]))
        few = small.fields(0, ("phi", "uy", "mu"))   # a part of the mask, without P
        for name in few:
            assert np.array_equal(few[name], a[name]), name
