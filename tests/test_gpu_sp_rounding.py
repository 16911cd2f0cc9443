"""The single-phase steps round as they always have: u and p for a source that does
not vary in y against values recorded from the two-kernel step (tests/golden/
make_sp_constant_in_y.py). Away from walls u_y is then nothing but the rounding
residue of the step's sums, so a sum in another order or a product rounded elsewhere
shows as a difference of the size of u_y itself, in every model and kernel (tiles,
row marches, one unit a thread; pairs of cells, one cell, FP64). Each field may be off
by the 2-norm bound of its type: 2e-5 (FP32), 1e-9 (FP64); a recorded field of zeros
is zero."""
import importlib.util
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
spec = importlib.util.spec_from_file_location("make_sp", os.path.join(HERE, "golden", "make_sp_constant_in_y.py"))
make_sp = importlib.util.module_from_spec(spec)
spec.loader.exec_module(make_sp)


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1902_08933_gb300 import build, lbm
    build.build()
    return lbm


@pytest.fixture(scope="module")
def recorded():
    out = {}
    with open(make_sp.OUT) as f:
        for line in f:
            if not line.startswith("#"):
                t = line.split()
                out[tuple(t[:7])] = np.array(t[7:], dtype=np.float64)
    return out


@pytest.mark.parametrize("model", list(make_sp.MODELS))
def test_source_constant_in_y_keeps_its_residue(L, recorded, model):
    for case in make_sp.cases():
        if case[0] != model:
            continue
        got = make_sp.run(L, *case)
        for k, v in got.items():
            ref = recorded[tuple(map(str, case)) + (k,)]
            bound = 2e-5 if case[2] == "f32" else 1e-9
            assert np.linalg.norm(v - ref) <= bound * np.linalg.norm(ref), (case, k, v, ref)
