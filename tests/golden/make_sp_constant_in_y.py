"""Writes sp_constant_in_y.txt: u and p of the single-phase models on the GPU for a
source that does not vary in y, at 16 cells of each grid, as the two-kernel step of
commit c59f52a gave them (Remark 3: one kernel). Such a source drives no u_y away
from walls: what is recorded there is the rounding residue of the step's sums, which
pins the order and the rounding of each of them. Run in a tree of that commit, with
the library built, on a GPU:
    python tests/golden/make_sp_constant_in_y.py
"""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
sys.path.insert(0, ROOT)
OUT = os.path.join(os.path.dirname(os.path.abspath(__file__)), "sp_constant_in_y.txt")
MODELS = {"remark3": (0, 0), "remark1": (1, 0), "remark2": (2, 0), "remark4": (0, 1)}
# (form, nx, ny, steps): grids of tiles and grids of marches (Remark 3: one cell or pair
# a thread); pairs of cells in FP32 with nx even
GRIDS = [("f32", 16, 6, 40), ("f32", 15, 6, 40), ("f64", 15, 6, 40),
         ("f32", 130, 1200, 12), ("f32", 131, 1200, 12), ("f64", 131, 1200, 12)]


def cases():
    for model in MODELS:
        for walls in (0, 1):
            for form, nx, ny, steps in GRIDS:
                yield model, walls, form, nx, ny, steps


def run(lbm, model, walls, form, nx, ny, steps):
    """The sampled fields {name: 16 values}."""
    cfg = dict(nx=nx, ny=ny, walls_y=walls, nu=0.1, model=MODELS[model][0], scheme=MODELS[model][1], p0=1.0 / 3.0)
    if model == "remark4":
        cfg.update(force_x=1e-6, drag_lin=1e-3, drag_quad=0.1)
    x = np.arange(nx) / nx
    S = 1e-4 * (np.sin(2 * np.pi * x + 0.3) + 0.5 * np.sin(6 * np.pi * x + 1.1)) * np.ones((ny, 1))
    with lbm.SourceFlow(cfg, form, source=S) as sim:
        sim.step(steps)
        f = sim.fields()
    rows, cols = [0, 1, ny // 2, ny - 1], [0, nx // 4, nx // 2, nx - 2]
    return {k: f[k][np.ix_(rows, cols)].ravel() for k in ("ux", "uy", "p")}


def main():
    from paper_1902_08933_gb300 import lbm
    with open(OUT, "w") as f:
        f.write("# single-phase u and p for a source constant in y: make_sp_constant_in_y.py\n")
        for c in cases():
            for k, v in run(lbm, *c).items():
                f.write("%s %s %s\n" % (" ".join(map(str, c)), k, " ".join("%.17g" % x for x in v)))


if __name__ == "__main__":
    main()
