"""Nested factorisation on either side of the number of boxes (two per SM, 304) where its factorisation goes from CTAs
of 256 threads to 128, and where three or more boxes share an SM in the apply: lines shorter and longer than a
warp.  G against the oracle's and the apply as in test_gpu_nf_stages.py, with its tolerances."""
import numpy as np
import pytest

import oracle as O
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("px,py,nz", [(19, 16, 3), (18, 17, 3), (34, 18, 5), (18, 17, 37)])
def test_more_boxes_than_two_per_sm(precision, px, py, nz):
    nx, ny = px + 3, py + 2
    g = O.Geometry(nx, ny, nz, px, py, 1, ov=1, near_width=0, far_mode=0)
    s = synth.grid_jacobian(nx, ny, nz, 37)
    pc = O.Precond(g, s.row_ptr, s.col_idx, s.vals, solver=O.NF_COLSUM)
    sol = asm2.Solver(precision=precision, local_solver="nf_colsum")
    sol.set_grid(nx, ny, nz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(px, py, 1, 1, 0, (2, 2, 2), "none")
    sol.factor()
    for k in (0, px + 1, px * py // 2, px * py - 1):
        _, G = pc.sub_nf(k)
        assert np.abs(sol.nf_diagonal(k) - G).max() <= (1e-12 if precision == "fp64" else 2e-5) * np.abs(G).max()
    z, zo = sol.apply(s.b), pc.apply(s.b)
    assert np.linalg.norm(z - zo) <= (1e-10 if precision == "fp64" else 1e-5) * np.linalg.norm(zo)
