"""Nested factorisation at the line lengths where its shared-memory operands go from two stages to one:
160 | 161 cells in FP64 (1,440 bytes a cell against the 227 KB of a CTA), 241 | 242 in FP32 (960), and a
box one line wide, where no next line of the plane exists to be fetched.  G against the oracle's within
1e-12 of max |G| (FP64) or 2e-5 (FP32: the bound of its apply, doubled); the apply as in the other tests."""
import numpy as np
import pytest

import oracle as O
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nx,bz", [("fp64", 3, 160), ("fp64", 3, 161), ("fp64", 1, 161), ("fp32", 3, 241),
                                             ("fp32", 3, 242), ("fp32", 1, 242), ("fp32", 1, 5)])
def test_factor_at_the_stage_limit(precision, nx, bz):
    g = O.Geometry(nx, 3, bz, 1, 1, 1, ov=0, near_width=0, far_mode=0)
    s = synth.grid_jacobian(nx, 3, bz, 31)
    pc = O.Precond(g, s.row_ptr, s.col_idx, s.vals, solver=O.NF_COLSUM)
    sol = asm2.Solver(precision=precision, local_solver="nf_colsum")
    sol.set_grid(nx, 3, bz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(1, 1, 1, 0, 0, (2, 2, 2), "none")
    sol.factor()
    _, G = pc.sub_nf(0)
    assert np.abs(sol.nf_diagonal(0) - G).max() <= (1e-12 if precision == "fp64" else 2e-5) * np.abs(G).max()
    z, zo = sol.apply(s.b), pc.apply(s.b)
    assert np.linalg.norm(z - zo) <= (1e-10 if precision == "fp64" else 1e-5) * np.linalg.norm(zo)
