"""A row of many blocks (a cell coupled to the first cells of the grid): the preconditioner apply on both sides of
the 255 entries that the factor stream by lane takes, and the product with A, against the oracle.

Applies: the tolerances of the parity tests (1e-12, FP32 factors 1e-5, FP16 ones 5e-3).  Product: the longest sum
has 3 (lower + 1) products, so within (3 (lower + 1) + 4) eps of |A| |x| in the maximum norm."""
import numpy as np
import pytest

import oracle as O
from hub_rows import hub_system
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp16s": 5e-3}


def solver(g, s, precision):
    sol = asm2.Solver(precision=precision)
    sol.set_grid(g.nx, g.ny, g.nz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(g.px, g.py, g.pz, g.ov, g.near_width, g.cnear, g.far_mode)
    sol.factor()
    return sol


@pytest.mark.parametrize("precision", list(TOL))
@pytest.mark.parametrize("lower", [20, 100, 255, 256, 300])
@pytest.mark.parametrize("boxes", [1, 2])
def test_apply_matches_oracle(boxes, lower, precision):
    """One box without lumps (the row is a fine row), and two with them (part of it becomes lumps)."""
    g = (O.Geometry(10, 10, 6, 1, 1, 1, ov=0, near_width=0, far_mode=0) if boxes == 1 else
         O.Geometry(10, 10, 6, 2, 1, 1, ov=1))
    s = hub_system(10, 10, 6, 3, lower)
    sol = solver(g, s, precision)
    z, zo = sol.apply(s.b), O.Precond(g, s.row_ptr, s.col_idx, s.vals).apply(s.b)
    assert np.linalg.norm(z - zo) <= TOL[precision] * np.linalg.norm(zo)
    sol.set_tuning(apply_smem=0)  # the stream by rows
    assert np.array_equal(z, sol.apply(s.b))
    sol.close()


@pytest.mark.parametrize("lower", [7, 8, 30, 31, 300])
def test_spmv_matches_oracle(lower):
    s = hub_system(10, 10, 6, 3, lower)
    sol = asm2.Solver(precision="fp64")
    sol.set_grid(10, 10, 6)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(1, 1, 1, 0)
    x = synth.rhs(s.n_cells, 5)
    y, yo = sol.spmv(x), O.spmv(s.row_ptr, s.col_idx, s.vals, x)
    scale = O.spmv(s.row_ptr, s.col_idx, np.abs(s.vals), np.abs(x)).max()
    assert np.abs(y - yo).max() <= (3 * (lower + 1) + 4) * np.finfo(float).eps * scale
    sol.close()
