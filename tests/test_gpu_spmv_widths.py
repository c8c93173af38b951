"""y = A x for rows of one to seven blocks (the loads run one block ahead, two blocks a turn) and for row counts
around a CTA's 128 and an item's 256, against the oracle: each sum has at most 21 products, so within
25 eps of |A| |x| in the maximum norm."""
import numpy as np
import pytest

import oracle as O
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (1, 1, 2), (1, 1, 5), (2, 1, 5), (2, 2, 5), (3, 2, 5), (3, 3, 4), (1, 1, 127),
                                      (16, 8, 1), (43, 3, 1), (16, 16, 1), (257, 1, 1)])
def test_spmv_matches_oracle(nx, ny, nz):
    s = synth.grid_jacobian(nx, ny, nz, 7)
    sol = asm2.Solver(precision="fp64")
    sol.set_grid(nx, ny, nz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(1, 1, 1, 0)
    x = synth.rhs(s.n_cells, 5)
    y, yo = sol.spmv(x), O.spmv(s.row_ptr, s.col_idx, s.vals, x)
    scale = O.spmv(s.row_ptr, s.col_idx, np.abs(s.vals), np.abs(x)).max()
    assert np.abs(y - yo).max() <= 25 * np.finfo(float).eps * scale
