"""ORTHOMIN with a right-hand side so small that (q, q) of the last directions lies below 2^-1024, where its
reciprocal overflows though it is still good to twelve digits: the steps of the unscaled problem (every operation
scales by the same power of two), and its solution within the 1e-8 of the ORTHOMIN tests.  The oracle's own
solution moves by less than 1e-15 over these scales."""
import numpy as np
import pytest

import oracle as O
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-490, -495, -500])
def test_small_right_hand_side(exponent):
    s = synth.grid_jacobian(10, 10, 5, 1)
    pc = O.Precond(O.Geometry(10, 10, 5, 2, 2, 1, ov=1), s.row_ptr, s.col_idx, s.vals)
    xo, oi = O.orthomin(s.row_ptr, s.col_idx, s.vals, s.b, pc, 10, 1e-8, 2000)
    sol = asm2.Solver(precision="fp64", restart=10, krylov="orthomin")
    sol.set_grid(10, 10, 5)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(2, 2, 1, 1)
    sol.factor()
    x, info = sol.solve(np.ldexp(s.b, exponent), 1e-8, 2000)
    assert oi.converged and info["converged"] and info["iterations"] == oi.iters
    assert np.linalg.norm(np.ldexp(x, -exponent) - xo) <= 1e-8 * np.linalg.norm(xo)
    sol.close()
