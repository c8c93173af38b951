"""Every inner product and Gram entry of a block of 1 .. 32 directions, and of a block's first vector after a full
one: the iterate after n = 1 .. 33 steps of one cycle, by each kernel that takes a block's sums together (the
cooperative Gram-Schmidt, its per-launch form, ORTHOMIN's projections).  A step's coefficients are all of a block's
sums, so one lost share of one sum moves the iterate.  Tolerance as in the other block tests: the oracle's iterate
and residual within 1e-8."""
import numpy as np
import pytest

import oracle as O
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system():
    """Slowly converging (additive Schwarz without lumps, 576 boxes)."""
    g = O.Geometry(24, 24, 8, 12, 12, 4, ov=0, near_width=0, far_mode=0)
    s = synth.grid_jacobian(24, 24, 8, 3)
    return g, s, O.Precond(g, s.row_ptr, s.col_idx, s.vals)


@pytest.mark.parametrize("kernel", ["cooperative", "per_launch", "orthomin"])
def test_iterate_after_each_number_of_steps(system, kernel):
    g, s, pc = system
    om = kernel == "orthomin"
    sol = asm2.Solver(precision="fp64", restart=40, krylov="orthomin" if om else "gmres")
    sol.set_grid(g.nx, g.ny, g.nz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(g.px, g.py, g.pz, 0, 0, (2, 2, 2), "none")
    sol.factor()
    sol.set_tuning(coop_ortho=kernel == "cooperative")
    for n in range(1, 34):
        xo, oi = (O.orthomin if om else O.gmres)(s.row_ptr, s.col_idx, s.vals, s.b, pc, 40, 1e-8, n)
        x, info = sol.solve(s.b, 1e-8, n)
        assert not oi.converged and info["iterations"] == n == oi.iters
        assert np.linalg.norm(x - xo) <= 1e-8 * np.linalg.norm(xo), n
        assert abs(info["rel_residual"] - oi.relres) <= 1e-8 * oi.relres, n
    sol.close()
