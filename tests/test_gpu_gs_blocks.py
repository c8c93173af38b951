"""Blocked modified Gram-Schmidt (one reduction per block of basis vectors) at the edges of its blocks
and of its kernels' size ranges.

In exact arithmetic the coefficients are those of modified Gram-Schmidt, and the rounding is of the same
order, so the tolerances are those of the GMRES parity tests: the oracle's iteration count, and a solution
within 1e-8 (relative) of the oracle's, both true residuals being below 1e-8."""
import numpy as np
import pytest

import oracle as O
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


def solve(g, s, restart, coop, max_iter=2000, precision="fp64"):
    sol = asm2.Solver(precision=precision, restart=restart)
    sol.set_grid(g.nx, g.ny, g.nz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(g.px, g.py, g.pz, g.ov, g.near_width, g.cnear, {0: "none", 1: "partition"}[g.far_mode])
    sol.factor()
    sol.set_tuning(coop_ortho=coop)
    x, info = sol.solve(s.b, 1e-8, max_iter)
    sol.close()
    return x, info


@pytest.mark.parametrize("coop", [True, False])
@pytest.mark.parametrize("restart", [1, 2, 8, 9, 16])
def test_short_restarts(restart, coop):
    """One-vector cycles, a group of eight, one vector more, two groups."""
    g = O.Geometry(9, 7, 5, 1, 1, 1, ov=0, near_width=0) if restart < 8 else O.Geometry(13, 11, 7, 4, 3, 1, ov=0)
    s = synth.grid_jacobian(g.nx, g.ny, g.nz, 3)
    pc = O.Precond(g, s.row_ptr, s.col_idx, s.vals)
    xo, oi = O.gmres(s.row_ptr, s.col_idx, s.vals, s.b, pc, restart, 1e-8, 2000)
    x, info = solve(g, s, restart, coop)
    assert oi.converged and info["converged"] and info["iterations"] == oi.iters
    assert np.linalg.norm(x - xo) <= 1e-8 * np.linalg.norm(xo)


@pytest.mark.parametrize("coop", [True, False])
@pytest.mark.parametrize("restart", [31, 32, 33, 64, 80])
def test_cycles_of_more_than_one_block(restart, coop):
    """75 steps of a slowly converging system (additive Schwarz without lumps, 576 boxes): cycles of one
    block of 31 or 32 vectors, of 32 and 1, of two and of three blocks.  The iterate after a fixed number
    of steps is the oracle's within 1e-8, and so is the residual."""
    g = O.Geometry(24, 24, 8, 12, 12, 4, ov=0, near_width=0, far_mode=0)
    s = synth.grid_jacobian(24, 24, 8, 3)
    pc = O.Precond(g, s.row_ptr, s.col_idx, s.vals)
    xo, oi = O.gmres(s.row_ptr, s.col_idx, s.vals, s.b, pc, restart, 1e-8, 75)
    x, info = solve(g, s, restart, coop, 75)
    assert not oi.converged and info["status"] == 4 and info["iterations"] == 75 == oi.iters
    assert np.linalg.norm(x - xo) <= 1e-8 * np.linalg.norm(xo)
    assert abs(info["rel_residual"] - oi.relres) <= 1e-8 * oi.relres


@pytest.mark.parametrize("grid", [(32, 39, 35), (43, 32, 32)])
def test_both_sides_of_the_short_vector_limit(grid):
    """131,040 unknowns: a whole cycle per block; 132,096: blocks of four (one launch) or eight (a
    launch per block).  The two paths differ only in the order of their sums."""
    nx, ny, nz = grid
    g = O.Geometry(nx, ny, nz, 4, 4, 2, ov=1)
    s = synth.grid_jacobian(nx, ny, nz, 4)
    x1, i1 = solve(g, s, 30, True, precision="fp32")
    x2, i2 = solve(g, s, 30, False, precision="fp32")
    for x, i in ((x1, i1), (x2, i2)):
        r = s.b - O.spmv(s.row_ptr, s.col_idx, s.vals, x)
        assert i["converged"] and np.linalg.norm(r) <= 1e-8 * (1 + 1e-6) * np.linalg.norm(s.b)
    assert i1["iterations"] == i2["iterations"]
    assert np.linalg.norm(x1 - x2) <= 1e-8 * np.linalg.norm(x2)


@pytest.mark.parametrize("k", [31, 32, 33, 40])
def test_orthomin_over_block_edges(k):
    """45 ORTHOMIN(k) steps of a slowly converging system: the ring wraps, and the stored directions fill one
    block of 32, one more, and a second.  The iterate and the residual are the oracle's within 1e-8."""
    g = O.Geometry(24, 24, 8, 12, 12, 4, ov=0, near_width=0, far_mode=0)
    s = synth.grid_jacobian(24, 24, 8, 3)
    pc = O.Precond(g, s.row_ptr, s.col_idx, s.vals)
    xo, oi = O.orthomin(s.row_ptr, s.col_idx, s.vals, s.b, pc, k, 1e-8, 45)
    sol = asm2.Solver(precision="fp64", restart=k, krylov="orthomin")
    sol.set_grid(24, 24, 8)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(12, 12, 4, 0, 0, (2, 2, 2), "none")
    sol.factor()
    x, info = sol.solve(s.b, 1e-8, 45)
    assert not oi.converged and info["status"] == 4 and info["iterations"] == 45 == oi.iters
    assert np.linalg.norm(x - xo) <= 1e-8 * np.linalg.norm(xo)
    assert abs(info["rel_residual"] - oi.relres) <= 1e-8 * oi.relres
