"""ORTHOMIN's projections run with one CTA per SM while a launch has no more work items than SMs and with two
beyond that.  Each system's arithmetic does not depend on the others in a batch, so the same system solved alone (94
items) and beside others (470) gives the same bits, below and above 32 stored directions."""
import numpy as np
import pytest

from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [3, 34])
def test_alone_and_in_a_batch_of_many_items(k):
    systems = [synth.grid_jacobian(40, 40, 20, 50 + i) for i in range(5)]
    sols = []
    for s in systems:
        sol = asm2.Solver(precision="fp64", restart=k, krylov="orthomin")
        sol.set_grid(40, 40, 20)
        sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
        sol.set_partition(5, 5, 1, 1)
        sol.factor()
        sols.append(sol)
    alone = [sol.solve(s.b, 1e-12, 45) for sol, s in zip(sols, systems)]
    xs, infos = asm2.solve_batch(sols, [s.b for s in systems], 1e-12, 45)
    for (x, info), y, other in zip(alone, xs, infos):
        assert info["iterations"] == other["iterations"]
        np.testing.assert_array_equal(x, y)
