"""Handles on several threads and streams at once, with subdomains of different sizes: the launches ask for different
amounts of shared memory of the same kernels, and every call gives what the handle gives alone."""
import threading

import numpy as np
import pytest
import torch

from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("local", ["colsum", "nf_colsum"])
def test_factor_and_apply_on_several_threads(local):
    grids = [((10, 8, 40), (2, 2, 1))] + [((6, 6, 4), (2, 2, 1))] * 4
    work = []
    for k, (grid, part) in enumerate(grids):
        s = synth.grid_jacobian(*grid, 40 + k)
        stream = torch.cuda.Stream()
        sol = asm2.Solver(precision="fp32", local_solver=local, stream=stream.cuda_stream)
        sol.set_grid(*grid)
        sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
        if local == "colsum":
            sol.set_partition(*part, 1)
        else:
            sol.set_partition(*part, 1, 0, (2, 2, 2), "none")
        sol.factor()
        work.append((sol, s, sol.apply(s.b), stream))
    failed = []

    def turn(sol, s, want):
        try:
            for _ in range(20):
                sol.update_values(s.vals)
                sol.factor()
                for _ in range(100):
                    if not np.array_equal(sol.apply(s.b), want):
                        failed.append("other values")
        except Exception as e:  # noqa: BLE001
            failed.append(repr(e))

    threads = [threading.Thread(target=turn, args=w[:3]) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[:3]
    for w in work:
        w[0].close()
