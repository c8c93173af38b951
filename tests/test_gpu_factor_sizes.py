"""The block ILU(0) factorisation on both sides of the subdomain counts where its CTA size changes (one CTA
per SM, two per SM: 152 and 304 on this GPU), and with a level wider than a CTA takes at once: the apply against
the oracle's within 1e-10, as the factors differ by rounding only (boxes of a few cells, condition below 1e4)."""
import numpy as np
import pytest

import oracle as O
from paper_1401_7227_gb300 import asm2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,px,py", [(38, 16, 2, 19, 8), (34, 18, 2, 17, 9), (38, 32, 2, 19, 16), (122, 10, 2, 61, 5),
                                            (60, 60, 3, 1, 1), (3, 1, 1, 3, 1)])
def test_apply_matches_oracle(nx, ny, nz, px, py):
    g = O.Geometry(nx, ny, nz, px, py, 1, ov=1)
    s = synth.grid_jacobian(nx, ny, nz, 9)
    pc = O.Precond(g, s.row_ptr, s.col_idx, s.vals)
    sol = asm2.Solver(precision="fp64")
    sol.set_grid(nx, ny, nz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(px, py, 1, 1, g.near_width, g.cnear, g.far_mode)
    sol.factor()
    z, zo = sol.apply(s.b), pc.apply(s.b)
    assert np.linalg.norm(z - zo) <= 1e-10 * np.linalg.norm(zo)
