"""Test systems with one long row: a grid Jacobian whose last cell is coupled to the first cells of the grid as
well (a well cell and its perforations)."""
import dataclasses

import numpy as np

from paper_1401_7227_gb300 import synth


def hub_system(nx, ny, nz, seed, lower):
    """The last cell's row has `lower` blocks to the left of its diagonal."""
    s = synth.grid_jacobian(nx, ny, nz, seed)
    n, hub = s.n_cells, s.n_cells - 1
    near = [int(c) for c in s.col_idx[s.row_ptr[hub]:s.row_ptr[hub + 1] - 1]]
    far = [c for c in range(n - 1) if c not in near][:lower - len(near)]
    size = 0.05 * np.linalg.norm(s.vals[s.row_ptr[hub + 1] - 1], 2)
    rng = np.random.default_rng(seed)
    blocks = size * rng.uniform(-1.0, 1.0, (2, len(far), 3, 3)) / len(far)
    rows = [dict(zip(s.col_idx[s.row_ptr[r]:s.row_ptr[r + 1]].tolist(), s.vals[s.row_ptr[r]:s.row_ptr[r + 1]]))
            for r in range(n)]
    for k, c in enumerate(far):
        rows[hub][c], rows[c][hub] = blocks[0, k], blocks[1, k]
    cols = [sorted(r) for r in rows]
    return dataclasses.replace(
        s, row_ptr=np.cumsum([0] + [len(c) for c in cols]).astype(np.int32),
        col_idx=np.concatenate(cols).astype(np.int32),
        vals=np.ascontiguousarray([rows[r][c] for r in range(n) for c in cols[r]]))
