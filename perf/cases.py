"""The work that a user of this package has it do, as measurable cases.

Every case goes through the public entry points of ``paper_1401_7227_gb300.asm2``: a linear solve
(set-up kept, a new right-hand side), a Newton step (new values on a known pattern, re-factorisation
and solve), a batch of independent systems, a stream of served requests, and the two operators on
their own (the matrix product and the preconditioner).  Sizes and options come from the package's
workloads (``synth.WORKLOADS``, ``synth.batch_grid``, the served grids of ``bench.py``) and from odd
grids between them, where no extent is a multiple of a lump, a box or a warp.

The inputs are black-oil-like Jacobians with the recipe of ``paper_1401_7227_gb300/synth.py``
(layered lognormal permeability, upwinded saturation rows, conservative block columns, two wells),
built on the GPU so that a million cells take a fraction of a second.
"""
import math

import numpy as np
import torch

from paper_1401_7227_gb300 import asm2

RTOL = 1e-8
MAX_ITER = 2000


def _grid(nx, ny, nz, px, py, pz, overlap, **more):
    return dict(nx=nx, ny=ny, nz=nz, px=px, py=py, pz=pz, overlap=overlap, **more)


def listed():
    return [
        # the smallest call: one solve of a few hundred cells, where latency and launches are the cost
        dict(name="solve_10x10x5_fp64", kind="solve", **_grid(10, 10, 5, 2, 2, 1, 1), precision="fp64", restart=30,
             sigma=1.0, local="colsum", krylov="gmres", iters=26),
        # the same matrix, a new right-hand side: the mid-size workload in the default precision
        dict(name="solve_64x64x16_fp64", kind="solve", **_grid(64, 64, 16, 8, 8, 1, 1), precision="fp64", restart=30,
             sigma=1.0, local="colsum", krylov="gmres", iters=31),
        # the paper's other accelerator, truncated instead of restarted
        dict(name="solve_30x30x9_orthomin", kind="solve", **_grid(30, 30, 9, 3, 3, 1, 1), precision="fp64", restart=30,
             sigma=1.0, local="colsum", krylov="orthomin", iters=31),
        # one Newton step of the mid-size workload with the mixed-precision factors
        dict(name="step_64x64x16_fp32", kind="step", **_grid(64, 64, 16, 8, 8, 1, 1), precision="fp32", restart=30,
             sigma=1.0, local="colsum", krylov="gmres", iters=31),
        # a ragged field, half-precision factor storage
        dict(name="step_97x83x29_fp16s", kind="step", **_grid(97, 83, 29, 12, 10, 1, 1), precision="fp16s", restart=30,
             sigma=1.0, local="colsum", krylov="gmres", iters=33),
        # a Newton step of half a million cells in full precision
        dict(name="step_128x128x32_fp64", kind="step", **_grid(128, 128, 32, 16, 16, 1, 2), precision="fp64",
             restart=30, sigma=2.0, local="colsum", krylov="gmres", iters=42),
        # the headline: a Newton step of a million cells with FP32 factors
        dict(name="step_128x128x64_fp32", kind="step", **_grid(128, 128, 64, 16, 16, 2, 2), precision="fp32",
             restart=30, sigma=2.0, local="colsum", krylov="gmres", iters=80),
        # nested factorisation as the local solver (boxes without lumps)
        dict(name="step_64x64x32_nf_fp32", kind="step", **_grid(64, 64, 32, 8, 8, 1, 2), precision="fp32", restart=30,
             sigma=1.0, local="nf_colsum", krylov="gmres", iters=8),
        # many independent small and middling systems in the same launches
        dict(name="batch_48_fp32", kind="batch", count=48, base=1000, precision="fp32", restart=20, iters=30),
        # requests of several sizes through the serving loop, host arrays in and out
        dict(name="serve_12_fp32", kind="serve", count=12, base=77, cells=40000, precision="fp32", restart=30,
             iters=35),
        # the operators alone: a caller's own Krylov method, or a check of a residual
        dict(name="spmv_61x47x53", kind="spmv", **_grid(61, 47, 53, 1, 1, 1, 0), precision="fp64", restart=30,
             sigma=1.0, local="colsum", krylov="gmres", iters=1),
        dict(name="apply_75x50x31_fp64", kind="apply", **_grid(75, 50, 31, 9, 6, 1, 1), precision="fp64", restart=30,
             sigma=1.0, local="colsum", krylov="gmres", iters=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "step", "step", "step", "batch", "serve", "spmv", "apply"])
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16s"])
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 4, 60), base=rng.randrange(2000, 9000),
                    precision=rng.choice(["fp32", "fp64"]), restart=rng.choice([20, 30]), iters=30)
    if kind == "serve":
        return dict(kind=kind, count=rng.randrange(3, 17), base=rng.randrange(2000, 9000),
                    cells=_log_int(rng, 4000, 60000), precision=rng.choice(["fp32", "fp64"]), restart=30, iters=35)
    # cells log-uniform, flat fields as in the workloads (the vertical extent a quarter to a half)
    cells = _log_int(rng, 400, 400000 if kind in ("spmv", "step") else 150000)
    flat = rng.uniform(0.2, 0.6)
    nx = max(4, int(round((cells / flat) ** (1 / 3) * rng.uniform(0.8, 1.25))))
    nz = max(2, int(round(flat * (cells / flat) ** (1 / 3))))
    ny = max(4, int(round(cells / (nx * nz))))
    side = rng.uniform(6.0, 10.0)
    px, py = (min(16, max(1, int(round(n / side)))) for n in (nx, ny))
    pz = 2 if nz > 32 else 1
    local, krylov = "colsum", "gmres"
    if kind in ("step", "solve") and rng.random() < 0.15 and precision != "fp16s":
        local = "nf_colsum"
    elif kind == "solve" and precision == "fp64" and cells < 12000 and rng.random() < 0.3:
        krylov = "orthomin"
    if krylov == "orthomin":
        px, py, pz = min(px, 3), min(py, 3), 1
    return dict(kind=kind, **_grid(nx, ny, nz, px, py, pz, rng.choice([1, 1, 2])), precision=precision,
                restart=30 if krylov == "orthomin" else rng.choice([20, 30]), sigma=1.0, local=local, krylov=krylov,
                iters=40)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
_OFFS = ((-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 1), (0, 1, 0), (1, 0, 0))  # (y, x, z) of the six neighbours


def _sides(o):
    """Index tuples over [ny, nx, nz]: the cells that have the neighbour at offset o, and those neighbours."""
    a = tuple(slice(1, None) if d < 0 else slice(None, -1) if d > 0 else slice(None) for d in o)
    b = tuple(slice(None, -1) if d < 0 else slice(1, None) if d > 0 else slice(None) for d in o)
    return a, b


class System:
    """A BSR 3x3 system: host row_ptr / col_idx, values [nnzb, 3, 3] and b [3 n] on the GPU."""

    def __init__(self, nx, ny, nz, seed, sigma):
        self.nx, self.ny, self.nz = nx, ny, nz
        dev = torch.device("cuda")
        g = torch.Generator(dev).manual_seed(seed)
        f64 = dict(dtype=torch.float64, device=dev)
        n = nx * ny * nz
        shape = (ny, nx, nz)

        def uniform(lo, hi, *size):
            return lo + (hi - lo) * torch.rand(*size, generator=g, **f64)

        kx = 100.0 * torch.exp(0.8 * sigma * torch.randn(nz, generator=g, **f64) +
                               0.6 * torch.randn(*shape, generator=g, **f64))
        fy = torch.arange(ny, **f64)[:, None, None] / max(1, ny - 1)
        fx = torch.arange(nx, **f64)[None, :, None] / max(1, nx - 1)
        phi = 1.0 - 0.5 * (fx + fy) + 0.1 * uniform(-1.0, 1.0, *shape)
        cell = torch.arange(n, device=dev).view(shape)
        vals = torch.zeros(*shape, 7, 3, 3, **f64)
        cols = torch.zeros(*shape, 7, dtype=torch.int64, device=dev)
        valid = torch.zeros(*shape, 7, dtype=torch.bool, device=dev)
        tsum = torch.zeros(*shape, **f64)
        diag = torch.zeros(*shape, 3, 3, **f64)
        lo = torch.tensor([0.8, -0.2, -0.2, 0.2, 0.5, -0.1, 0.2, -0.1, 0.5], **f64).view(3, 3)
        hi = torch.tensor([1.2, 0.2, 0.2, 0.6, 1.0, 0.1, 0.6, 0.1, 1.0], **f64).view(3, 3)
        for d, o in enumerate(_OFFS):
            s = d if d < 3 else d + 1  # the diagonal is slot 3: columns ascend within a row
            a, b = _sides(o)
            k = kx * (0.1 if o[2] else 1.0)
            t = (5000.0 if o[2] else 2.0) * 2.0 * k[a] * k[b] / (k[a] + k[b])
            tsum[a] += t
            m = lo + (hi - lo) * torch.rand(*t.shape, 3, 3, generator=g, **f64)
            m[..., 1:, 1:] *= (phi[b] > phi[a])[..., None, None]  # saturation terms only from upstream
            blk = -t[..., None, None] * m
            diag[b] -= blk  # conservative: the block columns add up to the accumulation
            vals[(*a, s)] = blk
            cols[(*a, s)] = cell[b]
            valid[(*a, s)] = True
        acc = uniform(0.5, 1.5, *shape, 3) * torch.tensor([1e-3, 0.5, 0.5], **f64) * tsum[..., None]
        diag += torch.diag_embed(acc)
        well = torch.zeros(*shape, dtype=torch.bool, device=dev)
        well[0, 0] = True
        well[-1, -1] = True
        diag[well] += 200.0 * torch.eye(3, **f64)
        vals[..., 3, :, :] = diag
        cols[..., 3] = cell
        valid[..., 3] = True
        valid = valid.view(n, 7)
        self.vals = vals.view(n, 7, 3, 3)[valid].contiguous()
        self.col_idx = cols.view(n, 7)[valid].to(torch.int32).cpu().numpy()
        self.row_ptr = np.zeros(n + 1, dtype=np.int32)
        np.cumsum(valid.sum(1).cpu().numpy(), out=self.row_ptr[1:])
        self.b = uniform(-1.0, 1.0, 3 * n)

    def to_host(self):
        self.vals, self.b = self.vals.cpu().numpy(), self.b.cpu().numpy()
        return self


def _system(case, seed):
    return System(case["nx"], case["ny"], case["nz"], seed, case["sigma"])


def _batch_grids(case):
    """(8, 8, 4) * s with s log-uniform on [1, 5], as the batched workload has them."""
    rng = np.random.default_rng(case["base"])
    grids = []
    for _ in range(case["count"]):
        s = math.exp(rng.uniform(0.0, math.log(5.0)))
        nx, nz = max(2, round(8 * s)), max(2, round(4 * s))
        p = min(8, max(2, round(nx / 6)))
        grids.append((nx, nx, nz, p, p, 1))
    return grids


def _serve_grids(case):
    """Cells log-uniform up to case["cells"], boxes of about eight cells, as the served stream has them."""
    rng = np.random.default_rng(case["base"])
    grids = []
    for _ in range(case["count"]):
        n = math.exp(rng.uniform(math.log(2000), math.log(case["cells"])))
        nx = max(2, round((2 * n) ** (1 / 3)))
        nz = max(2, round(n / nx ** 2))
        p = min(16, max(1, round(nx / 8)))
        grids.append((nx, nx, nz, p, p, 2 if nz > 32 else 1))
    return grids


def _solver(case, system, grid, overlap):
    local = case.get("local", "colsum")
    s = asm2.Solver(precision=case["precision"], restart=case["restart"], local_solver=local,
                    krylov=case.get("krylov", "gmres"))
    s.set_grid(*grid[:3])
    s.set_matrix(system.row_ptr, system.col_idx, system.vals)
    if local == "nf_colsum":
        s.set_partition(*grid[3:], overlap, 0, (2, 2, 2), "none")
    else:
        s.set_partition(*grid[3:], overlap)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        grids = _batch_grids(case)
        systems = [System(*g[:3], seed * 1000 + i, 1.0) for i, g in enumerate(grids)]
        solvers = [_solver(case, s, g, 1) for s, g in zip(systems, grids)]
        for s in solvers:
            s.factor()
        return dict(kind=kind, solvers=solvers, b=[s.b for s in systems])
    if kind == "serve":
        grids = _serve_grids(case)
        systems = [System(*g[:3], seed * 1000 + i, 1.0).to_host() for i, g in enumerate(grids)]
        server = asm2.Server(precision=case["precision"], restart=case["restart"], max_cached=64)
        return dict(kind=kind, server=server, systems=systems, parts=[g[3:] for g in grids])
    system = _system(case, seed)
    grid = tuple(case[k] for k in ("nx", "ny", "nz", "px", "py", "pz"))
    solver = _solver(case, system, grid, case["overlap"])
    if kind != "spmv":
        solver.factor()
    return dict(kind=kind, solver=solver, vals=system.vals, b=system.b)


def run(state):
    kind = state["kind"]
    if kind == "spmv":
        return state["solver"].spmv(state["b"])
    if kind == "apply":
        return state["solver"].apply(state["b"])
    if kind == "batch":
        xs, infos = asm2.solve_batch(state["solvers"], state["b"], rtol=RTOL, max_iter=MAX_ITER)
        return {"x": xs, "iterations": np.array([i["iterations"] for i in infos])}
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(s, s.b, partition=p, overlap=1, rtol=RTOL, max_iter=MAX_ITER)
                   for s, p in zip(state["systems"], state["parts"])]
        done = {}
        while len(done) < len(tickets):
            server.progress(4)
            for t in tickets:
                if t not in done and (r := server.result(t)) is not None:
                    done[t] = r
        return {"x": [done[t][0] for t in tickets],
                "iterations": np.array([done[t][1]["iterations"] for t in tickets])}
    solver = state["solver"]
    if kind == "step":
        solver.update_values(state["vals"])
        solver.factor()
    x, info = solver.solve(state["b"], rtol=RTOL, max_iter=MAX_ITER)
    return {"x": x, "iterations": info["iterations"]}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _blocks(nx, ny, nz):
    n = nx * ny * nz
    return 7 * n - 2 * (nx * ny + ny * nz + nx * nz)


def _solve_work(grid, overlap, precision, restart, iters, step, apply_only=False):
    """Fine rows only (the lumps add a few percent): every factor block, the matrix and the basis
    vectors once per iteration, and for a step the matrix in and the factors out once."""
    nx, ny, nz, px, py, pz = grid
    n, nnzb = nx * ny * nz, _blocks(nx, ny, nz)

    def spans(m, p):
        return [min(m, m * (t + 1) // p + overlap) - max(0, m * t // p - overlap) for t in range(p)]

    local = sum(_blocks(x, y, z) for x in spans(nx, px) for y in spans(ny, py) for z in spans(nz, pz))
    w = {"fp64": 8, "fp32": 4, "fp16s": 2}[precision]
    apply_b, apply_f = local * (9 * w + 4) + 48 * n, 18 * local
    if apply_only:
        return apply_b, apply_f
    spmv_b, spmv_f = nnzb * 76 + 48 * n, 18 * nnzb
    j = min(iters, restart) / 2  # mean number of basis vectors of an Arnoldi step
    vec_b, vec_f = 24 * n * (j + 3), 12 * n * (j + 1)
    b, f = iters * (apply_b + spmv_b + vec_b), iters * (apply_f + spmv_f + vec_f)
    if step:
        b, f = b + nnzb * 72 + local * 9 * w, f + 54 * local
    return b, f


def work(case):
    kind = case["kind"]
    if kind == "spmv":
        n, nnzb = case["nx"] * case["ny"] * case["nz"], _blocks(case["nx"], case["ny"], case["nz"])
        return {"bytes": nnzb * 76 + 48 * n, "flops": 18 * nnzb}
    if kind in ("batch", "serve"):
        grids, step = (_batch_grids(case), False) if kind == "batch" else (_serve_grids(case), True)
        each = [_solve_work(g, 1, case["precision"], case["restart"], case["iters"], step) for g in grids]
    else:
        grid = tuple(case[k] for k in ("nx", "ny", "nz", "px", "py", "pz"))
        each = [_solve_work(grid, case["overlap"], case["precision"], case["restart"], case["iters"], kind == "step",
                            kind == "apply")]
    return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}


# ---------------------------------------------------------------------------------------------
# what a pass returns, in 64 bits and without the package
# ---------------------------------------------------------------------------------------------
def _product(s, x):
    rows = torch.repeat_interleave(torch.arange(len(s.row_ptr) - 1, device=x.device),
                                   torch.from_numpy(np.diff(s.row_ptr)).to(x.device).long())
    cols = torch.from_numpy(s.col_idx).to(x.device).long()
    y = torch.zeros(len(s.row_ptr) - 1, 3, dtype=torch.float64, device=x.device)
    y.index_add_(0, rows, torch.einsum("eij,ej->ei", s.vals, x.view(-1, 3)[cols]))
    return y.view(-1)


def _solution(s):
    """A^{-1} b by block elimination over the xz planes (the matrix is block tridiagonal in y), with
    two steps of refinement; None where the planes are too large for that."""
    m, planes = 3 * s.nx * s.nz, s.ny
    if 8 / 3 * m ** 3 * planes > 4e12 or 8 * m * m * planes > 4e10:
        return None
    dev = s.b.device
    rows = np.repeat(np.arange(len(s.row_ptr) - 1), np.diff(s.row_ptr))
    cells = s.nx * s.nz
    r, c = (torch.from_numpy(v).to(dev).long() for v in (rows, s.col_idx.astype(np.int64)))

    def block(j, k):
        e = ((r // cells == j) & (c // cells == k)).nonzero()[:, 0]
        out = torch.zeros(cells, 3, cells, 3, dtype=torch.float64, device=dev)
        out[r[e] - j * cells, :, c[e] - k * cells, :] = s.vals[e]
        return out.view(m, m)

    lus, gains = [], []
    for j in range(planes):
        d = block(j, j)
        if j:
            gain = torch.linalg.solve(d_prev.T, block(j, j - 1).T).T  # lower block times the inverse before it
            d = d - gain @ block(j - 1, j)
            gains.append(gain)
        lus.append(torch.linalg.lu_factor(d))
        d_prev = d

    def solve(b):
        y = [v for v in b.view(planes, m).clone()]
        for j in range(1, planes):
            y[j] = y[j] - gains[j - 1] @ y[j - 1]
        for j in reversed(range(planes)):
            if j + 1 < planes:
                y[j] = y[j] - block(j, j + 1) @ y[j + 1]
            y[j] = torch.linalg.lu_solve(*lus[j], y[j][:, None])[:, 0]
        return torch.cat(y)

    x = solve(s.b)
    for _ in range(2):
        x = x + solve(s.b - _product(s, x))
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":  # incomplete factorisations of coarsened matrices, row by row: minutes in numpy
        return None
    if kind in ("batch", "serve"):  # the systems of up to a few thousand cells, the others too slow in all
        grids = _batch_grids(case) if kind == "batch" else _serve_grids(case)
        xs = [_solution(System(*g[:3], seed * 1000 + i, 1.0)) if g[0] * g[1] * g[2] <= 4000 else None
              for i, g in enumerate(grids)]
        return {"x": xs, "iterations": None}
    system = _system(case, seed)
    if kind == "spmv":
        return _product(system, system.b)
    x = _solution(system)
    return None if x is None else {"x": x, "iterations": None}
