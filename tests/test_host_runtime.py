"""The host runtime (``csrc/api.cpp``) on the CPU, with a stand-in for the CUDA runtime and the kernels
(``tests/fake_device.cpp``): what it copies, keeps and accounts for, not what the kernels compute."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

from paper_1401_7227_gb300 import asm2, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1401_7227_gb300", "csrc")


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    # entry points that no test here reaches stay undefined (bound lazily)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,lazy",
                    f"-I{os.path.join(ROOT, 'include')}", f"-I{CSRC}", f"-I{cuda_inc}", os.path.join(CSRC, "api.cpp"),
                    os.path.join(CSRC, "symbolic.cpp"), os.path.join(ROOT, "tests", "fake_device.cpp"), "-o", out,
                    "-lpthread"], check=True)
    return out


@pytest.fixture
def fake(fake_path, monkeypatch):
    """The package's classes on the fake device; its counters are reset."""
    lib = C.CDLL(fake_path, mode=os.RTLD_LAZY)
    lib.fk_calls.restype = lib.fk_live_bytes.restype = lib.fk_h2d_bytes.restype = C.c_longlong
    monkeypatch.setattr(asm2._build, "LIB", fake_path)
    monkeypatch.setattr(asm2, "_lib", None)
    monkeypatch.setattr(asm2.C, "CDLL", lambda path: lib)
    lib.fk_reset(152)
    asm2.load()
    yield lib
    lib.fk_reset(152)


def make_solver(s, part, **opt):
    sol = asm2.Solver(stream=0, **opt)
    sol.set_grid(s.nx, s.ny, s.nz)
    sol.set_matrix(s.row_ptr, s.col_idx, s.vals)
    sol.set_partition(*part, 1)
    sol.factor()
    return sol


def test_the_words_a_solve_starts_from_outlive_their_copies(fake):
    """Control words and tolerance of each system are copied without a wait: their source must not be a variable of
    a function that returns before the copy is sure to have been made."""
    systems = [synth.grid_jacobian(6, 6, 3, k) for k in range(3)]
    sols = [make_solver(s, (2, 2, 1)) for s in systems]
    fake.fk_reset(152)
    sols[0].solve(systems[0].b, 1e-8, 3)
    asm2.solve_batch(sols, [s.b for s in systems], rtol=1e-8, max_iter=3)
    assert fake.fk_calls(b"finish") > 0
    assert fake.fk_late_stack_copies() == 0
    for sol in sols:
        sol.close()


def serve(srv, tickets):
    """Runs the server until every ticket has its result; the largest number of systems in flight."""
    most, left = 0, list(tickets)
    for _ in range(10000):
        most = max(most, srv.progress(1)[0])
        left = [t for t in left if srv.result(t) is None]
        if not left:
            return most
    raise AssertionError("requests did not finish")


@pytest.mark.parametrize("kept", [0, 1, 2])
def test_server_accounts_for_factor_streams_uploaded_after_admission(fake, kept):
    """On 2 SMs one system of four subdomains applies by lane, two together by rows, whose stream is uploaded when
    the second one joins.  What is resident at the end is what the kept systems hold on the device."""
    fake.fk_reset(2)
    systems = [synth.grid_jacobian(10, 10, 5, k) for k in range(4)]
    empty = fake.fk_live_bytes()
    srv = asm2.Server(precision="fp32", stream=0, max_cached=kept)
    serve(srv, [srv.submit(s, s.b, partition=(2, 2, 1), max_iter=4, matrix_key=k) for k, s in enumerate(systems)])
    assert fake.fk_calls(b"apply_rows") > 0
    live, st = fake.fk_live_bytes() - empty, srv.stats()
    srv.close()
    assert st["completed"] == 4 and st["evictions"] == (4 - kept if kept else 0)
    tables = 64 << 10  # the server's own work-item tables
    assert live - tables <= st["resident_bytes"] <= live
    assert fake.fk_live_bytes() == empty


def test_server_admits_within_its_budget_when_streams_are_uploaded_later(fake):
    """On 2 SMs two systems of four subdomains apply by lane and three by rows.  A budget for three with one stream
    each, but not with both: two at a time."""
    fake.fk_reset(2)
    systems = [synth.grid_jacobian(20, 20, 8, k) for k in range(3)]

    def resident(n, budget=0):
        srv = asm2.Server(precision="fp32", stream=0, max_cached=n, hbm_budget=budget)
        most = serve(srv, [srv.submit(s, s.b, partition=(2, 2, 1), max_iter=40, matrix_key=k)
                           for k, s in enumerate(systems[:n])])
        size = srv.stats()["resident_bytes"]
        srv.close()
        return most, size

    (_, by_lane), (most, both) = resident(1), resident(3)
    rows = both // 3 - by_lane
    assert most == 3 and rows > 0
    need = 3200 * 6144  # the server's estimate for a new system with one stream
    assert resident(3, 2 * by_lane + need + rows // 2)[0] == 2
    assert resident(3, both + need)[0] == 3


def test_a_new_factorisation_packs_the_one_stream_in_use(fake):
    """On 2 SMs one system applies by lane and three together by rows.  Each factorisation fills the stream that the
    last apply read; the other is filled when an apply needs it again, once."""
    fake.fk_reset(2)
    systems = [synth.grid_jacobian(10, 10, 5, k) for k in range(3)]
    sols = [make_solver(s, (2, 2, 1), precision="fp32") for s in systems]

    def packs():
        by_rows, by_lane = fake.fk_calls(b"pack"), fake.fk_calls(b"pack_lanes")
        fake.fk_reset(2)
        return by_rows, by_lane

    def new_values():
        for s, sol in zip(systems, sols):
            sol.update_values(s.vals)
            sol.factor()

    def batch():
        asm2.solve_batch(sols, [s.b for s in systems], max_iter=3)

    # (two launches fill a stream: fine rows, lump rows)
    assert packs() == (0, 6)                       # new systems: by lane
    batch()
    assert fake.fk_calls(b"apply_rows") > 0 and packs() == (6, 0)
    new_values()
    batch()
    assert packs() == (6, 0)
    sols[0].solve(systems[0].b, max_iter=3)
    assert fake.fk_calls(b"apply_lanes") > 0 and packs() == (0, 2)
    sols[0].solve(systems[0].b, max_iter=3)
    batch()
    assert packs() == (0, 0)                       # both hold the current factors
    new_values()
    assert packs() == (6, 0)
    for sol in sols:
        sol.close()


@pytest.mark.parametrize("precision,nz,form", [("fp32", 8, "lanes"),    # two CTAs per SM: one wave
                                               ("fp32", 40, "rows"),    # one by lane, two by rows
                                               ("fp16s", 44, "rows"),
                                               ("fp32", 64, "lanes"),   # one either way
                                               ("fp64", 40, "lanes")])
def test_a_second_wave_by_lane_gives_way_to_one_by_rows(fake, precision, nz, form):
    """Four subdomains on 3 SMs, with more local rows the taller the boxes."""
    fake.fk_reset(3)
    s = synth.grid_jacobian(18, 18, nz, 1)
    sol = make_solver(s, (2, 2, 1), precision=precision)
    sol.solve(s.b, max_iter=3)
    other = "rows" if form == "lanes" else "lanes"
    assert fake.fk_calls(f"apply_{form}".encode()) > 0 and fake.fk_calls(f"apply_{other}".encode()) == 0
    assert fake.fk_calls(b"pack_lanes") == (2 if form == "lanes" else 0)
    sol.close()


def test_a_stream_uploaded_in_a_solve_goes_without_its_values(fake):
    """On 2 SMs three systems of four subdomains apply by rows, which no one of them does alone: the first solve
    uploads their streams and pack lists, the second nothing of the kind."""
    fake.fk_reset(2)
    systems = [synth.grid_jacobian(16, 16, 8, k) for k in range(3)]
    sols = [make_solver(s, (2, 2, 1)) for s in systems]
    sent = []
    for _ in range(2):
        fake.fk_reset(2)
        asm2.solve_batch(sols, [s.b for s in systems], max_iter=3)
        sent.append(fake.fk_h2d_bytes())
    assert fake.fk_calls(b"apply_rows") > 0
    stats = sols[0].stats()
    lists, streams = 3 * 12 * stats["local_blocks"], 3 * stats["factor_bytes"]
    assert lists < sent[0] - sent[1] < lists + streams // 4
    sols.append(make_solver(systems[0], (2, 2, 1)))
    fake.fk_reset(2)
    asm2.solve_batch(sols, [s.b for s in systems] + [systems[0].b], max_iter=3)
    assert fake.fk_calls(b"place") == 1  # (one system had no stream by rows yet)
    for sol in sols:
        sol.close()


def test_factor_bytes_are_those_of_the_stream_the_apply_reads(fake):
    """By lane every packet has ten positions and a table entry, so that stream is the larger one."""
    s = synth.grid_jacobian(16, 16, 8, 1)
    sol = make_solver(s, (2, 2, 1), precision="fp64")
    by_lane = sol.stats()["factor_bytes"]
    sol.set_tuning(apply_smem=0)
    by_rows = sol.stats()["factor_bytes"]
    assert by_rows > 72 * sol.stats()["local_blocks"] and by_lane > 1.05 * by_rows
    sol.close()
