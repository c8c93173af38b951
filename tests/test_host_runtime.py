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
    lib.fk_calls.restype = lib.fk_live_bytes.restype = C.c_longlong
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
