"""The factor stream by lane (``csrc/packets.h``) against the stream by rows, on the CPU
(``tests/packets_check.cpp``): every chunk holds the same rows with the same operands, values and D^{-1} in the
same order and the same sharing of a row over lanes, every value has a place of its own, and what a row does
not have reads the zero row.  So both layouts give the same bits."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle as O
from hub_rows import hub_system
from paper_1401_7227_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1401_7227_gb300", "csrc")

GEOMS = {
    "cfg1": O.Geometry(10, 10, 5, 2, 2, 1, ov=1),
    "ragged": O.Geometry(9, 7, 6, 3, 2, 2, ov=1, near_width=1, cnear=(2, 3, 2)),
    "cfar": O.Geometry(12, 6, 5, 3, 1, 1, ov=2, near_width=2, cnear=(3, 2, 2), far_mode=2, cfar=(4, 3, 5)),
    "no_lumps": O.Geometry(6, 6, 3, 3, 3, 1, ov=0, near_width=0, far_mode=0),
    "more_lumps_than_rows": O.Geometry(8, 8, 4, 8, 8, 1, ov=0, near_width=2),
    "one_cell_boxes": O.Geometry(3, 3, 3, 3, 3, 3, ov=0, near_width=1, cnear=(1, 1, 1)),
    "long_lump_rows": O.Geometry(32, 32, 64, 4, 4, 1, ov=1),  # rows of ~130 blocks
    "levels_split_over_chunks": O.Geometry(40, 40, 8, 1, 1, 1, ov=0, near_width=0, far_mode=0),
}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("pk") / "libpk.so")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", f"-I{os.path.join(ROOT, 'include')}", f"-I{CSRC}",
                    f"-I{cuda_inc}", os.path.join(CSRC, "symbolic.cpp"), os.path.join(ROOT, "tests", "packets_check.cpp"),
                    "-o", out, "-lpthread"], check=True)
    return C.CDLL(out)


@pytest.mark.parametrize("name,prec,chunk", [(n, p, 0) for n in GEOMS for p in (0, 1, 2)] +
                         [("cfg1", 0, 12288), ("long_lump_rows", 1, 8192), ("levels_split_over_chunks", 0, 8192)])
def test_same_rows_by_lane(lib, name, prec, chunk):
    g = GEOMS[name]
    s = synth.grid_jacobian(g.nx, g.ny, g.nz, 3)
    geo = np.array([g.nx, g.ny, g.nz, g.px, g.py, g.pz, g.ov, g.near_width, *g.cnear, g.far_mode, *g.cfar], dtype=np.int32)
    rp, ci = (np.ascontiguousarray(a, dtype=np.int32) for a in (s.row_ptr, s.col_idx))
    err = C.create_string_buffer(256)
    bad = lib.pk_check(geo.ctypes.data_as(C.c_void_p), s.n_cells, s.nnzb, rp.ctypes.data_as(C.c_void_p),
                       ci.ctypes.data_as(C.c_void_p), prec, chunk, err, 256)
    assert bad == 0, err.value.decode()


@pytest.mark.parametrize("lower,prec", [(n, p) for n in (254, 255, 256, 300) for p in (0, 1, 2)] + [(512, 1), (512, 2)])
def test_rows_of_more_entries_than_a_packet_counts(lib, lower, prec):
    """A packet's kind word has eight bits for its entries: up to 255 the rows are there by lane, beyond it there is
    no stream by lane and the handle applies by rows."""
    s = hub_system(10, 10, 6, 3, lower)
    geo = np.array([10, 10, 6, 1, 1, 1, 0, 0, 1, 1, 1, 0, 1, 1, 1], dtype=np.int32)
    rp, ci = (np.ascontiguousarray(a, dtype=np.int32) for a in (s.row_ptr, s.col_idx))
    err = C.create_string_buffer(256)
    bad = lib.pk_check(geo.ctypes.data_as(C.c_void_p), s.n_cells, s.nnzb, rp.ctypes.data_as(C.c_void_p),
                       ci.ctypes.data_as(C.c_void_p), prec, 0, err, 256)
    assert (bad, err.value.decode()) == ((0, "") if lower <= 255 else (1, "chunk count"))


@pytest.mark.parametrize("slots", [2, 3, 5, 8])
def test_an_expired_wait_drains_the_copies_in_flight_and_no_others(lib, slots):
    """A wait for a copy that was never issued would poll until its own limit."""
    for n in (1, 2, 3, 7, 20):
        for expire in range(n):
            assert lib.pk_drain_check(slots, n, expire) == 0, (n, expire)


@pytest.mark.parametrize("name", GEOMS)
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_no_packets_where_the_rows_cannot_fit_a_cta(lib, name, prec):
    """The rule that spares the analysis the packets of boxes too large for a CTA's shared memory leaves out no system
    whose subdomains fit, whatever the limit, and keeps none whose largest box alone does not."""
    g = GEOMS[name]
    s = synth.grid_jacobian(g.nx, g.ny, g.nz, 3)
    geo = np.array([g.nx, g.ny, g.nz, g.px, g.py, g.pz, g.ov, g.near_width, *g.cnear, g.far_mode, *g.cfar], dtype=np.int32)
    rp, ci = (np.ascontiguousarray(a, dtype=np.int32) for a in (s.row_ptr, s.col_idx))
    fits, row = C.c_int(), 24 if prec == 0 else 16
    p = lambda a: a.ctypes.data_as(C.c_void_p)
    spans = [max(min(n, n * (t + 1) // q + g.ov) - max(0, n * t // q - g.ov) for t in range(q))
             for n, q in ((g.nx, g.px), (g.ny, g.py), (g.nz, g.pz))]
    box = int(np.prod(spans)) * row
    for smem in (box - 1, box, box + 32, 2 * box, 40 * box, 232448):
        want = lib.pk_wanted(p(geo), s.n_cells, s.nnzb, p(rp), p(ci), prec, 152, smem, C.byref(fits))
        assert want == (1 if smem >= box else 0)
        assert want == 1 or fits.value == 0
    assert lib.pk_wanted(p(geo), s.n_cells, s.nnzb, p(rp), p(ci), prec, (g.px * g.py * g.pz - 1) // 2, 232448, C.byref(fits)) == 0
