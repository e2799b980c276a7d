"""The size of work units (csrc/pic_balance.cpp), compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "pic_balance.cpp"
extern "C" {
int64_t t_min(const int64_t* np, int64_t nb, int nw) { return pic::min_unit_particles(np, nb, nw); }
int64_t t_share(int64_t nu, int ctas, int64_t np) { return pic::unit_share(nu, ctas, np); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("units")
    (d / "shim.cpp").write_text(SHIM)
    so = d / "shim.so"
    csrc = os.path.join(ROOT, "paper_2104_11385_gb300", "csrc")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", csrc, str(d / "shim.cpp"), "-o", str(so)])
    L = ctypes.CDLL(str(so))
    L.t_min.restype = L.t_share.restype = ctypes.c_int64
    return L


def least(lib, np_box, nw):
    a = np.ascontiguousarray(np_box, np.int64)
    return lib.t_min(a.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(a.size), nw)


def units(np_box, m):
    return int(np.maximum(1, np.asarray(np_box) // m).sum())


@pytest.mark.parametrize("nw", [1, 152, 304])
@pytest.mark.parametrize("boxes,heavy", [(8, 8), (16, 4), (64, 32), (64, 64), (512, 16), (4096, 64)])
@pytest.mark.parametrize("total", [0, 1, 1000, 40000, 131072, 300000, 1300000, 9000000, 600000000])
def test_between_256_and_4096(lib, nw, boxes, heavy, total):
    counts = np.zeros(boxes, np.int64)
    counts[:heavy] = total // heavy
    m = least(lib, counts, nw)
    n = int(counts.sum())
    assert 256 <= m <= 4096
    if n >= 4096 * nw:
        assert m == min(4096, n // (4 * nw))
    elif units(counts, 1024) <= nw:
        # as many units as fit one per worker: the next finer cut would not
        assert units(counts, m) <= nw
        assert m == 256 or units(counts, m - 1) > nw
    else:
        assert m == max(256, min(1024, n // nw))


def test_few_boxes_leave_no_worker_idle(lib):
    """64 boxes, half of them empty, 4096 particles in the others, 304 workers"""
    counts = np.where(np.arange(64) % 2 == 0, 4096, 0)
    assert units(counts, least(lib, counts, 304)) >= 272


@pytest.mark.parametrize("nu,ctas,np_,want", [(8, 152, 32768, 16), (8, 152, 400, 1), (8, 152, 0, 1), (76, 152, 10 ** 6, 2),
                                              (77, 152, 10 ** 6, 1), (1, 304, 10 ** 6, 304), (0, 304, 10, 1)])
def test_share(lib, nu, ctas, np_, want):
    assert lib.t_share(ctypes.c_int64(nu), ctas, ctypes.c_int64(np_)) == want
