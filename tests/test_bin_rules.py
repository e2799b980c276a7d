"""Which of the binning's kernels takes an input (csrc/pic_bin.h), compiled for
the host, and their results on the GPU on both sides of each limit."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <stdint.h>
#include <string>
typedef int cudaError_t;
typedef void* cudaStream_t;
#include "../../include/pic_api.h"
#include "pic_bin.h"
extern "C" {
int t_count(int nb, long long np, int ctas) { return bin_count_in_shared(nb, np, ctas); }
int t_scatter(int nb, long long np, int ctas) { return bin_scatter_in_shared(nb, np, ctas); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("bin")
    (d / "cuda_runtime.h").write_text("#pragma once\n")
    (d / "shim.cpp").write_text(SHIM)
    so = d / "shim.so"
    csrc = os.path.join(ROOT, "paper_2104_11385_gb300", "csrc")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(d), "-I", csrc, str(d / "shim.cpp"), "-o",
                           str(so)])
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("boxes", [1, 8, 64, 512, 8192, 8193])
@pytest.mark.parametrize("npart", [1, 10001, 100000, 262143, 262144, 1000000, 16777216])
def test_scatter_has_chunks_for_the_chip(lib, boxes, npart):
    f = lambda g: bool(g(boxes, ctypes.c_longlong(npart), 304))
    assert f(lib.t_count) == (boxes <= 8192 and npart >= 4 * 304 * boxes)
    assert f(lib.t_scatter) == (f(lib.t_count) and npart >= 262144)


@pytest.mark.gpu
@pytest.mark.parametrize("boxes,npart", [(1, 10001), (1, 262143), (1, 262144), (8, 30000), (64, 262143), (64, 262144),
                                         (8192, 9961471), (8192, 9961472), (8193, 9961472)])
def test_results_on_both_sides(boxes, npart):
    import torch
    from paper_2104_11385_gb300 import sim as S
    n, box, d = (4, 1, 4 * boxes), (4, 1, 4), 0.3
    g = torch.Generator(device="cuda")
    g.manual_seed(npart)
    x = torch.rand(npart, dtype=torch.float64, device="cuda", generator=g) * (4 * d * 0.999)
    z = torch.rand(npart, dtype=torch.float64, device="cuda", generator=g) * (4 * boxes * d * 0.999)
    off = torch.empty(boxes + 1, dtype=torch.int64, device="cuda")
    perm = torch.empty(npart, dtype=torch.int64, device="cuda")
    S.bin_particles(2, n, box, (d, 1.0, d), x, None, z, off, perm)
    torch.cuda.synchronize()
    want = torch.floor(z / d).to(torch.int64) // 4
    counts = torch.bincount(want, minlength=boxes)
    assert torch.equal(off[1:], torch.cumsum(counts, 0)) and int(off[0]) == 0
    assert torch.equal(want[perm], torch.repeat_interleave(torch.arange(boxes, device="cuda"), counts))
    assert torch.equal(torch.sort(perm)[0], torch.arange(npart, device="cuda"))
