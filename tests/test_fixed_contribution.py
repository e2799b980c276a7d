"""Current contributions of the fixed-point deposit (csrc/pic_fix.cuh), compiled
for the host: amplitude x weight against exact rationals, over the whole range
of weights, and the weights of a particle on a node."""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

from test_fixed_point import ROOT, SHIM, Q, ll

MORE = r"""
extern "C" {
int t_contribution(double c, double q, long long p, long long T, unsigned long long* m, int* e, double* v) {
    const Amp a = amp_scale(amp_mul(amp_of(c), amp_of(q)), p);
    *m = a.m; *e = (int)(((a.es + (1024u << 20)) >> 20) & 0x7FFu) - 1024;
    return contribution(a, T, *v);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("contribution")
    (d / "cuda_runtime.h").write_text("#pragma once\n")
    (d / "shim.cpp").write_text(SHIM + MORE)
    so = d / "shim.so"
    csrc = os.path.join(ROOT, "paper_2104_11385_gb300", "csrc")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(d), "-I", csrc, str(d / "shim.cpp"), "-o",
                           str(so)])
    return ctypes.CDLL(str(so))


def contribution(lib, c, q, p, T):
    m, e, v = ctypes.c_ulonglong(), ctypes.c_int(), ctypes.c_double()
    some = lib.t_contribution(ctypes.c_double(c), ctypes.c_double(q), ll(p), ll(T), *map(ctypes.byref, (m, e, v)))
    return m.value, e.value, v.value if some else 0.0


def test_every_weight(lib):
    r = np.random.default_rng(21)
    weights = [Q, Q - 1, 1, 2, 3] + [int(r.integers(1 << k, 2 << k)) for k in range(62) for _ in range(8)]
    for T in weights:
        c, q = (float(np.ldexp(r.uniform(0.5, 1), int(r.integers(-20, 20)))) for _ in range(2))
        p = int(r.integers(1, Q)) >> int(r.integers(0, 40))
        sign = -1 if r.random() < 0.5 else 1
        m, e, v = contribution(lib, c, q, sign * p, T)
        assert m >= 1 << 58
        amp = Fr(m) * Fr(2) ** e  # the amplitude as held: its own error has its own test
        want = amp * Fr(T, Q)
        got = Fr(v) * sign
        # half an ulp, and up to 2 units that the product drops (8 / m <= 2^-55 of the amplitude)
        assert -want / (1 << 53) - 8 * Fr(2) ** e <= got - want <= want / (1 << 53), (T, float(want), v)


def test_no_weight_no_current(lib):
    for T in (0, -1, -2, -16):
        assert contribution(lib, -3.0, 0.7, Q // 3, T)[2] == 0.0
