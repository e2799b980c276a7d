"""The fixed-point arithmetic of the particle kernel's gather and deposit
(csrc/pic_fix.cuh), compiled for the host with stand-ins for the device
intrinsics and compared with exact rational arithmetic."""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <cmath>
#include <cstring>
#include <algorithm>
#define __device__
#define __forceinline__ inline
#define __noinline__
using std::max; using std::min;
static inline long long __double_as_longlong(double x) { long long b; memcpy(&b, &x, 8); return b; }
static inline double __longlong_as_double(long long b) { double x; memcpy(&x, &b, 8); return x; }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
static inline int __clzll(long long v) { return v ? __builtin_clzll(v) : 64; }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, int s) { s &= 31; return s ? (hi << s) | (lo >> (32 - s)) : hi; }
static inline int __clz(int v) { return v ? __builtin_clz(v) : 32; }
static inline long long __double2ll_rn(double x) { return std::llrint(x); }
#include "pic_fix.cuh"
template <int ORDER> static void sup(double x, int kind, int* s, long long* w) {
    const CellQ c = cell_q(x);
    const SupQ<ORDER> u = kind == 0 ? node_support<ORDER>(c, 0) : half_support<ORDER>(c, 0, kind == 2);
    *s = u.s;
    for (int k = 0; k <= ORDER; ++k) w[k] = ORDER == 1 && k == 0 ? kOneQ - u.w[1] : u.w[k];
}
extern "C" {
void t_support(int order, double x, int kind, int* s, long long* w) {
    if (order == 1) sup<1>(x, kind, s, w);
    else if (order == 2) sup<2>(x, kind, s, w);
    else sup<3>(x, kind, s, w);
}
long long t_mulq(long long a, long long b) { return mulq(limb_of(a), limb_of(b)); }
long long t_lerp(long long a, long long b, long long w) { return lerpq(a, b, limb_of(w)); }
long long t_line(int n, const long long* f, const long long* w) {
    AccQ s;
    for (int k = 0; k < n; ++k) s.mac(f[k], limb_of(w[k]));
    return s.get();
}
unsigned long long t_mulhi(unsigned long long a, unsigned long long b) { return mulhi(a, b); }
double t_round(double v, int emax, int fb) {  // through the tile's fixed point and back
    return fb == 62 ? fix_double(tile_fix<62>(v, emax), emax + 1) : fix_double(tile_fix<60>(v, emax), emax + 3);
}
void t_scale(double c, double q, long long p, unsigned long long* m, int* e, unsigned* s, int* safe) {
    const Amp a = amp_scale(amp_mul(amp_of(c), amp_of(q)), p);
    const unsigned h = a.es + (1024u << 20);
    *m = a.m; *e = (int)((h >> 20) & 0x7FFu) - 1024; *s = h >> 31; *safe = in_range(exp_range(c, 1.0, c), exp_field(q));
}
double t_pack(unsigned long long v, int x, int round) {
    const unsigned hi = (unsigned)(x + 1085) << 20;
    return round ? pack_double<true>(v, hi) : pack_double<false>(v, hi);
}
}
"""
Q = 1 << 62


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix")
    csrc = os.path.join(ROOT, "paper_2104_11385_gb300", "csrc")
    src = d / "shim.cpp"
    # the header's only CUDA include is replaced by the stand-ins above
    (d / "cuda_runtime.h").write_text("#pragma once\n")
    src.write_text(SHIM)
    so = d / "shim.so"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(d), "-I", csrc, str(src), "-o",
                           str(so)])
    L = ctypes.CDLL(str(so))
    for f in ("t_mulq", "t_lerp", "t_line"):
        getattr(L, f).restype = ctypes.c_longlong
    L.t_mulhi.restype = ctypes.c_ulonglong
    L.t_round.restype = L.t_pack.restype = ctypes.c_double
    return L


def ll(v):
    return ctypes.c_longlong(int(v))


def shape(order, t):
    """B-spline of the order at distance t, exact"""
    a = abs(t)
    if order == 0:
        return Fr(1) if -Fr(1, 2) <= t < Fr(1, 2) else Fr(0)
    if order == 1:
        return max(Fr(0), 1 - a)
    if order == 2:
        return Fr(3, 4) - a * a if a <= Fr(1, 2) else (max(Fr(0), Fr(3, 2) - a) ** 2) / 2
    return Fr(2, 3) - a * a + a ** 3 / 2 if a <= 1 else max(Fr(0), 2 - a) ** 3 / 6


POSITIONS = [0.0, 1e-300, 2.0 ** -70, 2.0 ** -11, 2.0 ** -10, 0.25, 0.5, np.nextafter(0.5, 0), 1.0, np.nextafter(1.0, 0),
             7.5, np.nextafter(8.0, 0), 511.99999999999994, 1048575.5, -2.0 ** -30, -0.5, -1.0, -1.25]


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("kind", [0, 1, 2])  # nodes, half nodes, half nodes of the energy-conserving gather
def test_supports(lib, order, kind):
    r = np.random.default_rng(5)
    xs = POSITIONS + list(r.uniform(0, 512, 200)) + list(r.uniform(0, 1, 50))
    for x in map(float, xs):
        s, w = ctypes.c_int(), (ctypes.c_longlong * 4)()
        lib.t_support(order, ctypes.c_double(x), kind, ctypes.byref(s), w)
        got = [w[k] for k in range(order + 1)]
        assert sum(got) == Q and min(got) >= 0, (x, got)
        o = order - 1 if kind == 2 else order
        for k in range(order + 1):
            t = Fr(x) - (s.value + k) - (Fr(1, 2) if kind else 0)
            # truncation of the offset and of each product: a few units
            assert abs(Fr(got[k], Q) - shape(o, t)) <= Fr(12, Q), (x, k)


def test_products(lib):
    r = np.random.default_rng(6)
    edge = [0, 1, 2 ** 31 - 1, 2 ** 31, 2 ** 32, 2 ** 61, Q - 1, Q]
    w = edge + [int(v) for v in r.integers(0, Q, 300)]
    v = edge[:-1] + [int(t) for t in r.integers(-Q + 1, Q, 301)]
    # the dropped product of the low limbs is at most 1 unit for two balanced
    # limbs, 2 for an unsigned and a balanced one, and each result truncates 1
    for a, b in zip(w + w[::-1], v + [-t for t in v]):
        assert abs(lib.t_mulq(ll(a), ll(b)) - Fr(a * b, Q)) <= 2
        assert abs(lib.t_lerp(ll(b), ll(-b // 3), ll(a)) - (b + Fr(a, Q) * (-b // 3 - b))) <= 3
        m, n = Q + a - (a == Q), abs(b) << 1
        assert 0 <= Fr(m * n, 1 << 64) - lib.t_mulhi(ctypes.c_ulonglong(m), ctypes.c_ulonglong(n)) <= 3
    big = 2 ** 60 - 1
    for f in ([big] * 4, [-big] * 4, [big, -big, big, -big], [int(t) for t in r.integers(-big, big, 4)]):
        for ws in ([Q, 0, 0, 0], [Q // 4] * 4, [Q // 6, 2 * (Q // 3) + 1, Q // 6, 0]):
            got = lib.t_line(4, (ctypes.c_longlong * 4)(*f), (ctypes.c_longlong * 4)(*ws))
            assert abs(got - sum(Fr(a * b, Q) for a, b in zip(f, ws))) <= 9


@pytest.mark.parametrize("fb", [62, 60])
def test_tile_values(lib, fb):
    r = np.random.default_rng(7)
    for emax in (128, 1000, 1023, 1900):
        top = float(np.ldexp(1.0, emax - 1023))
        vals = [0.0, top, -top, np.nextafter(2 * top, 0), 5e-324, top * 2.0 ** -52, top * 2.0 ** -70]
        vals += list(r.uniform(-2, 2, 100) * top) + list(r.uniform(-2, 2, 50) * top * 2.0 ** -fb)
        for v in map(float, vals):
            got = lib.t_round(ctypes.c_double(v), emax, fb)
            # half a unit of the tile, then half an ulp (values down to 2^-(fb - 53) of the largest are exact)
            tol = Fr(top) * 2 / (1 << (fb + 1))
            if abs(v) >= top * 2.0 ** (54 - fb):
                assert got == v
            assert abs(Fr(got) - Fr(v)) <= tol + abs(Fr(v)) / (1 << 53)


def test_pack(lib):
    r = np.random.default_rng(9)
    vals = [1, 2, 3, 2 ** 31, 2 ** 32 - 1, 2 ** 32, 2 ** 53 - 1, 2 ** 53 + 1, 2 ** 62 - 1, 2 ** 63 - 1]
    for v in vals + [int(t) >> int(k) for t, k in zip(r.integers(1, 2 ** 63 - 1, 300), r.integers(0, 62, 300))]:
        v = max(v, 1)
        for x in (-700, -62, 0, 100):
            want = Fr(v) * Fr(2) ** x
            assert abs(Fr(lib.t_pack(ctypes.c_ulonglong(v), x, 1)) - want) <= want / (1 << 53)
            low = Fr(lib.t_pack(ctypes.c_ulonglong(v), x, 0))
            assert low <= want and want - low < want / (1 << 52)


def test_amplitudes(lib):
    r = np.random.default_rng(8)
    for _ in range(300):
        c, q = (float(np.ldexp(r.uniform(-1, 1), int(r.integers(-200, 200)))) for _ in range(2))
        p = int(r.integers(-Q, Q)) >> int(r.integers(0, 62))
        m, e, s, safe = ctypes.c_ulonglong(), ctypes.c_int(), ctypes.c_uint(), ctypes.c_int()
        lib.t_scale(ctypes.c_double(c), ctypes.c_double(q), ll(p), *map(ctypes.byref, (m, e, s, safe)))
        want = Fr(c) * Fr(q) * Fr(p, Q)
        got = Fr(m.value) * Fr(2) ** e.value * (-1 if s.value else 1)
        assert safe.value == 1
        assert abs(got - want) <= abs(want) * Fr(1, 1 << 56)
    for c, q in ((1e-300, 1e-10), (1e300, 1e10), (float("inf"), 1.0), (float("nan"), 1.0)):
        m, e, s, safe = ctypes.c_ulonglong(), ctypes.c_int(), ctypes.c_uint(), ctypes.c_int()
        lib.t_scale(ctypes.c_double(c), ctypes.c_double(q), ll(Q), *map(ctypes.byref, (m, e, s, safe)))
        assert safe.value == 0
