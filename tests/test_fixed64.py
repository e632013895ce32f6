"""The fixed-point arithmetic of the FP64 hop (csrc/fixed64.cuh) compiled for the host, against exact rationals."""

import ctypes as C
import math
import os
import random
import struct
import subprocess
from fractions import Fraction as F

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_14450_gb300", "csrc")
SOURCE = r"""
#include "fixed64.cuh"
using namespace wd::fx;
extern "C" void row(const double* u, const double* p, const double* q, const int* minus, int E, double* out) {
    int u0[6], u1[6], n0[3], n1[3], h0[6], h1[6];
    for (int i = 0; i < 6; ++i) link_digits(u[i], u0[i], u1[i]);
    for (int b = 0; b < 3; ++b) { n0[b] = -u0[2 * b + 1]; n1[b] = -u1[2 * b + 1]; }
    for (int i = 0; i < 6; ++i) {
        unsigned w[2], x[2];
        memcpy(w, p + i, 8);
        memcpy(x, q + i, 8);
        digits(sum(fixed(w[1], w[0], E), signed_by(fixed(x[1], x[0], E), minus[i] ? -1 : 0)), h0[i], h1[i]);
    }
    long long re, im;
    row_mul(u0, u1, n0, n1, h0, h1, re, im);
    out[0] = to_double(re, E);
    out[1] = to_double(im, E);
}
extern "C" double link(double u, int* d) { link_digits(u, d[0], d[1]); return link_value(d[0], d[1]); }
"""
# One link row times one column, in units of 2^(E-1078): reals cut below 1/8 each (2 per entry, sqrt(6)/8 * 2 in
# all), u0 h0 left out (6 * 2/8), link entries off by 2^-62 (6/32), one rounding (1/2).
BOUND = 2 * math.sqrt(6) / 8 + 1.5 + 0.1875 + 0.5


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed64")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")], check=True)
    L = C.CDLL(str(d / "t.so"))
    L.link.argtypes, L.link.restype = [C.c_double, C.POINTER(C.c_int)], C.c_double
    return L


def exponent(x):
    return struct.unpack("<Q", struct.pack("<d", abs(x)))[0] >> 52


def values(rng, kind):
    u = [rng.gauss(0, 1) for _ in range(6)]
    n = math.sqrt(sum(x * x for x in u))
    u = [x / n for x in u]
    scale = 2.0 ** rng.randint(-940, 990)
    p, q = ([rng.gauss(0, 1) * scale for _ in range(6)] for _ in range(2))
    if kind == "unit":
        u = [0.0] * 6
        u[rng.randrange(6)] = rng.choice([1.0, -1.0, 1.0 + 1e-6])
    elif kind == "largest":      # every real at the top of its binade, signs such that all terms add up
        u = [math.copysign(1 / math.sqrt(6), x) for x in u]
        p = [math.copysign((2 - 2.0 ** -52) * scale, x) for x in u]
        q = list(p)
    elif kind == "spread":
        p = [x * 10 ** rng.uniform(-40, 0) for x in p]
    elif kind == "zeros":
        p = [rng.choice([0.0, -0.0, 5e-324, x]) for x in p]
        q = [rng.choice([0.0, -0.0, -5e-324, x]) for x in q]
    return u, p, q


@pytest.mark.parametrize("kind", ["gauss", "unit", "largest", "spread", "zeros"])
def test_row_product_within_derived_bound(lib, kind):
    rng = random.Random(11)
    for _ in range(3000):
        u, p, q = values(rng, kind)
        E = max(map(exponent, p + q))
        if not 70 <= E <= 2030:
            continue
        E = min(2030, E + rng.choice([0, 0, 0, 1, 7, 64, 200]))      # a scale set by an earlier neighbour
        minus = [rng.randint(0, 1) if kind != "largest" else 0 for _ in range(6)]
        o = (C.c_double * 2)()
        lib.row((C.c_double * 6)(*u), (C.c_double * 6)(*p), (C.c_double * 6)(*q), (C.c_int * 6)(*minus), E, o)
        h = [F(a) + (-F(b) if m else F(b)) for a, b, m in zip(p, q, minus)]
        w = [F(x) for x in u]
        exact = (sum(w[2 * b] * h[2 * b] - w[2 * b + 1] * h[2 * b + 1] for b in range(3)),
                 sum(w[2 * b] * h[2 * b + 1] + w[2 * b + 1] * h[2 * b] for b in range(3)))
        for got, want in zip(o, exact):
            assert abs(F(got) - want) <= F(BOUND) * F(2) ** (E - 1078) + F(math.ulp(got)) / 2, (kind, u, p, q, E)
            if not any(h):
                assert got == 0.0


def test_link_digits(lib):
    rng = random.Random(5)
    d = (C.c_int * 2)()
    special = [0.0, 1.0, -1.0, 1.000001, -1.000001, 2.0 ** -30, -2.0 ** -30, 2.0 ** -62, 2.0 ** -30 - 2.0 ** -61]
    for u in special + [rng.uniform(-1, 1) for _ in range(5000)] + [rng.uniform(-1, 1) * 2.0 ** -30 for _ in range(5000)]:
        v = lib.link(u, d)
        assert d[0] != -2 ** 31 and abs(d[1]) <= 2 ** 29 + 2 ** 10      # both digits can be negated
        assert abs((F(d[1]) * 2 ** 32 + d[0]) / 2 ** 61 - F(u)) <= F(1, 2 ** 62) + (F(1, 2 ** 61) if d[0] == -2 ** 31 + 1 else 0)
        assert abs(v - u) <= 2.0 ** -60
