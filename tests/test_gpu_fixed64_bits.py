"""The fixed-point arithmetic of the FP64 hop (csrc/fixed64.cuh) on the device: the bits of its host build, which
tests/test_fixed64.py holds to exact rationals."""

import ctypes as C
import random
import subprocess

import numpy as np
import pytest

from paper_2602_14450_gb300 import build
from tests.test_fixed64 import CSRC, SOURCE, exponent, values

pytestmark = pytest.mark.gpu
DEVICE = r"""
#include "fixed64.cuh"
using namespace wd::fx;
__global__ void k(int n, const double* u, const double* p, const double* q, const int* minus, const int* E, double* out,
                  int* dig) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int u0[6], u1[6], n0[3], n1[3], h0[6], h1[6];
    for (int k = 0; k < 6; ++k) link_digits(u[6 * i + k], u0[k], u1[k]);
    for (int b = 0; b < 3; ++b) { n0[b] = -u0[2 * b + 1]; n1[b] = -u1[2 * b + 1]; }
    for (int k = 0; k < 6; ++k) {
        const double x = p[6 * i + k], y = q[6 * i + k];
        digits(sum(fixed(__double2hiint(x), __double2loint(x), E[i]),
                   signed_by(fixed(__double2hiint(y), __double2loint(y), E[i]), minus[6 * i + k] ? -1 : 0)), h0[k], h1[k]);
    }
    long long re, im;
    row_mul(u0, u1, n0, n1, h0, h1, re, im);
    out[2 * i] = to_double(re, E[i]);
    out[2 * i + 1] = to_double(im, E[i]);
    for (int k = 0; k < 6; ++k) { dig[12 * i + 2 * k] = u0[k]; dig[12 * i + 2 * k + 1] = u1[k]; }
}
extern "C" int run(int n, const void* const* in, const size_t* bytes, void* const* out) {
    void* d[7];
    for (int i = 0; i < 7; ++i)
        if (cudaMalloc(&d[i], bytes[i]) != cudaSuccess) return 1;
    for (int i = 0; i < 5; ++i)
        if (cudaMemcpy(d[i], in[i], bytes[i], cudaMemcpyHostToDevice) != cudaSuccess) return 2;
    k<<<(n + 127) / 128, 128>>>(n, (double*)d[0], (double*)d[1], (double*)d[2], (int*)d[3], (int*)d[4], (double*)d[5],
                                (int*)d[6]);
    for (int i = 0; i < 2; ++i)
        if (cudaMemcpy(out[i], d[5 + i], bytes[5 + i], cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    for (int i = 0; i < 7; ++i) cudaFree(d[i]);
    return 0;
}
"""


def test_device_gives_the_bits_of_the_host_build(tmp_path):
    (tmp_path / "h.cpp").write_text(SOURCE)
    (tmp_path / "d.cu").write_text(DEVICE)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(tmp_path / "h.so"), str(tmp_path / "h.cpp")],
                   check=True)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-I", CSRC, "-o", str(tmp_path / "d.so"),
                    str(tmp_path / "d.cu"), "-lcudart"], check=True)
    host, dev = C.CDLL(str(tmp_path / "h.so")), C.CDLL(str(tmp_path / "d.so"))
    host.link.argtypes, host.link.restype = [C.c_double, C.POINTER(C.c_int)], C.c_double
    rng = random.Random(23)
    rows = []
    for kind in ("gauss", "unit", "largest", "spread", "zeros"):
        for _ in range(2000):
            u, p, q = values(rng, kind)
            e = max(map(exponent, p + q))
            if 70 <= e <= 2030:
                minus = [rng.randint(0, 1) if kind != "largest" else 0 for _ in range(6)]
                rows.append((u, p, q, minus, min(2030, e + rng.choice([0, 0, 1, 7, 64, 200]))))
    n = len(rows)
    u, p, q = (np.array([r[i] for r in rows]) for i in range(3))
    minus, e = np.array([r[3] for r in rows], dtype=np.int32), np.array([r[4] for r in rows], dtype=np.int32)
    out, dig = np.zeros((n, 2)), np.zeros((n, 6, 2), dtype=np.int32)
    arrays = [u, p, q, minus, e, out, dig]
    ptr = lambda a: a.ctypes.data  # noqa: E731
    rc = dev.run(n, (C.c_void_p * 5)(*map(ptr, arrays[:5])), (C.c_size_t * 7)(*(a.nbytes for a in arrays)),
                 (C.c_void_p * 2)(ptr(out), ptr(dig)))
    assert rc == 0
    want, wdig = np.zeros((n, 2)), np.zeros_like(dig)
    at = lambda a, t: a.ctypes.data_as(C.POINTER(t))  # noqa: E731
    for i in range(n):
        host.row(at(u[i], C.c_double), at(p[i], C.c_double), at(q[i], C.c_double), at(minus[i], C.c_int), int(e[i]),
                 at(want[i], C.c_double))
        for k in range(6):
            host.link(u[i, k], at(wdig[i, k], C.c_int))
    assert np.array_equal(dig, wdig)
    assert np.array_equal(out.view(np.int64), want.view(np.int64))
