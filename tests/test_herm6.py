"""The inverses of the clover term's 6 x 6 blocks (csrc/herm6.cuh) compiled for the host, against extended precision."""

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_14450_gb300", "csrc")
SOURCE = r"""
#include "herm6.cuh"
using namespace wd::herm6;
// out = s^-1 as k_clover_build forms it; the number of blocks whose pivots were exchanged
extern "C" int inverses(int n, const double* s, double* out) {
    int exchanged = 0;
    for (int k = 0; k < n; ++k, s += 36, out += 36) {
        double r[36];
        for (int i = 0; i < 36; ++i) r[i] = s[i];
        if (!sweep_inverse(r)) {
            ++exchanged;
            if (!invert_pivoted(s, r)) return -1;
        }
        for (int i = 0; i < 36; ++i) out[i] = r[i];
    }
    return exchanged;
}
extern "C" int pivoted(const double* s) { double r[36]; return invert_pivoted(s, r); }
"""
UPPER = [(i, j) for i in range(6) for j in range(i + 1, 6)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("herm6")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")], check=True)
    return C.CDLL(str(d / "t.so"))


def blocks(n, size, seed):
    """1/2 + sum_k sigma_k (x) G_k with traceless Hermitian G_k of the given size."""
    rng = np.random.default_rng(seed)

    def g():
        a = rng.normal(size=(n, 3, 3)) + 1j * rng.normal(size=(n, 3, 3))
        a = (a + a.conj().swapaxes(1, 2)) / 2
        return size * (a - np.einsum("nii->n", a)[:, None, None] / 3 * np.eye(3))

    x, y, z = g(), g(), g()
    return np.block([[0.5 * np.eye(3) + z, x - 1j * y], [x + 1j * y, 0.5 * np.eye(3) - z]])


def pack(m):
    out = np.empty((len(m), 36))
    out[:, :6] = np.einsum("nii->ni", m).real
    for q, (i, j) in enumerate(UPPER):
        out[:, 6 + 2 * q], out[:, 7 + 2 * q] = m[:, i, j].real, m[:, i, j].imag
    return out


def unpack(s):
    m = np.zeros((len(s), 6, 6), dtype=np.clongdouble)
    for i in range(6):
        m[:, i, i] = s[:, i]
    for q, (i, j) in enumerate(UPPER):
        m[:, i, j] = s[:, 6 + 2 * q] + 1j * s[:, 7 + 2 * q].astype(np.longdouble)
        m[:, j, i] = m[:, i, j].conj()
    return m


def inverse(m):
    """Gauss-Jordan elimination with partial pivoting in extended precision."""
    r = np.arange(len(m))
    a = np.concatenate([m.astype(np.clongdouble), np.broadcast_to(np.eye(6, dtype=np.clongdouble), m.shape)], 2)
    for k in range(6):
        p = k + np.abs(a[:, k:, k]).argmax(1)
        a[r, p], a[:, k] = a[:, k].copy(), a[r, p].copy()
        a[:, k] /= a[:, k, k][:, None]
        for i in range(6):
            if i != k:
                a[:, i] -= a[:, i, k][:, None] * a[:, k]
    return a[:, :, 6:]


# sizes of an ordinary c_sw (0.03, 0.06: positive definite) up to strongly indefinite blocks
@pytest.mark.parametrize("size", [0.03, 0.06, 0.12, 0.25, 0.5, 2.0])
def test_inverse_within_condition_number(lib, size):
    m = blocks(20000, size, 7)
    s = np.ascontiguousarray(pack(m))
    out = np.empty_like(s)
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
    exchanged = lib.inverses(len(s), ptr(s), ptr(out))
    assert exchanged >= 0
    if size <= 0.06:
        assert exchanged == 0
    # elimination of order 6: about 10 roundings per element, carried by the condition number
    want = inverse(m)
    err = np.abs(unpack(out) - want).max((1, 2)) / np.abs(want).max((1, 2))
    assert (err <= 10 * 2.0 ** -53 * np.linalg.cond(m)).all(), (err / np.linalg.cond(m)).max() * 2 ** 53


def test_singular_block_is_refused(lib):
    s = np.zeros((1, 36))
    s[0, :5] = 0.6
    ptr = s.ctypes.data_as(C.POINTER(C.c_double))
    out = np.empty_like(s)
    assert lib.inverses(1, ptr, out.ctypes.data_as(C.POINTER(C.c_double))) == -1
