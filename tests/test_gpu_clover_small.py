"""C psi of the Wilson-clover matrix for weak fields: the components that C alone feeds keep their own precision."""

import pytest
import torch

from oracle import clover as CL
from oracle import wilson as W
from paper_2602_14450_gb300 import synth, wd
from tests.gpu_util import apply_op, lattice

pytestmark = pytest.mark.gpu
ROUND = {"fp32": 2.0 ** -24, "fp16": 2.0 ** -11, "bf16": 2.0 ** -8}


def off_diagonal(u, csw, kappa, dims, prec, j):
    """Column j of C at every even site from D_sw on a field of that component on the even sites (whose hops reach odd
    sites only), and the oracle's, both without the diagonal element."""
    psi = torch.zeros_like(synth.gaussian_source(dims, seed=1))
    psi.reshape(-1, 12)[:, j] = 1.0
    psi = W.restrict(psi, 0)
    lat = lattice(u, kappa, dims)
    lat.set_clover(csw)
    got = apply_op(lat, prec, 18, wd.WD_OP_FULL, psi, dims).reshape(-1, 12)
    want = CL.clover_matrix(u, csw, kappa).reshape(-1, 12, 12)[:, :, j]
    even = W.parity(dims).reshape(-1) == 0
    keep = [i for i in range(12) if i != j]
    return got[even][:, keep], want[even][:, keep]


# An element is the sum of at most two elements of each chiral block, rounded to storage, and is rounded once more.
@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("j", [0, 4, 8, 11])
def test_storage_precision_of_weak_fields(prec, j):
    dims = (4, 4, 4, 6)
    got, want = off_diagonal(synth.gauge_random(dims, 0.02, seed=9), 1.0, 0.12, dims, prec, j)
    assert (got - want).abs().amax() <= 8 * ROUND[prec] * want.abs().amax()


# Links within eps of 1. A real of F is a sum over four leaves of products of four links of which one factor is small, 16
# such terms: at most 22 roundings of 16 eps, and F itself is of size eps. 0.3 and 0.03: on both sides of the border
# between fixed point and FP64 arithmetic.
@pytest.mark.parametrize("eps", [0.3, 0.03, 1e-3, 1e-5, 1e-8])
@pytest.mark.parametrize("j", [0, 4, 8, 11])
def test_fp64_blocks_of_weak_fields(eps, j):
    dims = (2, 4, 4, 6)
    got, want = off_diagonal(synth.gauge_random(dims, eps, seed=9), 1.0, 0.12, dims, "fp64", j)
    assert (got - want).abs().amax() <= 22 * 16 * 1.1e-16 * want.abs().amax()
