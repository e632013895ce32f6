"""Clover blocks built in fixed point (SU(3) links), in FP64 arithmetic (other links) and with exchanged pivots."""

import pytest
import torch

from oracle import clover as CL
from oracle import wilson as W
from paper_2602_14450_gb300 import synth, wd
from tests.gpu_util import apply_op, lattice

pytestmark = pytest.mark.gpu


# (2, 2, 2, 2): neighbours coincide; (2, 6, 4, 10): a ragged last block. c_sw = 12 makes indefinite blocks, whose
# plain pivots can be small.
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 4, 10)])
@pytest.mark.parametrize("csw", [1.0, 12.0])
@pytest.mark.parametrize("scale", [1.0, 1.01])
def test_clover_operators_match_oracle(dims, csw, scale):
    kappa = 0.12
    u = scale * synth.gauge_random(dims, 0.7, seed=21)
    psi = synth.gaussian_source(dims, seed=22)
    lat = lattice(u, kappa, dims)
    lat.set_clover(csw)
    c = CL.clover_matrix(u, csw, kappa)
    want = CL.dirac_sw(u, c, psi, kappa)
    got = apply_op(lat, "fp64", 18, wd.WD_OP_FULL, psi, dims)
    assert (got - want).abs().max() <= 1e-13 * want.abs().max()
    want = CL.eo_operator_sw(u, torch.linalg.inv(c), W.restrict(psi, 0), kappa)
    got = apply_op(lat, "fp64", 18, wd.WD_OP_EO_A, psi, dims)
    # An inverse is good to its condition number times the roundings of the elimination, about 10 times 2^-53 per
    # element, grown by at most 1 / (2 x the smallest plain pivot taken, 5e-4); two blocks per operator.
    cond = torch.linalg.cond(c.reshape(-1, 12, 12)).max().item()
    assert (got - want).abs().max() <= 2 * 10 * 1.1e-16 * 1000 * cond * want.abs().max()
