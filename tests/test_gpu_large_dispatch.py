"""Kernels that the dispatch takes only beyond 160000 sites per parity, against the FP64 operator."""

import pytest
import torch

from paper_2602_14450_gb300 import synth, wd
from tests.gpu_util import TOL

pytestmark = pytest.mark.gpu
DIMS = (24, 24, 24, 24)       # 165,888 sites per parity, not a multiple of the larger blocks


@pytest.fixture(scope="module")
def lat():
    h = wd.Lattice(DIMS, 0.12)
    h.set_gauge(torch.view_as_real(synth.gauge_random(DIMS, 0.5, seed=41, device="cuda")).contiguous())
    return h


@pytest.mark.parametrize("csw", [0.0, 1.0])
@pytest.mark.parametrize("prec,recon,arith", [("bf16", 12, 32), ("bf16", 18, 32), ("fp16", 12, 32), ("fp16", 18, 32),
                                              ("fp16", 12, 16), ("fp32", 12, 32)])
def test_even_odd_operator_matches_fp64(lat, csw, prec, recon, arith):
    lat.set_clover(csw)
    lat.set_arith(arith)
    f = torch.randn(DIMS[::-1] + (4, 3, 2), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda",
                    dtype=torch.float64)
    out = []
    for p, r in ((prec, recon), ("fp64", 18)):
        a = torch.empty(lat.vector_bytes(p), dtype=torch.uint8, device="cuda")
        b = torch.empty_like(a)
        lat.pack(p, 0, f, a)
        lat.apply(p, r, wd.WD_OP_EO_A, a, b)
        lex = torch.zeros_like(f)
        lat.unpack(p, 0, b, lex)
        out.append(lex)
    assert (out[0] - out[1]).norm() <= TOL["fp16a" if arith == 16 else prec] * out[1].norm()
