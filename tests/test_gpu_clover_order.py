"""wd_set_clover while an earlier operator still waits on another stream: that operator gets the blocks it was given."""

import pytest
import torch

from paper_2602_14450_gb300 import synth, wd
from tests.gpu_util import lattice, packed

pytestmark = pytest.mark.gpu
DIMS = (8, 8, 8, 8)


@pytest.mark.parametrize("prec,recon", [("fp64", 18), ("fp32", 12), ("fp16", 12), ("bf16", 18)])
@pytest.mark.parametrize("op", [wd.WD_OP_EO_A, wd.WD_OP_FULL])
def test_pending_operator_keeps_its_blocks(prec, recon, op):
    lat = lattice(synth.gauge_random(DIMS, 0.5, seed=3), 0.12, DIMS)
    lex = synth.to_host_layout(synth.gaussian_source(DIMS, seed=4)).cuda()
    n = 2 if op == wd.WD_OP_FULL else 1
    nb = lat.vector_bytes(prec)
    src, want, got, other = (packed(lat, prec, n) for _ in range(4))
    for p in range(n):
        lat.pack(prec, p, lex, src[p * nb:(p + 1) * nb])
    lat.set_clover(1.0)
    lat.apply(prec, recon, op, src, want)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(int(2e8))          # about 0.1 s
        lat.apply(prec, recon, op, src, got)
    lat.set_clover(3.0)
    lat.apply(prec, recon, op, src, other)
    torch.cuda.synchronize()
    assert torch.equal(got, want) and not torch.equal(other, want)
