"""Loss and weight gradient of the learned preconditioner at the edges of its kernels' tiles (32 odd sites)."""

import pytest
import torch

from oracle import ptc
from oracle import wilson as W
from paper_2602_14450_gb300 import synth
from tests.gpu_util import lattice
from tests.test_gpu_precond import bf16_weights, packed_even, unpacked_even

pytestmark = pytest.mark.gpu
KAPPA = 0.12


# V/2 = 8 (neighbours coincide, less than a tile), 24, 144 (a ragged tile), 480; one and several samples
@pytest.mark.parametrize("dims,n", [((2, 2, 2, 2), 1), ((2, 2, 2, 6), 3), ((6, 2, 4, 6), 2), ((4, 4, 6, 10), 5)])
@pytest.mark.parametrize("bc", [(1, 1, 1, -1), (-1, 1, -1, 1)])
def test_gradient_matches_oracle(dims, n, bc):
    u = synth.gauge_random(dims, 0.5, seed=31)
    lat = lattice(u, KAPPA, dims, bc)
    flat, (w1, w2) = bf16_weights(seed=32)
    lat.precond_set(flat)
    mu = 0.7
    f = [[W.restrict(synth.gaussian_source(dims, seed=100 * k + i), 0) for i in range(n)] for k in (1, 2)]
    p = [[packed_even(lat, "fp32", x) for x in fs] for fs in f]
    v, y = (torch.stack([x.view(torch.float32) for x in ps]) for ps in p)
    loss, g = lat.precond_grad(v, y, mu)
    vs, ys = ([unpacked_even(lat, "fp32", x, dims) for x in ps] for ps in p)
    L, g1, g2 = ptc.grads(u, w1, w2, vs, ys, KAPPA, mu, bc)
    want = ptc.to_flat(g1, g2)
    # FP32 throughout: M and A sum ~600 products per real (2^-24 each), the gradient's sums run over that
    assert abs(loss - L) <= 600 * 6e-8 * L
    err = torch.linalg.vector_norm(g.cpu().double() - want) / torch.linalg.vector_norm(want)
    assert err.item() <= 2 * 600 * 6e-8
