"""Loss and weight gradient of the learned preconditioner over large batches."""

import pytest
import torch

from oracle import wilson as W
from paper_2602_14450_gb300 import synth
from tests.gpu_util import lattice
from tests.test_gpu_precond import bf16_weights, packed_even

pytestmark = pytest.mark.gpu


def samples(lat, dims, n):
    f = [[packed_even(lat, "fp32", W.restrict(synth.gaussian_source(dims, seed=100 * k + i), 0)) for i in range(n)]
         for k in (1, 2)]
    return [torch.stack([x.view(torch.float32) for x in xs]) for xs in f]


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 6)])
def test_more_samples_than_a_launch_takes(dims):
    """70000 samples: more than the 65535 of one chunk, so the sums of two chunks are added."""
    lat = lattice(synth.gauge_random(dims, 0.5, seed=31), 0.12, dims)
    lat.precond_set(bf16_weights(seed=32)[0])
    v, y = samples(lat, dims, 7)
    loss, g = lat.precond_grad(v, y, 0.7)
    many, gm = lat.precond_grad(v.repeat(10000, 1), y.repeat(10000, 1), 0.7)
    assert abs(many - 10000 * loss) <= 600 * 6e-8 * many
    # FP32 sums of a block over its share of the (sample, site, colour) rows, at most 70000 x 24 x 3 / 608 of them
    rows = 70000 * 24 * 3 / 608
    g = g.double()
    assert torch.linalg.vector_norm(gm.double() - 10000 * g) <= rows * 6e-8 * 10000 * torch.linalg.vector_norm(g)


# 2^60, 2^-75: squares beyond FP32; 2^-45: their rounding errors; 2^49: above and below the border at once
@pytest.mark.parametrize("k", [60, 49, -45, -75])
def test_loss_does_not_depend_on_the_scale_of_the_samples(k):
    dims = (4, 4, 6, 10)
    lat = lattice(synth.gauge_random(dims, 0.5, seed=31), 0.12, dims)
    lat.precond_set(bf16_weights(seed=32)[0])
    v, y = samples(lat, dims, 3)
    want, _ = lat.precond_grad(v, y, 0.7)
    got, _ = lat.precond_grad(v * 2.0 ** k, y * 2.0 ** k, 0.7)
    # M, A and the residuals scale exactly; the sums of squares are good to 2^-44
    assert abs(got - want) <= 1e-12 * want
