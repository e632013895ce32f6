"""wd_tune chooses among launches that differ, and the default it reports is the one that runs without it."""

import pytest

from paper_2602_14450_gb300 import synth
from tests.gpu_util import lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 16), (16, 16, 16, 32)])
def test_fixed_point_hop_has_one_kernel(dims):
    """FP64 on SU(3) links: every variant is the same kernel, of at most 128 threads; what is reported is what runs."""
    lat = lattice(synth.gauge_random(dims, 0.5, seed=17), 0.12, dims)
    for _ in range(4):
        r = lat.tune("fp64", 18)
        assert (r["variant"], r["variant_reducing"]) == (4, 4)
        assert r["block"] in (64, 128) and r["block_reducing"] in (64, 128)
        assert 0 < r["us"] <= r["default_us"]


def test_smallest_lattice_reports_the_default():
    """On 4^4 every block size is split down to one warp: the default's stands for all of its variant."""
    lat = lattice(synth.gauge_random((4, 4, 4, 4), 0.5, seed=17), 0.12, (4, 4, 4, 4))
    for prec, recon, block in (("fp32", 12, 64), ("bf16", 18, 128), ("fp16", 18, 128)):
        r = lat.tune(prec, recon)
        assert r["block"] in (block, 128) and r["us"] <= r["default_us"]
        if r["variant"] == (4 if prec == "fp32" else 1):
            assert r["block"] == block
