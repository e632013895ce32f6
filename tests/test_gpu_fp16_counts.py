"""Matvec counts of the FP16-arithmetic solves over several sources: a single solve's count moves by whole refinement
trips with the last bits of its dot products and residuals, the median over sources does not."""

import statistics

import pytest
import torch

from paper_2602_14450_gb300 import synth, wd
from tests.gpu_util import lattice, lex_dev

pytestmark = pytest.mark.gpu
DIMS = (8, 8, 8, 8)


@pytest.mark.parametrize("scheme,ftz", [("mixed_fp16", 0), ("mixed_fp16", 1), ("mixed_fp16_plain", 0)])
def test_median_count_of_fp16_arithmetic(scheme, ftz):
    """FP16 arithmetic takes at most 1.3 times the matvecs of FP32 arithmetic, plus 8, in the median over nine
    sources, and every solve reaches the tolerance."""
    lat = lattice(synth.gauge_smeared(DIMS, seed=20260214), 0.13, DIMS)
    counts = {16: [], 32: []}
    for seed in range(450, 459):
        b = lex_dev(synth.gaussian_source(DIMS, seed=seed))
        for bits in counts:
            lat.set_arith(bits)
            x = torch.zeros_like(b)
            p = wd.default_params(scheme)
            p.ftz = ftz
            st = lat.solve(b, x, 1e-10, scheme, params=p)
            assert st.status == wd.WD_OK and st.true_residual <= 1e-10
            counts[bits].append(st.inner_matvecs)
    assert statistics.median(counts[16]) <= 1.3 * statistics.median(counts[32]) + 8, counts
