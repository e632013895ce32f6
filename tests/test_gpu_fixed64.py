"""The fixed-point FP64 hop (SU(3) links) against the FP64-arithmetic one, which links scaled off SU(3) select."""

import pytest
import torch

from paper_2602_14450_gb300 import synth, wd
from tests.gpu_util import lattice, packed

pytestmark = pytest.mark.gpu
OFF = 1.0 + 1e-5      # the determinant deviates by 3e-5: not taken as SU(3)


def field(dims, kind):
    f = synth.to_host_layout(synth.gaussian_source(dims, seed=4))
    s = f.reshape(-1, 24)
    if kind == "tiny":            # results in the normal range, reals below the fixed-point range and subnormals
        s *= 1e-295 * 10.0 ** (-25 * torch.rand(s.shape[0], 1, generator=torch.Generator().manual_seed(1)).double())
    elif kind == "huge":
        s *= 1e300
    elif kind == "overflow":
        s *= 1e308
    elif kind == "spread":        # neighbours of very different size
        s *= 10.0 ** (400 * torch.rand(s.shape[0], 1, generator=torch.Generator().manual_seed(2)).double() - 200)
    elif kind == "point":
        s[1:] = 0.0
        s[0, 5:] = -0.0
    elif kind == "nonfinite":
        s[0, 3] = float("nan")
        s[37, 8] = float("inf")
        s[90, 20] = -float("inf")
        s[91, 0] = float("inf")
    return f


@pytest.mark.parametrize("dims,bc", [((2, 2, 2, 2), (1, 1, 1, -1)), ((4, 6, 4, 10), (-1, 1, -1, -1)),
                                     ((10, 4, 6, 8), (1, 1, 1, 1))])
@pytest.mark.parametrize("kind", ["gauss", "tiny", "huge", "overflow", "spread", "point", "nonfinite"])
def test_fixed_point_hop_matches_fp64_arithmetic(dims, bc, kind):
    if kind == "nonfinite" and dims == (2, 2, 2, 2):
        pytest.skip("too few sites")
    u = synth.gauge_random(dims, 0.5, seed=9)
    a, b = lattice(u, 0.1, dims, bc), lattice(u * OFF, 0.1, dims, bc)
    lex = field(dims, kind).cuda()
    for op, pin in ((wd.WD_OP_HOP_EO, 1), (wd.WD_OP_HOP_OE, 0)):
        src = packed(a, "fp64")
        a.pack("fp64", pin, lex, src)
        out = []
        for lat in (a, b):
            dst = packed(lat, "fp64")
            lat.apply("fp64", 18, op, src, dst)
            full = torch.zeros_like(lex)
            lat.unpack("fp64", 1 - pin, dst, full)
            out.append(full.cpu().reshape(-1, 24))
        x, y = out
        assert torch.equal(torch.isnan(x), torch.isnan(y))
        assert torch.equal(torch.isinf(x), torch.isinf(y)) and torch.equal(x[torch.isinf(x)], y[torch.isinf(y)])
        x, y = (torch.where(torch.isfinite(z), z, 0.0) for z in (x, y))
        # 36 fixed-point units of at most 2^-54 of the site's largest neighbour, ~25 roundings of the FP64 sum;
        # the site's largest neighbour bounds every result of the site, and is at most the lattice's
        size = lex.cpu().reshape(-1, 24)
        size = size[torch.isfinite(size)].abs().max()
        assert (x * OFF - y).abs().max() <= 16 * 1.0e-14 * size
        if kind == "spread":          # site by site, the larger of the two results sets the scale
            site = y.abs().amax(1, keepdim=True)
            assert ((x * OFF - y).abs() <= 1e-13 * site).all()
        if kind == "point":
            assert torch.equal(x == 0, y == 0)
