"""The FP64 hop of SU(3) links, component by component, against exact rational arithmetic.

The bound is the one FP64 arithmetic has: a real of H psi is a sum of products of link and half-spinor reals; each
product passes one rounding of the projection, six of the colour row and seven of the sum over directions, 14 in all
(15 with second-order terms), so the error is at most 15 x 2^-53 times the sum of the products' absolute values.
"""

from fractions import Fraction as F

import pytest
import torch

from oracle.gamma import projectors
from paper_2602_14450_gb300 import synth, wd
from tests.gpu_util import lattice, packed

pytestmark = pytest.mark.gpu
UNIT = F(15, 2 ** 53)


def exact_hop(u, psi, p, bc, split=()):
    """{site: 24 (value, sum of absolute products)} of the hop onto parity p, without the hops that wrap around in a
    direction of `split`; u [4, t, z, y, x, 3, 3], psi [t, z, y, x, 4, 3] complex128."""
    lt, lz, ly, lx = psi.shape[:4]
    ext = (lx, ly, lz, lt)
    uf, pf = u.reshape(4, -1, 3, 3).tolist(), psi.reshape(-1, 4, 3).tolist()
    # rows of (1 -/+ gamma): spin s is a sum of (spin t, re, im) with re, im in {0, +-1, +-2}
    rows = [[[[(t, int(c.real), int(c.imag)) for t, c in enumerate(r) if c != 0] for r in m] for m in mats.tolist()]
            for mats in projectors()]
    fr = lambda z: (F(z.real), F(z.imag))  # noqa: E731
    out = {}
    for site in range(lx * ly * lz * lt):
        c = [site % lx, (site // lx) % ly, (site // (lx * ly)) % lz, site // (lx * ly * lz)]
        if sum(c) % 2 != p:
            continue
        val, mag = [[F(0), F(0)] for _ in range(12)], [[F(0), F(0)] for _ in range(12)]
        for d in range(8):
            mu, fwd = d >> 1, d % 2 == 0
            wrap = c[mu] == (ext[mu] - 1 if fwd else 0)
            if wrap and mu in split:
                continue
            n = list(c)
            n[mu] = (c[mu] + (1 if fwd else -1)) % ext[mu]
            site_n = n[0] + lx * (n[1] + ly * (n[2] + lz * n[3]))
            ph = bc[mu] if wrap else 1
            f = [[fr(z) for z in s] for s in pf[site_n]]
            m = uf[mu][site] if fwd else uf[mu][site_n]
            lk = [[fr(m[a][b]) if fwd else fr(m[b][a].conjugate()) for b in range(3)] for a in range(3)]
            for s in range(4):
                h, ha = [], []
                for b in range(3):
                    re = sum(x * f[t][b][0] - y * f[t][b][1] for t, x, y in rows[0 if fwd else 1][mu][s])
                    im = sum(x * f[t][b][1] + y * f[t][b][0] for t, x, y in rows[0 if fwd else 1][mu][s])
                    h.append((re, im))
                    ha.append([sum(abs(x) * abs(f[t][b][i]) + abs(y) * abs(f[t][b][1 - i])
                                   for t, x, y in rows[0 if fwd else 1][mu][s]) for i in range(2)])
                for a in range(3):
                    k = 3 * s + a
                    for b in range(3):
                        lr, li = lk[a][b]
                        val[k][0] += ph * (lr * h[b][0] - li * h[b][1])
                        val[k][1] += ph * (lr * h[b][1] + li * h[b][0])
                        mag[k][0] += abs(lr) * ha[b][0] + abs(li) * ha[b][1]
                        mag[k][1] += abs(lr) * ha[b][1] + abs(li) * ha[b][0]
        out[site] = [(v, m) for vs, ms in zip(val, mag) for v, m in zip(vs, ms)]
    return out


def check(got, want):
    """got: lexicographic [V, 24]; every real within the bound of FP64 arithmetic."""
    for site, reals in want.items():
        for i, (v, m) in enumerate(reals):
            assert abs(F(got[site][i]) - v) <= UNIT * m, (site, i, got[site][i], float(v), float(m))


def smooth(dims, eps, seed):
    """SU(3) links with off-diagonal entries of size eps around diagonal phases."""
    u = synth.gauge_random(dims, eps, seed=seed)
    ph = synth.gaussian_source(dims, seed=seed + 1)[..., 0, :2].real
    a, b = ph[..., 0], ph[..., 1]
    d = torch.polar(torch.ones_like(torch.stack([a, b, -a - b], -1)), torch.stack([a, b, -a - b], -1))
    return d[None, ..., :, None] * u


def fields(dims, kind):
    """Links and spinors of a kind."""
    u = synth.gauge_random(dims, 0.5, seed=9)
    psi = synth.gaussian_source(dims, seed=4)
    v = psi.reshape(-1, 4, 3)
    if kind == "small entries":     # one colour only: the others are fed by small link entries alone
        u = smooth(dims, 1e-9, 9)
        v[:, :, 1:] = 0.0
    elif kind == "tiny entries":    # below the last bit of a fixed-point link
        u = smooth(dims, 1e-20, 9)
        v[:, :, 1:] = 0.0
    elif kind == "unit links":
        u = torch.eye(3, dtype=u.dtype).expand_as(u).contiguous()
        v[:, :, 2] *= 1e-8
    elif kind == "spins":           # two spins much smaller
        v[:, 2:] *= 1e-8
    elif kind == "one spin":
        v[:, 1:] = 0.0
    elif kind == "time slices":     # large t neighbours, which feed two spins of a site
        psi[::2] *= 1e-8
    elif kind == "spread":          # sites of very different size
        v *= 10.0 ** (30 * torch.rand(v.shape[0], 1, 1, generator=torch.Generator().manual_seed(2)).double() - 15)
    elif kind == "point":
        v[1:] = 0.0
        v[0, 1:] = 0.0
    elif kind == "small":           # reals at the lower end of the fixed-point range
        v *= 2.0 ** -950
    elif kind == "large":
        v *= 2.0 ** 1000
    return u, psi


KINDS = ["gauss", "small entries", "tiny entries", "unit links", "spins", "one spin", "time slices", "spread", "point",
         "small", "large"]


@pytest.mark.parametrize("dims,bc", [((2, 2, 2, 4), (1, 1, 1, -1)), ((4, 2, 6, 2), (-1, 1, -1, 1))])
@pytest.mark.parametrize("kind", KINDS)
def test_every_component_within_the_bound_of_fp64_arithmetic(dims, bc, kind):
    u, psi = fields(dims, kind)
    lat = lattice(u, 0.1, dims, bc)
    dev = lat.unitarity()
    assert max(dev) < 1e-6
    for op, p in ((wd.WD_OP_HOP_EO, 0), (wd.WD_OP_HOP_OE, 1)):
        src, dst = packed(lat, "fp64"), packed(lat, "fp64")
        lat.pack("fp64", 1 - p, lex(psi), src)
        lat.apply("fp64", 18, op, src, dst)
        got = torch.zeros_like(lex(psi))
        lat.unpack("fp64", p, dst, got)
        check(got.cpu().reshape(-1, 24).tolist(), exact_hop(u, psi, p, bc))


def lex(psi):
    return synth.to_host_layout(psi).cuda()


def test_relative_error_of_gaussian_fields_is_that_of_fp64_arithmetic():
    """Relative L2 error of a hop (the figure in csrc/fixed64.cuh), in fixed point and, with links scaled off SU(3), in
    FP64 arithmetic; run with -s to print them."""
    dims, bc = (4, 2, 4, 4), (1, 1, 1, -1)
    u, psi = fields(dims, "gauss")
    err = []
    for links in (u, u * (1.0 + 1e-5)):
        lat = lattice(links, 0.1, dims, bc)
        src, dst = packed(lat, "fp64"), packed(lat, "fp64")
        lat.pack("fp64", 1, lex(psi), src)
        lat.apply("fp64", 18, wd.WD_OP_HOP_EO, src, dst)
        got = torch.zeros_like(lex(psi))
        lat.unpack("fp64", 0, dst, got)
        got = got.cpu().reshape(-1, 24).tolist()
        want = exact_hop(links, psi, 0, bc)
        num = sum((F(got[s][i]) - v) ** 2 for s, r in want.items() for i, (v, _) in enumerate(r))
        err.append((float(num) / float(sum(v * v for r in want.values() for v, _ in r))) ** 0.5)
    print("relative L2 error: fixed point %.3e, FP64 arithmetic %.3e" % tuple(err))
    assert err[0] <= err[1] <= 2e-16


@pytest.mark.parametrize("dims,split", [((2, 2, 4, 4), (3,)), ((4, 2, 2, 6), (0, 3)), ((2, 4, 4, 2), (1, 2))])
def test_split_hop_takes_its_scale_from_its_own_neighbours(dims, split):
    """Interior hop of a sub-lattice whose field is larger on one face: the sites of the opposite face, whose hops
    across the face are left out, keep their accuracy."""
    u = synth.gauge_random(dims, 0.5, seed=5)
    psi = synth.gaussian_source(dims, seed=6)
    for mu in split:
        face = [slice(None)] * 4
        face[3 - mu] = 0
        psi[tuple(face)] *= 1e9
    # sites of the opposite faces with no neighbour of their own on a face that is larger
    lx, ly, lz, _ = dims

    def checked(s):
        c = [s % lx, (s // lx) % ly, (s // (lx * ly)) % lz, s // (lx * ly * lz)]
        return all(c[mu] > 1 for mu in split) and any(c[mu] == dims[mu] - 1 for mu in split)
    bc = (1, 1, 1, -1)
    lat = lattice(u, 0.1, dims, bc)
    grid = [2 if mu in split else 1 for mu in range(4)]
    lat.dd_set_partition(grid, (0, 0, 0, 0))
    for p in (0, 1):
        src, dst = packed(lat, "fp64"), packed(lat, "fp64")
        lat.pack("fp64", 1 - p, lex(psi), src)
        lat.dd_hop_interior("fp64", 18, p, src, None, 1.0, 0.0, dst)
        got = torch.zeros_like(lex(psi))
        lat.unpack("fp64", p, dst, got)
        want = {s: w for s, w in exact_hop(u, psi, p, bc, split).items() if checked(s)}
        assert want
        check(got.cpu().reshape(-1, 24).tolist(), want)
