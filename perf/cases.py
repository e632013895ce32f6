"""Timed cases of the library: its operators, solvers and the learned preconditioner, through the public calls of
``paper_2602_14450_gb300.wd``, and the values they should give, in float64 torch.

A case is one user-level pass on one lattice (x, y, z, t) of a kind:

* ``apply``    one application of an operator (hop, even-odd A, full D_W) to packed vectors, in the storage precision,
               link format and FP16 arithmetic of the case, with or without the clover term, for one or several
               right-hand sides;
* ``solve``    one whole solve of D_W x = b on device vectors;
* ``gauge``    a new gauge field in: set_gauge (with the clover term), then the first low-precision and the first
               FP64 even-odd operator on it;
* ``precond``  one application of the learned preconditioner M;
* ``grad``     loss and weight gradient of M on a mini-batch.
"""

from __future__ import annotations

import math

import torch

from paper_2602_14450_gb300 import synth, wd

BC = (1, 1, 1, -1)
OPS = {"hop_eo": wd.WD_OP_HOP_EO, "hop_oe": wd.WD_OP_HOP_OE, "eo": wd.WD_OP_EO_A, "full": wd.WD_OP_FULL}
DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
SIZE = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
CDT = torch.complex128
C_MID = 12


def _case(name, kind, dims, **more):
    c = {"name": name, "kind": kind, "x": dims[0], "y": dims[1], "z": dims[2], "t": dims[3], "kappa": 0.12}
    c.update(more)
    return c


def _apply(name, dims, prec, recon, op, arith=16, nrhs=1, csw=0.0):
    return _case(name, "apply", dims, prec=prec, recon=recon, op=op, arith=arith, nrhs=nrhs, csw=csw)


def listed():
    return [
        # The inner operator of a small-lattice solve (the 8^4 workload): launches and latency.
        _apply("eo_fp16_8x8x8x8", (8, 8, 8, 8), "fp16", 12, "eo"),
        # The inner operator of the benchmark's solve: FP16 storage and arithmetic, 12-real links, 32^3 x 64.
        _apply("eo_fp16_32x32x32x64", (32, 32, 32, 64), "fp16", 12, "eo"),
        # The inner operator with the clover term in the library's default stencil arithmetic, a medium lattice.
        _apply("eo_clover_fp16_24x24x24x48", (24, 24, 24, 48), "fp16", 12, "eo", arith=32, csw=1.0),
        # The inner operator of the FP32-mixed solve on the 16^3 x 32 workload.
        _apply("eo_fp32_16x16x16x32", (16, 16, 16, 32), "fp32", 12, "eo"),
        # A BF16 hop with full links on a lattice whose extents are no powers of two.
        _apply("hop_bf16_12x20x28x36", (12, 20, 28, 36), "bf16", 18, "hop_eo"),
        # The true residual's operator: the full Wilson matrix in FP64 on the benchmark's lattice.
        _apply("full_fp64_32x32x32x64", (32, 32, 32, 64), "fp64", 18, "full"),
        # The 12 spin-colour sources of a propagator at once, on the batched workload's lattice.
        _apply("eo_fp16_24x24x24x48_12rhs", (24, 24, 24, 48), "fp16", 12, "eo", nrhs=12),
        # The headline: the FP16-mixed solve on the benchmark's lattice to the stopping norm of the paper's Table 2, with
        # a kappa at which the low-precision solver needs about 500 matrix-vector products on these links.
        _case("solve_fp16_32x32x32x64", "solve", (32, 32, 32, 64), scheme="mixed_fp16", arith=16, kappa=0.139,
              tol=1e-13),
        # The FP64 solver: the comparator, and what makes the training samples of M (16^3 x 32, about 400 products).
        _case("solve_fp64_16x16x16x32", "solve", (16, 16, 16, 32), scheme="fp64", arith=16, kappa=0.139,
              tol=1e-13),
        # The next configuration of an ensemble, with the clover term: upload, link formats, clover blocks, first use.
        _case("gauge_clover_24x24x24x48", "gauge", (24, 24, 24, 48), csw=1.0, arith=16),
        # The learned preconditioner inside the FP16 solve on the benchmark's lattice.
        _case("precond_fp16_32x32x32x64", "precond", (32, 32, 32, 64), prec="fp16"),
        # One training step's loss and gradient on the training lattice with the trainer's mini-batch.
        _case("grad_16x16x16x32_4", "grad", (16, 16, 16, 32), samples=4),
    ]


def _dims(rng, lo, hi):
    """Even extents with a volume of lo..hi sites, spread over its logarithm."""
    while True:
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = (want / 2) ** 0.25
        d = [max(4, 2 * round(side * math.exp(rng.uniform(-0.4, 0.4)) / 2)) for _ in range(3)]
        d.append(max(4, 2 * round(want / (d[0] * d[1] * d[2]) / 2)))
        v = d[0] * d[1] * d[2] * d[3]
        if lo <= v <= hi and max(d) <= 96:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["batch"] + ["solve"] * 2 + ["gauge", "precond", "grad"])
    if kind == "apply":
        prec = rng.choice(["fp64", "fp64", "fp32", "fp16", "fp16", "bf16"])
        recon = 18 if prec == "fp64" else rng.choice([12, 18])
        op = rng.choice(["hop_eo", "hop_oe", "eo", "eo", "full"])
        csw = rng.choice([0.0, 0.0, 0.0, 1.0]) if op in ("eo", "full") else 0.0
        hi = 1 << 20 if csw else 1 << 21
        c = _apply("", _dims(rng, 256, hi), prec, recon, op, rng.choice([16, 32]), 1, csw)
    elif kind == "batch":
        c = _apply("", _dims(rng, 256, 1 << 18), rng.choice(["fp16", "fp16", "fp32", "bf16"]), 12,
                   rng.choice(["hop_oe", "eo"]), rng.choice([16, 32]), rng.choice([2, 3, 5, 12]))
    elif kind == "solve":
        scheme = rng.choice(["mixed_fp16", "mixed_fp16", "mixed_fp32", "mixed_bf16", "fp64"])
        c = _case("", "solve", _dims(rng, 1 << 11, 1 << 17), scheme=scheme, arith=rng.choice([16, 32]),
                  tol=1e-12)
    elif kind == "gauge":
        c = _case("", "gauge", _dims(rng, 1 << 10, 1 << 19), csw=rng.choice([0.0, 1.0]), arith=rng.choice([16, 32]))
    elif kind == "precond":
        c = _case("", "precond", _dims(rng, 256, 1 << 20), prec=rng.choice(["fp16", "fp16", "fp32"]))
    else:
        c = _case("", "grad", _dims(rng, 1 << 17, 5 << 16), samples=rng.choice([4, 6, 8]))
    del c["name"]
    return c


# --- inputs -------------------------------------------------------------------------------------------------------

def _size(case):
    return (case["x"], case["y"], case["z"], case["t"])


def _generator(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + what)
    return g


def _links(case, seed):
    """SU(3) links around 1 + i H / 2 with Gaussian H, as the library's rough links; complex [4, t, z, y, x, 3, 3]."""
    x, y, z, t = _size(case)
    n = 4 * x * y * z * t
    g = _generator(seed, 1)
    lam = (synth.gell_mann() / 2).cuda().reshape(8, 9)
    h = torch.randn((n, 8), generator=g, device="cuda", dtype=torch.float64)
    w = torch.complex(-0.5 * (h @ lam.imag), 0.5 * (h @ lam.real)).reshape(n, 3, 3)
    w.diagonal(dim1=-2, dim2=-1).add_(1.0)
    return _su3(w).reshape(4, t, z, y, x, 3, 3)


def _su3(w):
    """Rows 0 and 1 by Gram-Schmidt, row 2 their conjugate cross product."""
    a = w[:, 0] / torch.linalg.vector_norm(w[:, 0], dim=-1, keepdim=True)
    b = w[:, 1] - (a.conj() * w[:, 1]).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], 1)


def _fields(case, seed, count, what=2):
    """`count` Gaussian quark fields, float64 in the lexicographic host layout [count, t, z, y, x, 4, 3, 2]."""
    x, y, z, t = _size(case)
    return torch.randn((count, t, z, y, x, 4, 3, 2), generator=_generator(seed, what), device="cuda",
                       dtype=torch.float64)


def _weights(seed):
    """BF16 weights of M near the identity, as a trained M has them, in float32."""
    w = 0.02 * torch.randn(wd.PRECOND_FLOATS, generator=_generator(seed, 3), device="cuda", dtype=torch.float32)
    one = torch.zeros((2, 9, C_MID, 4, 4, 2), device="cuda")
    one[:, 0, 0, range(4), range(4), 0] = 1.0
    return (w + one.reshape(-1)).to(torch.bfloat16).float().cpu()


def _lattice(case, u):
    lat = wd.Lattice(_size(case), case["kappa"], BC)
    lat.set_gauge(torch.view_as_real(u))
    lat.set_arith(case.get("arith", 32))
    if case.get("csw"):
        lat.set_clover(case["csw"])
    return lat


def _parities(op):
    """(input parities, output parities) of an operator's packed vectors."""
    return {"hop_eo": ([1], [0]), "hop_oe": ([0], [1]), "eo": ([0], [0]), "full": ([0, 1], [0, 1])}[op]


def _packed(lat, prec, parities, f):
    """Packed vectors [count, len(parities) * V/2 * 24] of fields f."""
    n = lat.vector_bytes(prec) // SIZE[prec]
    out = torch.empty((f.shape[0], len(parities), n), dtype=DTYPE[prec], device="cuda")
    for i in range(f.shape[0]):
        for j, p in enumerate(parities):
            lat.pack(prec, p, f[i], out[i, j])
    return out


def prepare(case, seed):
    kind = case["kind"]
    u = _links(case, seed)
    if kind == "gauge":
        lat = _lattice(case, u)
        f = _fields(case, seed, 1)
        s = {"case": case, "lat": lat, "u": torch.view_as_real(u).contiguous()}
        for prec in ("fp16", "fp64"):
            s[prec] = _packed(lat, prec, [0], f)
            s["out_" + prec] = torch.empty_like(s[prec])
        return s
    lat = _lattice(case, u)
    links = u if kind == "grad" else None
    del u
    s = {"case": case, "lat": lat}
    if kind == "apply":
        pi, po = _parities(case["op"])
        s["in"] = _packed(lat, case["prec"], pi, _fields(case, seed, case["nrhs"]))
        s["out"] = torch.empty((case["nrhs"], len(po), s["in"].shape[2]), dtype=s["in"].dtype, device="cuda")
        run(s)   # the packed links and clover blocks are built on first use
    elif kind == "solve":
        s["b"] = _fields(case, seed, 1)[0]
        s["x"] = torch.zeros_like(s["b"])
    elif kind == "precond":
        lat.precond_set(_weights(seed))
        s["in"] = _packed(lat, case["prec"], [0], _fields(case, seed, 1))
        s["out"] = torch.empty_like(s["in"])
        run(s)
    else:
        lat.precond_set(_weights(seed))
        v, y = _samples(case, seed, links)
        s["v"] = _packed(lat, "fp32", [0], v).flatten(1)
        s["y"] = _packed(lat, "fp32", [0], y).flatten(1)
    return s


def _samples(case, seed, u):
    """Training pairs: Gaussian v, and y = v + K v + K K v, K = kappa^2 H_eo H_oe, which A^-1 v is to second order."""
    v = _fields(case, seed, case["samples"])
    y = v.clone()
    for i in range(case["samples"]):
        f = _on(torch.view_as_complex(v[i]), _size(case), 0)
        for _ in range(2):
            f = case["kappa"] ** 2 * _hop(u, _hop(u, f))
            y[i] += torch.view_as_real(f)
    return v, y


def run(s):
    case, lat = s["case"], s["lat"]
    kind = case["kind"]
    if kind == "apply":
        op = OPS[case["op"]]
        if case["nrhs"] == 1:
            lat.apply(case["prec"], case["recon"], op, s["in"], s["out"])
        else:
            lat.apply_batch(case["prec"], case["recon"], op, case["nrhs"], s["in"], s["out"])
        return s["out"]
    if kind == "solve":
        lat.solve(s["b"], s["x"], case["tol"], case["scheme"])
        return s["x"]
    if kind == "gauge":
        lat.set_gauge(s["u"])
        lat.apply("fp16", 12, wd.WD_OP_EO_A, s["fp16"], s["out_fp16"])
        lat.apply("fp64", 18, wd.WD_OP_EO_A, s["fp64"], s["out_fp64"])
        return [s["out_fp16"], s["out_fp64"]]
    if kind == "precond":
        lat.precond_apply(case["prec"], s["in"], s["out"])
        return s["out"]
    loss, grad = lat.precond_grad(s["v"], s["y"], 1.0)
    return [torch.tensor(loss, dtype=torch.float32), grad]


# --- what a pass cannot do without ----------------------------------------------------------------------------------

HOP_FLOPS = 1320.0      # per output site, in this spin basis


def work(case):
    x, y, z, t = _size(case)
    vh = x * y * z * t // 2
    kind = case["kind"]
    if kind == "apply":
        b, n = SIZE[case["prec"]], case["nrhs"]
        sides = len(_parities(case["op"])[0])
        hops = 2 if case["op"] in ("eo", "full") else 1
        links = vh * 8 * case["recon"] * b
        clover = (2 * vh * 80 * b) if case["csw"] else 0
        return {"bytes": 2 * n * sides * vh * 24 * b + links + clover,
                "flops": n * vh * (hops * HOP_FLOPS + (2 * 264 if case["csw"] else 0))}
    if kind == "solve":
        # the links and a vector in and out of every application of A, in the solver's working precision
        b = {"fp64": 8, "mixed_fp32": 4}.get(case["scheme"], 2)
        recon = 18 if case["scheme"] == "fp64" else 12
        n = 500 if case["kappa"] > 0.13 else 50
        return {"bytes": n * vh * (8 * recon + 48) * b + 2 * 2 * vh * 192, "flops": n * vh * 2 * HOP_FLOPS}
    if kind == "gauge":
        extra = 2 * vh * 80 * (2 + 8) if case["csw"] else 0
        return {"bytes": 2 * vh * 4 * 144 + vh * 8 * (12 * 2 + 18 * 8) + 2 * vh * 24 * (2 + 8) + extra,
                "flops": vh * 4 * HOP_FLOPS + (2 * vh * 12 * 12 * 12 * 8 / 3 if case["csw"] else 0)}
    transport = 8 * 4 * 66                                    # 8 links times 4 colour vectors, per site
    if kind == "precond":
        b = SIZE[case["prec"]]
        recon = 12 if b == 2 else 18
        return {"bytes": vh * (2 * 24 + 8 * recon) * b, "flops": vh * (2 * transport + (64 + 9) * 4 * 4 * 3 * 8)}
    layer = 9 * C_MID * 4 * 4 * 3 * 8
    return {"bytes": case["samples"] * vh * 2 * 24 * 4 + vh * 8 * 18 * 4,
            "flops": case["samples"] * vh * 3 * (2 * layer + 2 * layer)}


# --- the same in float64 --------------------------------------------------------------------------------------------

def _gammas():
    s = torch.zeros((3, 2, 2), dtype=CDT)
    s[0] = torch.tensor([[0, 1], [1, 0]])
    s[1] = torch.tensor([[0, -1j], [1j, 0]])
    s[2] = torch.tensor([[1, 0], [0, -1]])
    g = torch.zeros((4, 4, 4), dtype=CDT)
    for k in range(3):
        g[k, :2, 2:] = -1j * s[k]
        g[k, 2:, :2] = 1j * s[k]
    g[3] = torch.diag(torch.tensor([1, 1, -1, -1], dtype=CDT))
    return g.cuda()


def _shift(f, mu, step, phase, first=0):
    """f(x + step mu) with the boundary phase; the lattice axes start at axis `first`."""
    ax = first + 3 - mu
    r = torch.roll(f, -step, ax)
    if phase == 1:
        return r
    sign = torch.ones(f.shape[ax], dtype=torch.float64, device=f.device)
    sign[-1 if step > 0 else 0] = phase
    return r * sign.reshape([-1 if a == ax else 1 for a in range(f.dim())])


def _transports(u, f, first=0):
    """U_mu(x) f(x + mu) and U_mu(x - mu)^+ f(x - mu) for mu = 0..3."""
    for mu in range(4):
        yield mu, 0, _shift(f, mu, 1, BC[mu], first) @ u[mu].transpose(-1, -2)
        yield mu, 1, _shift(f, mu, -1, BC[mu], first) @ _shift(u[mu], mu, -1, 1).conj()


def _hop(u, f):
    g, one, out = _gammas(), torch.eye(4, dtype=CDT, device="cuda"), torch.zeros_like(f)
    for mu, side, h in _transports(u, f):
        out += (one + (g[mu] if side else -g[mu])) @ h
    return out


def _parity(dims):
    x, y, z, t = (torch.arange(d, device="cuda") for d in dims)
    return (t[:, None, None, None] + z[:, None, None] + y[:, None] + x) % 2


def _on(f, dims, p):
    return f * (_parity(dims) == p).to(torch.float64)[..., None, None]


def _clover(u, dims, kappa, csw):
    """C = 1 - csw kappa sum sigma F, [t, z, y, x, 12, 12], and its inverse."""
    g = _gammas()
    c = torch.zeros(u.shape[1:5] + (4, 3, 4, 3), dtype=CDT, device="cuda")
    dag = lambda m: m.conj().transpose(-1, -2)  # noqa: E731
    at = lambda m, mu, s: _shift(m, mu, s, 1)  # noqa: E731
    for mu in range(4):
        for nu in range(mu + 1, 4):
            a, b = u[mu], u[nu]
            am, bm = at(a, mu, -1), at(b, nu, -1)
            q = a @ at(b, mu, 1) @ dag(at(a, nu, 1)) @ dag(b)
            q = q + b @ dag(at(am, nu, 1)) @ dag(at(b, mu, -1)) @ am
            q = q + dag(am) @ dag(at(bm, mu, -1)) @ at(am, nu, -1) @ bm
            q = q + dag(bm) @ at(a, nu, -1) @ at(bm, mu, 1) @ dag(a)
            f = (q - dag(q)) / 8j
            f = f - torch.eye(3, dtype=CDT, device="cuda") * f.diagonal(dim1=-2, dim2=-1).mean(-1)[..., None, None]
            sig = 0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])
            c -= csw * kappa * sig[:, None, :, None] * f[..., None, :, None, :]
    c = c.reshape(u.shape[1:5] + (12, 12)) + torch.eye(12, dtype=CDT, device="cuda")
    return c, torch.linalg.inv(c)


def _block(c, f):
    return (c @ f.reshape(f.shape[:4] + (12, 1))).reshape(f.shape)


def _operator(case, u, f, op, blocks):
    dims, k = _size(case), case["kappa"]
    if op in ("hop_eo", "hop_oe"):
        return _hop(u, f)
    if op == "full":
        return (_block(blocks[0], f) if blocks else f) - k * _hop(u, f)
    h = _on(_hop(u, f), dims, 1)
    h = _hop(u, _block(blocks[1], h) if blocks else h)
    return f - k * k * (_block(blocks[1], h) if blocks else h)


def _lay(case, f, prec, parities):
    """Float64 values of a field's packed vectors, as _packed stores them."""
    x, y, z, t = _size(case)
    k = 16 // SIZE[prec]
    r = torch.view_as_real(f.contiguous()).reshape(-1, 24)
    p = _parity(_size(case)).reshape(-1)
    return torch.stack([r[p == q].reshape(-1, 24 // k, k).transpose(0, 1).reshape(-1) for q in parities])


def _stored(f, prec):
    """A float64 field as it is after storage in `prec`."""
    return torch.view_as_complex(f.to(DTYPE[prec]).to(torch.float64).contiguous())


def _even_odd_solve(case, u, b):
    """x with D_W x = b by BiCGStab on the even-odd system, restarted from the true residual until it stands still."""
    dims, k = _size(case), case["kappa"]
    on = lambda f, p: _on(f, dims, p)  # noqa: E731
    A = lambda f: f - k * k * on(_hop(u, on(_hop(u, f), 1)), 0)  # noqa: E731
    dot = lambda a, c: torch.vdot(a.reshape(-1), c.reshape(-1))  # noqa: E731
    rhs = on(b, 0) + k * on(_hop(u, on(b, 1)), 0)
    x, goal = torch.zeros_like(rhs), 1e-14 * float(torch.linalg.vector_norm(b))
    for _ in range(4):
        r = rhs - A(x)
        if float(torch.linalg.vector_norm(r)) <= goal:
            break
        r0, p, rho, stop = r.clone(), r.clone(), dot(r, r), max(goal / 2, 1e-10 * float(torch.linalg.vector_norm(r)))
        for _ in range(600):
            v = A(p)
            alpha = rho / dot(r0, v)
            s = r - alpha * v
            w = A(s)
            omega = dot(w, s) / dot(w, w)
            x = x + alpha * p + omega * s
            r = s - omega * w
            if float(torch.linalg.vector_norm(r)) <= stop:
                break
            new = dot(r0, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
    return x + on(b, 1) + k * on(_hop(u, x), 1)


def _layer(u, w, f):
    """w [9, out, in, 4, 4] on f [in, t, z, y, x, 4, 3]: hop 0 is the identity, 1 + 2 mu + side a transport."""
    out = torch.einsum("oist,i...tc->o...sc", w[0], f)
    for mu, side, h in _transports(u, f, 1):
        out = out + torch.einsum("oist,i...tc->o...sc", w[1 + 2 * mu + side], h)
    return out


def _network(case, u, w, f):
    """M f for an even-site field; w: the flat complex weights of both layers."""
    w1, w2 = w.reshape(2, 9, C_MID, 4, 4)
    h = _layer(u, w1[:, :, None], f[None])
    return _on(_layer(u, w2[:, None], h)[0], _size(case), 0)


def exact(case, seed):
    kind, dims = case["kind"], _size(case)
    if kind == "solve" and dims[0] * dims[1] * dims[2] * dims[3] > 1 << 17:
        return None     # minutes
    u = _links(case, seed)
    if kind == "solve":
        x = _even_odd_solve(case, u, torch.view_as_complex(_fields(case, seed, 1)[0]))
        return torch.view_as_real(x).contiguous()
    blocks = _clover(u, dims, case["kappa"], case["csw"]) if case.get("csw") else None
    if kind == "apply":
        f, (pi, po), out = _fields(case, seed, case["nrhs"]), _parities(case["op"]), []
        for i in range(case["nrhs"]):
            g = _stored(f[i], case["prec"])
            g = g if len(pi) == 2 else _on(g, dims, pi[0])
            out.append(_lay(case, _operator(case, u, g, case["op"], blocks), case["prec"], po))
        return torch.stack(out)
    if kind == "gauge":
        f = _fields(case, seed, 1)[0]
        return [_lay(case, _operator(case, u, _on(_stored(f, p), dims, 0), "eo", blocks), p, [0])[None]
                for p in ("fp16", "fp64")]
    w = torch.view_as_complex(_weights(seed).double().reshape(-1, 2).contiguous()).cuda()
    if kind == "precond":
        f = _on(_stored(_fields(case, seed, 1)[0], case["prec"]), dims, 0)
        w1, w2 = w.reshape(2, 9, C_MID, 4, 4)
        out = torch.zeros_like(f)
        for c in range(C_MID):      # one hidden channel at a time
            out += _layer(u, w2[:, None, c:c + 1], _layer(u, w1[:, c:c + 1, None], f[None]))[0]
        return _lay(case, out, case["prec"], [0])[None]
    v, y = _samples(case, seed, u)
    total, grad, k = 0.0, torch.zeros_like(w), case["kappa"]
    for i in range(case["samples"]):
        a, b = (_on(_stored(q[i], "fp32"), dims, 0) for q in (v, y))
        leaf = w.clone().requires_grad_(True)
        m = _network(case, u, leaf, a)
        e = _operator(case, u, m, "eo", None)
        e = _on(e, dims, 0) - a
        loss = (m - b).abs().square().sum() / b.abs().square().sum() + e.abs().square().sum() / a.abs().square().sum()
        loss.backward()
        total += float(loss.detach())
        grad += leaf.grad
    return [total, torch.view_as_real(grad).reshape(-1)]
