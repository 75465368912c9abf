"""What the speed of this framework is measured on: single operator applications, link construction, whole overlap
applications and one differentiated step, each through the entry point that a program calls.

Every case holds a lattice (lx, ly, lz, lt), a number of right-hand sides and options.  Gauge fields are seeded SU(3)
fields exp(i eps Q) with the width that gives a mean plaquette near 0.6 after three stout steps of 0.1 (the field of the
benchmark's workload); sources are complex Gaussian, or the 12 spin-colour point sources.  ``exact`` restates the
operators in plain torch in 64 bits: path-averaged links by their last hop, the hypercube stencil by rolled fields, the
clover term from its four leaves, the rational by dense shifted solves on small lattices.
"""
from __future__ import annotations

import itertools
import math

import torch

import paper_1701_00726_gb300 as bri

EPS = 0.927  # width of the links before smearing: mean plaquette 0.6 after three stout steps of 0.1
SMEAR = 0.1
SMEAR_STEPS = 3
M0 = -1.0  # the overlap's kernel sits at m0 = -rho, rho = 1
FLOPS_BRI = 30168  # per site and right-hand side, both from the operator's definition
FLOPS_WIL = 1368
DENSE_SITES = 384  # largest lattice on which the rational is solved densely


# ------------------------------------------------------------------ the cases
def _case(op, dims, **kw):
    c = {"op": op, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3]}
    c.update(kw)
    return c


def listed():
    return [
        # one operator on a lattice of the test suite's size, one source: launch latency (a call in an interactive check)
        _case("bri", (4, 4, 4, 4), nrhs=1, prec="f32", dagger=False, c_sw=0.0, name="bri_f32_4x4x4x4_1"),
        # the benchmark's lattice, one source, clover: the solver's operator when a single system is left, bound by links
        _case("bri", (24, 24, 24, 48), nrhs=1, prec="f32", dagger=False, c_sw=1.0, name="bri_f32_24x24x24x48_1"),
        # the 12 spin-colour sources of a propagator on the batched workload's main lattice: links shared by sources
        _case("bri", (16, 16, 16, 32), nrhs=12, prec="f32", dagger=True, c_sw=1.0, name="bri_f32_16x16x16x32_12"),
        # BF16-stored links, odd extents, an odd number of sources, no clover
        _case("bri", (18, 15, 14, 21), nrhs=3, prec="bf16", dagger=False, c_sw=0.0, name="bri_bf16_18x15x14x21_3"),
        # the FP64 operator of residuals, final applications and the massive solves
        _case("bri", (16, 16, 16, 32), nrhs=1, prec="f64", dagger=True, c_sw=1.0, name="bri_f64_16x16x16x32_1"),
        # the double-word FP32 operator that forms the mixed solver's residuals
        _case("bri", (16, 16, 16, 32), nrhs=4, prec="dw", dagger=False, c_sw=1.0, name="bri_dw_16x16x16x32_4"),
        # the Wilson kernel next to it, at the benchmark's size
        _case("wil", (24, 24, 24, 48), nrhs=2, prec="f32", dagger=False, c_sw=1.0, name="wil_f32_24x24x24x48_2"),
        # preparing a configuration: 80 path-averaged links and the clover term, then reading the stored links back
        _case("links", (16, 16, 16, 32), c_sw=1.0, name="links_16x16x16x32"),
        # the plain FP64 overlap on the smallest configuration: 12 Gaussian sources, Kenney-Laub order 8
        _case("overlap", (4, 4, 4, 4), nrhs=12, prec="f64", order=8, tol=1e-12, c_sw=0.0, name="overlap_f64_4x4x4x4_12"),
        # the benchmark's mixed-precision workload (4 sources, order 16, 1e-10, clover) on the 16^3 x 32 lattice
        _case("overlap", (16, 16, 16, 32), nrhs=4, prec="f32", order=16, tol=1e-10, c_sw=1.0,
              name="overlap_mixed_16x16x16x32_4"),
        # independent configurations of uneven volume in one call: 12 point sources on the largest, one elsewhere
        _case("batch", (8, 8, 8, 16), nrhs=12, prec="f32", order=12, tol=1e-10, c_sw=1.0, more="8x8x8x8 12x12x12x12 8x8x8x24",
              name="batch_mixed_8x8x8x16_12"),
        # one differentiated step (links, overlap, and the gradient for source and links), mixed, order 12
        _case("step", (16, 16, 16, 16), nrhs=1, prec="f32", order=12, tol=1e-10, c_sw=0.0, name="step_mixed_16x16x16x16_1"),
    ]


def _dims(rng, lo, hi, least=2):
    """Four extents whose product is about log-uniform in [lo, hi]; odd extents as likely as even ones."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = v ** 0.25
    d = [max(least, round(side * math.exp(rng.uniform(-0.35, 0.35)))) for _ in range(3)]
    d.append(max(least, round(v / (d[0] * d[1] * d[2]))))
    while d[0] * d[1] * d[2] * d[3] > hi:
        d[d.index(max(d))] -= 1
    return tuple(d)


def draw(rng):
    op = rng.choice(["bri", "bri", "bri", "bri", "wil", "links", "overlap", "overlap", "batch", "step"])
    c_sw = rng.choice([0.0, 1.0])
    if op in ("bri", "wil"):
        prec = rng.choice(["f32", "f32", "bf16", "f64", "dw"] if op == "bri" else ["f32", "f64"])
        nrhs = rng.choice([1, 1, 2, 3, 4, 5, 7, 8, 12])
        most = {"f64": 131072, "dw": 524288}.get(prec, 1572864) // nrhs
        return _case(op, _dims(rng, 128, min(most, 663552)), nrhs=nrhs, prec=prec, dagger=rng.choice([False, True]), c_sw=c_sw)
    if op == "links":
        return _case(op, _dims(rng, 256, 131072), c_sw=c_sw)
    if op == "overlap":
        prec = rng.choice(["f32", "f32", "f64"])
        nrhs = rng.choice([1, 2, 3, 4, 12])
        most = 3072 if prec == "f64" else 524288
        return _case(op, _dims(rng, 64, most // nrhs), nrhs=nrhs, prec=prec, order=rng.choice([4, 8, 12, 16]),
                     tol=1e-12 if prec == "f64" else 1e-10, c_sw=c_sw)
    if op == "batch":
        nrhs = rng.choice([1, 3, 4, 12])
        more = " ".join("x".join(map(str, _dims(rng, 256, 16384))) for _ in range(rng.choice([1, 2, 4])))
        return _case(op, _dims(rng, 256, 98304 // nrhs), nrhs=nrhs, prec="f32", order=rng.choice([8, 12]), tol=1e-10, c_sw=c_sw,
                     more=more)
    return _case(op, _dims(rng, 128, 65536, 3), nrhs=1, prec="f32", order=rng.choice([8, 12]), tol=1e-10, c_sw=c_sw)


def _lattices(case):
    """[(dims, number of sources)] of a case: one, or the batch's."""
    out = [((case["lx"], case["ly"], case["lz"], case["lt"]), case.get("nrhs", 0))]
    for text in case.get("more", "").split():
        out.append((tuple(int(v) for v in text.split("x")), 1))
    return out


# ------------------------------------------------------------------ inputs
def _roll(f, mu, s):
    """Field value at n + s e_mu of a field with leading axes (t, z, y, x)."""
    return torch.roll(f, -s, dims=3 - mu)


def _dag(m):
    return m.transpose(-1, -2).conj()


def _mm(a, b):
    """Products of 3x3 (or 3xN) matrices, field by field."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _expi(h):
    """exp(i h) of traceless Hermitian h with a moderate norm: scaled Taylor series, squared back."""
    a = 1j * h / 16.0
    eye = torch.eye(3, dtype=h.dtype, device=h.device)
    out = eye + a / 10.0
    for k in range(9, 0, -1):
        out = eye + _mm(a, out) / k
    for _ in range(4):
        out = _mm(out, out)
    return out


def _generators():
    lam = torch.zeros((8, 3, 3), dtype=torch.complex128)
    for a, (i, j) in enumerate([(0, 1), (0, 2), (1, 2)]):
        lam[2 * a, i, j] = lam[2 * a, j, i] = 1
        lam[2 * a + 1, i, j], lam[2 * a + 1, j, i] = -1j, 1j
    lam[6, 0, 0], lam[6, 1, 1] = 1, -1
    lam[7] = torch.diag(torch.tensor([1, 1, -2], dtype=torch.complex128)) / math.sqrt(3.0)
    return lam.cuda()


def _gauge(dims, gen):
    """SU(3) links [Lt, Lz, Ly, Lx, 4, 3, 3], exp(i eps Q) followed by isotropic stout smearing."""
    lx, ly, lz, lt = dims
    w = torch.randn((lt, lz, ly, lx, 4, 8), dtype=torch.float64, device="cuda", generator=gen)
    q = (w.to(torch.complex128) @ _generators().reshape(8, 9)).reshape(w.shape[:-1] + (3, 3)) * 0.5
    u = _expi(EPS * q)
    eye = torch.eye(3, dtype=u.dtype, device="cuda")
    for _ in range(SMEAR_STEPS):
        new = torch.empty_like(u)
        for mu in range(4):
            um = u[..., mu, :, :]
            staple = torch.zeros_like(um)
            for nu in range(4):
                if nu == mu:
                    continue
                un = u[..., nu, :, :]
                staple += _mm(_mm(un, _roll(um, nu, 1)), _dag(_roll(un, mu, 1)))
                back = _roll(un, nu, -1)
                staple += _mm(_mm(_dag(back), _roll(um, nu, -1)), _roll(back, mu, 1))
            om = SMEAR * _mm(staple, _dag(um))
            q = 0.5j * (_dag(om) - om)
            q = q - q.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] * eye / 3.0
            new[..., mu, :, :] = _mm(_expi(0.5 * (q + _dag(q))), um)
        u = new
    return u.contiguous()


def _sources(dims, nrhs, gen, dtype, point=False):
    lx, ly, lz, lt = dims
    shape = (nrhs, lt, lz, ly, lx, 4, 3)
    if point:  # spin-colour unit vectors at one site
        x = torch.zeros(shape, dtype=dtype, device="cuda")
        at = [int(torch.randint(0, n, (1,), device="cuda", generator=gen)) for n in (lt, lz, ly, lx)]
        for r in range(nrhs):
            x[r, at[0], at[1], at[2], at[3], (r // 3) % 4, r % 3] = 1.0
        return x
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=gen).to(dtype)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    wide = case.get("prec") in ("f64", "dw") or case["op"] in ("overlap", "batch", "step")
    dtype = torch.complex128 if wide else torch.complex64
    out = []
    for i, (dims, nrhs) in enumerate(_lattices(case)):
        u = _gauge(dims, gen)
        x = _sources(dims, nrhs, gen, dtype, case["op"] == "batch" and nrhs == 12) if nrhs else None
        out.append((dims, u, x))
    return out, gen


def prepare(case, seed):
    """The user's arrays and, but for the calls that make them, the lattices with their links."""
    inputs, gen = _inputs(case, seed)
    state = {"case": case, "lats": [], "us": [], "xs": []}
    for dims, u, x in inputs:
        lat = bri.Lattice(dims)
        if case["op"] not in ("links", "step"):
            lat.build_links(u, case["c_sw"])
        state["lats"].append(lat)
        state["us"].append(u if case["op"] in ("links", "step") else None)
        state["xs"].append(x)
    if case["op"] == "step":
        state["eta"] = torch.randn(state["xs"][0].shape, dtype=torch.complex128, device="cuda", generator=gen)
        state["us"][0].requires_grad_(True)
        state["xs"][0].requires_grad_(True)
    return state


# ------------------------------------------------------------------ one pass
def _solver_prec(case):
    return {"f64": bri.PREC_F64, "f32": bri.PREC_F32}[case["prec"]]


def run(state):
    case, lat, x = state["case"], state["lats"][0], state["xs"][0]
    op = case["op"]
    if op == "bri":
        return lat.bri_apply(x, M0, dagger=case["dagger"], bf16_links=case["prec"] == "bf16", double_word=case["prec"] == "dw")
    if op == "wil":
        return lat.wils_apply(x, M0, dagger=case["dagger"])
    if op == "links":
        lat.build_links(state["us"][0], case["c_sw"])
        return lat.links()
    if op == "overlap":
        return lat.overlap_apply(x, case["order"], tol=case["tol"], prec=_solver_prec(case))[0]
    if op == "batch":
        return bri.overlap_apply_batch(state["lats"], state["xs"], case["order"], tol=case["tol"], prec=_solver_prec(case))[0]
    u = state["us"][0]
    y = bri.overlap(x, u, lat, case["order"], tol=case["tol"], prec=_solver_prec(case), c_sw=case["c_sw"])
    return (y.detach(),) + torch.autograd.grad((y,), (x, u), (state["eta"],))


# ------------------------------------------------------------------ what a pass cannot do without
def _iterations(order, tol):
    """CG steps of the smallest shift by the condition-number bound, with the kernel's spectrum in [0, 1.3]."""
    sigma = math.tan(math.pi / (4 * order + 2)) ** 2
    return 0.5 * math.sqrt((1.3 + sigma) / sigma) * math.log(2.0 / tol)


def work(case):
    op = case["op"]
    size = 16 if case.get("prec") in ("f64", "dw") else 8
    byt = flops = 0.0
    for dims, nrhs in _lattices(case):
        v = float(dims[0] * dims[1] * dims[2] * dims[3])
        clover = v * 72 * size / 2 if case["c_sw"] else 0.0
        spinors = v * nrhs * 12 * size * 2
        if op == "bri":
            byt += v * 360 * (4 if case["prec"] == "bf16" else size) + clover + spinors
            flops += v * nrhs * FLOPS_BRI
        elif op == "wil":
            byt += v * 36 * size + clover + spinors
            flops += v * nrhs * FLOPS_WIL
        elif op == "links":  # thin links in, the three stored copies and the clover term out, and the copy handed back
            byt += v * (36 * 16 + 360 * (16 + 8 + 4) + 2 * 360 * 16) + (v * 72 * 12 if case["c_sw"] else 0.0)
            flops += v * 208 * 198  # one 3x3 product for every last hop of every offset
        else:
            it = _iterations(case["order"], case["tol"]) * (2 if op == "step" else 1)
            byt += 2 * it * (v * 360 * size + clover + spinors)
            flops += 2 * it * v * nrhs * FLOPS_BRI * (2 if op == "step" else 1)
    return {"bytes": byt, "flops": flops}


# ------------------------------------------------------------------ the same in plain 64-bit torch
def _gammas():
    s = [[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]]
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    for k in range(3):
        p = torch.tensor(s[k], dtype=torch.complex128)
        g[k, :2, 2:], g[k, 2:, :2] = -1j * p, 1j * p
    g[3, :2, 2:] = g[3, 2:, :2] = torch.eye(2, dtype=torch.complex128)
    return g.cuda()


def _g5(x):
    return x * torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=x.device).view(4, 1)


def _offsets():
    """The 81 offsets (dx, dy, dz, dt), x fastest."""
    return [tuple(reversed(d)) for d in itertools.product((-1, 0, 1), repeat=4)]


def _transporters(u):
    """Average over the shortest paths of every offset, grouped by their last hop."""
    w = {(0, 0, 0, 0): torch.eye(3, dtype=u.dtype, device=u.device).expand(u.shape[:4] + (3, 3))}
    for d in sorted(_offsets(), key=lambda d: sum(map(abs, d)))[1:]:
        hops = [mu for mu in range(4) if d[mu]]
        acc = 0
        for mu in hops:
            before = tuple(0 if k == mu else v for k, v in enumerate(d))
            step = u[..., mu, :, :] if d[mu] > 0 else _dag(_roll(u[..., mu, :, :], mu, -1))
            for k in range(4):
                if before[k]:
                    step = _roll(step, k, before[k])
            acc = acc + _mm(w[before], step)
        w[d] = acc / len(hops)
    return w


def _clover(u, c_sw):
    """-(c_sw/2) sum sigma F as a matrix field [t, z, y, x, 4, 3, 4, 3]."""
    g = _gammas()
    c = torch.zeros(u.shape[:4] + (4, 3, 4, 3), dtype=u.dtype, device=u.device)
    for mu, nu in itertools.combinations(range(4), 2):
        um, un = u[..., mu, :, :], u[..., nu, :, :]
        plaq = _mm(_mm(um, _roll(un, mu, 1)), _mm(_dag(_roll(um, nu, 1)), _dag(un)))  # from n, counter-clockwise
        q = plaq
        # the leaf of n - mu, moved so that it starts and ends at n, and so on round the clover
        um_m, un_m, um_n, un_n = _roll(um, mu, -1), _roll(un, mu, -1), _roll(um, nu, -1), _roll(un, nu, -1)
        q = q + _mm(_mm(un, _dag(_roll(um_m, nu, 1))), _mm(_dag(un_m), um_m))
        q = q + _mm(_mm(_dag(um_m), _dag(_roll(un_m, nu, -1))), _mm(_roll(um_m, nu, -1), un_n))
        q = q + _mm(_mm(_dag(un_n), um_n), _mm(_roll(un_n, mu, 1), _dag(um)))
        f = (q - _dag(q)) / 8j
        f = f - f.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] * torch.eye(3, dtype=u.dtype, device=u.device) / 3.0
        sig = 0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])
        c += -0.5 * c_sw * torch.einsum("st,...ab->...satb", sig, f)
    return c


class _Plain:
    """D of either kernel at m0 = -1 on one gauge field."""

    def __init__(self, u, kernel, c_sw):
        self.c = _clover(u, c_sw) if c_sw else None
        g, one = _gammas(), torch.eye(4, dtype=u.dtype, device=u.device)
        w = _transporters(u)
        self.terms = []
        for d in _offsets():
            k = sum(map(abs, d))
            if kernel == "bri":
                lap = 2.0 ** (4 - k) / 64.0 - (4.0 if k == 0 else 0.0)
                m = (-0.5 * lap + (M0 if k == 0 else 0.0)) * one
                for mu in range(4):
                    m = m + d[mu] * 4.0 ** (4 - k) / 432.0 * g[mu]
            elif k == 0:
                m = (4.0 + M0) * one
            elif k == 1:
                mu = [i for i in range(4) if d[i]][0]
                m = -0.5 * one + 0.5 * d[mu] * g[mu]
            else:
                continue
            self.terms.append((d, m, w[d]))

    def __call__(self, x, dagger=False):
        if dagger:
            return _g5(self(_g5(x)))
        y = torch.zeros_like(x)
        for d, m, w in self.terms:
            xs = x
            shifts = [-d[mu] for mu in (3, 2, 1, 0)]
            if any(shifts):
                xs = torch.roll(xs, shifts, dims=(1, 2, 3, 4))
            xs = torch.einsum("st,...ta->...sa", m, xs)
            y += (w.unsqueeze(-3) * xs.unsqueeze(-2)).sum(-1)
        if self.c is not None:
            y += torch.einsum("...satb,r...tb->r...sa", self.c, x)
        return y


def _rational(n):
    """f(x) = x (c0 + sum w / (x^2 + sigma)), Kenney-Laub order n."""
    t = [(2 * i + 1) * math.pi / (4 * n + 2) for i in range(n)]
    return 1.0 / (2 * n + 1), [2.0 / ((2 * n + 1) * math.cos(a) ** 2) for a in t], [math.tan(a) ** 2 for a in t]


def _overlap(u, x, order, c_sw):
    """x + D (c0 + sum w (D^+ D + sigma)^-1) x with dense matrices."""
    plain = _Plain(u, "bri", c_sw)
    dim = x[0].numel()
    eye = torch.eye(dim, dtype=torch.complex128, device="cuda").reshape((dim,) + x.shape[1:])
    d = torch.cat([plain(part).reshape(-1, dim) for part in eye.split(256)]).T.contiguous()
    a = d.conj().T @ d
    b = x.reshape(x.shape[0], dim).T
    c0, ws, sigmas = _rational(order)
    acc = c0 * b
    one = torch.eye(dim, dtype=torch.complex128, device="cuda")
    for w, s in zip(ws, sigmas):
        acc = acc + w * torch.linalg.solve(a + s * one, b)
    return x + (d @ acc).T.reshape(x.shape)


def exact(case, seed):
    op = case["op"]
    if op == "step":  # a gradient through a solve: no plain restatement that ends in seconds
        return None
    inputs, _ = _inputs(case, seed)
    if op in ("bri", "wil"):
        _, u, x = inputs[0]
        return _Plain(u, op, case["c_sw"])(x.to(torch.complex128), case["dagger"])
    if op == "links":
        w = _transporters(inputs[0][1])
        return torch.stack([w[d].reshape(-1, 3, 3) for d in _offsets()[:40]], dim=1)
    out = []
    for dims, u, x in inputs:
        small = dims[0] * dims[1] * dims[2] * dims[3] <= DENSE_SITES
        out.append(_overlap(u, x, case["order"], case["c_sw"]) if small else None)
    if all(v is None for v in out):
        return None
    return out[0] if op == "overlap" else out
