"""The work a user of this library has it do, as measurable cases.

Each case is one pass through the public entry points: the potential
applies, the boundary operator, the particular solutions, setting a problem
up, the LGF spectrum of a new kappa^2 h^2, and whole solves, on the
geometries of the benchmark, the tests and the serving trace (spheres,
ellipsoids, tori, the star), at the grid sizes the library takes. The seed
picks the data and the level-set function that describes the body (the same
body by another function: the same point sets, so outputs of the same size,
but other boundary points and closure weights).

exact() restates the method in plain float64 torch: the point sets, the
closure, the lattice Green's function by its Bessel integral, zero-padded
FFT convolutions and unpreconditioned GMRES.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2502_05507_gb300 import Context, Problem

F64 = torch.float64
DIRS = ((0, 1), (0, -1), (1, 1), (1, -1), (2, 1), (2, -1))   # (axis, step), the order of the closure rows


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _case(name, call, N, shape, p, kappa2, layer="double", precision="mixed", nrhs=1, shift=0.0):
    c = dict(call=call, N=N, shape=shape, p0=float(p[0]), p1=float(p[1]), p2=float(p[2]), kappa2=float(kappa2),
             layer=layer, precision=precision, nrhs=nrhs, shift=float(shift))
    return dict(name=name, **c) if name else c


def listed():
    sphere, torus = (0.6, 0.0, 0.0), (0.5, 0.2, 0.0)
    return [
        # the operator of a caller's own Krylov loop on the smallest benchmark problem: launches and latency
        _case("operator_n32_f32", "operator", 32, "sphere", sphere, 0.0, "double", "fp32"),
        # the same, float64-accurate, single layer, on a flat body
        _case("operator_n64_df64", "operator", 64, "ellipsoid", (0.7, 0.3, 0.6), 10.0, "single", "df64"),
        # the reference arithmetic (float64 throughout) at the benchmark size
        _case("operator_n128_f64", "operator", 128, "torus", torus, 10.0, "double", "fp64"),
        # the potential on the whole grid, as plotting or coupling to another code needs it
        _case("potential_n128_f32", "potential", 128, "ellipsoid", (0.7, 0.55, 0.45), 0.0, "double", "fp32"),
        # the volume potential of a source given on the whole body
        _case("particular_n128_df64", "particular", 128, "sphere", sphere, 0.0, "double", "df64"),
        # a new geometry: classification, closure, source recipe and preconditioner of a moving body
        _case("setup_n128", "setup", 128, "torus", torus, 10.0),
        # a new kappa^2 h^2: what the first problem of each time step size or grid spacing pays
        _case("spectrum_n128", "spectrum", 128, "none", (0.0, 0.0, 0.0), 10.0),
        # whole solves: the smallest benchmark problem in the default (float64) arithmetic
        _case("solve_n32_f64", "solve", 32, "sphere", sphere, 0.0, "double", "fp64"),
        # the direct formulation, mixed precision
        _case("solve_n64_direct", "solve", 64, "torus", torus, 10.0, "direct", "mixed"),
        # the benchmark's single right-hand side
        _case("solve_n128", "solve", 128, "torus", torus, 10.0, "double", "mixed"),
        # the benchmark's headline: 64 right-hand sides on one geometry
        _case("batch64_n128", "solve", 128, "torus", torus, 0.0, "double", "mixed", 64),
        # the largest grid, a body with no thin axis
        _case("solve_n256_star", "solve", 256, "star", (0.6, 0.1, 0.0), 0.0, "double", "mixed"),
    ]


def draw(rng):
    """A case of the same ranges: bodies as in the serving trace (radii and semi-axes 0.3 to 0.8, tori that fit in
    0.8) or the star, kappa^2 0 or up to 100, every layer and precision; the heavier calls on the smaller grids."""
    shape = rng.choice(["sphere", "ellipsoid", "ellipsoid", "torus", "torus", "star"])
    if shape == "sphere":
        p = (rng.uniform(0.3, 0.8), 0.0, 0.0)
    elif shape == "ellipsoid":
        p = tuple(rng.uniform(0.3, 0.8) for _ in range(3))
    elif shape == "torus":
        r = rng.uniform(0.12, 0.25)
        p = (rng.uniform(0.35, 0.8 - r), r, 0.0)
    else:
        p = (rng.uniform(0.45, 0.65), rng.uniform(0.03, 0.1), 0.0)
    p = tuple(round(v, 4) for v in p)
    shift = round(rng.uniform(-0.5, 0.5), 3)   # the centre, off the grid's by parts of a grid step
    kappa2 = rng.choice([0.0, 10.0, round(math.exp(rng.uniform(0.0, math.log(100.0))), 3)])
    layer = rng.choice(["double", "double", "double", "single", "direct"])
    call = rng.choice(["operator", "operator", "potential", "particular", "box", "setup", "spectrum", "solve", "solve",
                       "batch"])
    N = rng.choice([32, 64, 128, 256])
    if call in ("operator", "potential", "particular"):
        return _case(None, call, N, shape, p, kappa2, layer, rng.choice(["fp32", "fp32", "df64", "fp64"]),
                     shift=shift)
    if call == "box":
        return _case(None, call, min(N, 128), shape, p, kappa2, "double", rng.choice(["df64", "fp64"]), shift=shift)
    if call == "setup":
        return _case(None, call, N, shape, p, kappa2, layer, shift=shift)
    if call == "spectrum":
        return _case(None, call, N, "none", (0.0, 0.0, 0.0), round(rng.uniform(0.1, 100.0), 3))
    if call == "solve":
        precision = rng.choice(["mixed", "mixed", "mixed", "df64", "fp64"]) if N <= 32 else "mixed"
        return _case(None, call, N, shape, p, kappa2, layer if N <= 128 else "double", precision, shift=shift)
    N = min(N, 128)
    nrhs = int(round(math.exp(rng.uniform(math.log(2), math.log(64 if N < 128 else 24)))))
    return _case(None, "solve", N, shape, p, kappa2, "double", "mixed", nrhs, shift)


# ------------------------------------------------------------------ inputs
def _h(case):
    return 2.0 / case["N"]


def _rng(seed):
    return np.random.default_rng(int(seed) & 0x7FFFFFFF)


def _axis(case):
    h = _h(case)
    return -1.0 + 0.5 * h + torch.arange(case["N"], dtype=F64, device=_dev()) * h


def _phi(case, seed):
    """Level-set samples of the body, times a smooth factor between 0.7 and 1.3 that the seed picks."""
    d = [case["shift"] * _h(case) * w for w in (1.0, -0.6, 0.3)]
    a = _axis(case)
    w = _rng(seed).uniform(1.0, 3.0, 3)
    factor = 1.0 + 0.3 * (torch.sin(w[0] * a).view(-1, 1, 1) * torch.cos(w[1] * a).view(1, -1, 1)
                          * torch.cos(w[2] * a).view(1, 1, -1))
    x, y, z = (a - d[0]).view(-1, 1, 1), (a - d[1]).view(1, -1, 1), (a - d[2]).view(1, 1, -1)
    p0, p1, p2 = case["p0"], case["p1"], case["p2"]
    if case["shape"] == "sphere":
        phi = x * x + y * y + z * z - p0 * p0
    elif case["shape"] == "ellipsoid":
        phi = x * x / p0 ** 2 + y * y / p1 ** 2 + z * z / p2 ** 2 - 1.0
    elif case["shape"] == "torus":
        phi = (torch.sqrt(x * x + y * y) - p0) ** 2 + z * z - p1 * p1
    else:   # star: r = p0 + p1 sin(5 theta) cos(3 varphi)
        r = torch.sqrt(x * x + y * y + z * z)
        theta = torch.arccos(torch.clamp(z / torch.where(r > 0, r, torch.ones_like(r)), -1.0, 1.0))
        phi = r - (p0 + p1 * torch.sin(5 * theta) * torch.cos(3 * torch.atan2(y, x)))
    return (phi * factor).contiguous()


def _directions(case, seed):
    a = _rng(seed + 77).standard_normal((case["nrhs"], 3))
    return a / np.linalg.norm(a, axis=1, keepdims=True)


def _source(case, seed):
    """f of u = exp(a . x) on every node, one per right-hand side (paper sign: -Lap u + kappa^2 u = f)."""
    a, ax = _directions(case, seed), _axis(case)
    f = torch.empty((case["nrhs"],) + (case["N"],) * 3, dtype=F64, device=_dev())
    for b in range(case["nrhs"]):
        ex, ey, ez = (torch.exp(float(v) * ax) for v in a[b])
        torch.mul((case["kappa2"] - 1.0) * ex.view(-1, 1, 1) * ey.view(1, -1, 1), ez.view(1, 1, -1), out=f[b])
    return f


def _boundary_data(case, seed, xyz):
    a = torch.as_tensor(_directions(case, seed), dtype=F64, device=xyz.device)
    return torch.exp(a @ xyz.T).contiguous()


def _density(n, seed):
    return torch.as_tensor(_rng(seed + 5).standard_normal(n), dtype=F64, device=_dev())


_context = None


def _ctx():
    global _context
    if _context is None:
        _context = Context(0)
    return _context


def _kappa2_of(case, seed):
    return case["kappa2"] * float(_rng(seed).uniform(0.9, 1.1))


def prepare(case, seed):
    # the library works on its context's stream: the tensors around its calls are made there too
    with torch.cuda.stream(_ctx().stream):
        return _prepare(case, seed)


def _prepare(case, seed):
    ctx, call = _ctx(), case["call"]
    st = dict(case=case, ctx=ctx)
    if call == "spectrum":
        st["s"] = _kappa2_of(case, seed) * _h(case) ** 2
        st["out"] = torch.empty((case["N"] + 1,) * 3, dtype=F64, device=_dev())
        return st
    h = _h(case)
    st["phi"] = _phi(case, seed)
    if call == "setup":
        # the spectrum of this kappa^2 h^2 is in the context from the problems before
        Problem(ctx, st["phi"], h, -1.0 + 0.5 * h, case["kappa2"], case["layer"]).close()
        return st
    prob = st["prob"] = Problem(ctx, st["phi"], h, -1.0 + 0.5 * h, case["kappa2"], case["layer"])
    if call in ("operator", "potential"):
        st["q"] = _density(prob.n_unknowns, seed)
        n = prob.n_unknowns if call == "operator" else (case["N"],) * 3
        st["out"] = torch.empty(n, dtype=F64, device=_dev())
    elif call in ("particular", "box"):
        st["f"] = _source(case, seed)[0]
        st["out"] = torch.empty((case["N"],) * 3, dtype=F64, device=_dev())
    else:
        st["f"] = _source(case, seed)
        st["g"] = _boundary_data(case, seed, prob.boundary_points(like=st["phi"]))
    return st


def run(state):
    with torch.cuda.stream(state["ctx"].stream):
        return _run(state)


def _run(state):
    case = state["case"]
    call, prec = case["call"], case["precision"]
    if call == "spectrum":
        return state["ctx"].lgf_spectrum(case["N"], state["s"], out=state["out"])
    if call == "setup":
        h = _h(case)
        prob = Problem(state["ctx"], state["phi"], h, -1.0 + 0.5 * h, case["kappa2"], case["layer"])
        points = prob.boundary_points(like=state["phi"])
        sizes = (prob.n_gm, prob.n_gp, prob.n_mp)
        prob.close()
        return points, sizes
    prob = state["prob"]
    if call == "solve":
        if case["nrhs"] == 1:
            density, u, _ = prob.solve(state["f"][0], state["g"][0], precision=prec)
        else:
            density, u, _ = prob.solve_batched(state["f"], state["g"], precision=prec)
        return density, u
    if call == "operator":
        v = prob.boundary_apply(state["q"], prec, out=state["out"])
    elif call == "potential":
        v = prob.potential_apply(state["q"], prec, out=state["out"])
    elif call == "particular":
        v = prob.particular(state["f"], prec, out=state["out"])
    else:
        v = prob.box_particular(state["f"], prec, out=state["out"])
    # a float32 apply carries 24 bits: its caller keeps it as float32
    return v.float() if prec == "fp32" else v


# -------------------------------------------------- the method in float64
def _shift(a, axis, step, fill):
    """out[x] = a[x + step] along `axis`, `fill` where that leaves the grid."""
    out = torch.full_like(a, fill)
    N = a.shape[axis]
    lo, hi = (0, N - 1) if step == 1 else (1, N)
    out.narrow(axis, lo, hi - lo).copy_(a.narrow(axis, lo + step, hi - lo))
    return out


class _Sets:
    """Point sets, closure rows and boundary points of level-set samples."""

    def __init__(self, phi, h):
        N = phi.shape[0]
        self.N, inside = N, phi < 0
        near = torch.zeros_like(inside)
        out_near = torch.zeros_like(inside)
        for ax, d in DIRS:
            near |= _shift(inside, ax, d, False)
            out_near |= _shift(~inside, ax, d, True)
        self.inside, self.gm_mask = inside, ~inside & near
        self.nplus = inside | self.gm_mask
        self.gm = torch.nonzero(self.gm_mask.reshape(-1)).reshape(-1)
        self.gp = torch.nonzero((inside & out_near).reshape(-1)).reshape(-1)
        self.n_mp = int(inside.sum())
        flat, pm = phi.reshape(-1), phi.reshape(-1)[self.gm]
        self.stride = (N * N, N, 1)
        best = torch.full_like(pm, -math.inf)
        partner = torch.zeros_like(self.gm)
        for ax, d in DIRS:   # the crossing nearest the node, the first direction on ties
            lin = self.gm + d * self.stride[ax]
            pp = flat[lin]
            t = torch.where(pp < 0, pp / (pp - pm), torch.full_like(pp, -math.inf))
            take = t > best
            best, partner = torch.where(take, t, best), torch.where(take, lin, partner)
        self.t, self.partner = best, partner
        o = -1.0 + 0.5 * h
        xm, xp = (torch.stack([o + (v // (N * N)).to(F64) * h, o + (v // N % N).to(F64) * h, o + (v % N).to(F64) * h], 1)
                  for v in (self.gm, partner))
        self.points = xp + best[:, None] * (xm - xp)

    def closure(self, v):
        v = v.reshape(-1)
        return self.t * v[self.gm] + (1.0 - self.t) * v[self.partner]


@functools.lru_cache(maxsize=1)
def _bessel(n, dev):
    """Nodes t = e^u of the trapezoid rule in u, their weights t du, and exp(-2t) I_k(2t) for k < n: the mean of
    exp(2t (cos x - 1)) cos(k x) over equidistant x where 2t is moderate, the large-argument series beyond."""
    du = 0.25
    u = torch.arange(-40.0, 80.0, du, dtype=F64, device=dev)
    t = torch.exp(u)
    k = torch.arange(n, dtype=F64, device=dev)
    rows = torch.empty((n, t.numel()), dtype=F64, device=dev)
    small = 2 * t < 1e5
    M = 3400
    j = torch.arange(M // 2 + 1, dtype=F64, device=dev)
    w = torch.full_like(j, 2.0 / M)
    w[0] = w[-1] = 1.0 / M
    e = torch.exp(-4 * t[small][None, :] * torch.sin(math.pi * j / M)[:, None] ** 2)
    kj = torch.remainder(k[:, None] * j[None, :], M)
    rows[:, small] = (torch.cos(2 * math.pi * kj / M) * w) @ e
    x = 2 * t[~small]
    term = torch.ones((n, x.numel()), dtype=F64, device=dev)
    acc = term.clone()
    for i in range(1, 24):
        term = term * (-(4 * k[:, None] ** 2 - (2 * i - 1) ** 2) / (8 * i * x))
        acc += term
    rows[:, ~small] = acc / torch.sqrt(2 * math.pi * x)
    return t, t * du, rows


def _lgf(n, s):
    """G_s on the offsets 0 <= i, j, k < n: the integral of exp(-s t) times three scaled Bessel functions of 2t."""
    t, wt, rows = _bessel(n, _dev())
    weighted = rows * (wt * torch.exp(-s * t))
    g = torch.empty((n, n, n), dtype=F64, device=rows.device)
    for i in range(n):
        g[i] = (weighted * rows[i]) @ rows.T
    return g


def _smooth(n):
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1 and n % 2 == 0:
            return n
        n += 1


class _Conv:
    """v = G_s * rho for sources and targets in one box of the grid (the whole grid when `whole`)."""

    def __init__(self, sets, s, whole):
        N = sets.N
        box = []
        for ax in range(3):
            if whole:
                box.append((0, N))
            else:
                on = torch.nonzero(sets.nplus.any(dim=(ax + 1) % 3, keepdim=True).any(dim=(ax + 2) % 3, keepdim=True).reshape(-1))
                box.append((max(0, int(on.min()) - 1), min(N, int(on.max()) + 2)))
        self.N, self.box = N, tuple(slice(a, b) for a, b in box)
        self.ext = [b - a for a, b in box]
        self.L = [_smooth(2 * e) for e in self.ext]
        g = _lgf(max(self.ext), s)
        idx = []
        for e, L in zip(self.ext, self.L):
            i = torch.arange(L, device=g.device)
            idx.append(torch.clamp(torch.minimum(i, L - i), max=e - 1))
        emb = g[idx[0]][:, idx[1]][:, :, idx[2]]
        self.hat = torch.fft.rfftn(emb).real.contiguous()

    def __call__(self, rho):
        r = torch.fft.rfftn(rho.reshape((self.N,) * 3)[self.box], s=self.L)
        r *= self.hat
        v = torch.fft.irfftn(r, s=self.L)
        out = torch.zeros((self.N,) * 3, dtype=F64, device=rho.device)
        out[self.box] = v[:self.ext[0], :self.ext[1], :self.ext[2]]
        return out


class _Method:
    def __init__(self, case, seed, whole=False):
        self.case, self.h = case, _h(case)
        self.s = case["kappa2"] * self.h ** 2
        self.sets = _Sets(_phi(case, seed), self.h)
        self.conv = _Conv(self.sets, self.s, whole)
        S = self.sets
        if case["layer"] == "direct":
            number = torch.zeros(S.N ** 3, dtype=torch.int64, device=S.gm.device)
            number[S.gp] = torch.arange(S.gp.numel(), device=S.gm.device)
            self.partner_unknown = S.gm.numel() + number[S.partner]

    @property
    def n(self):
        S = self.sets
        return S.gm.numel() + (S.gp.numel() if self.case["layer"] == "direct" else 0)

    def rho(self, q):
        S, layer = self.sets, self.case["layer"]
        r = torch.zeros(S.N ** 3, dtype=F64, device=q.device)
        if layer == "single":
            r[S.gm] = q
        elif layer == "double":
            count = torch.zeros_like(q)
            for ax, d in DIRS:
                lin = S.gm + d * S.stride[ax]
                out = ~S.nplus.reshape(-1)[lin]
                count += out
                r.index_add_(0, lin[out], -q[out])
            r[S.gm] += torch.where(count > 0, count, torch.ones_like(count)) * q
        else:
            r[torch.cat([S.gm, S.gp])] = q
            w = r.view((S.N,) * 3)
            lw = (6.0 + self.s) * w
            for ax, d in DIRS:
                lw = lw - _shift(w, ax, d, 0.0)
            r = torch.where(S.inside, torch.zeros_like(lw), lw).reshape(-1)
        return r

    def volume(self, f):
        return self.conv(torch.where(self.sets.inside, self.h ** 2 * f, torch.zeros_like(f)))

    def operator(self, q):
        S = self.sets
        if self.case["layer"] != "direct":
            return S.closure(self.conv(self.rho(q)))
        n = S.gm.numel()
        v = self.conv(self.rho(q)).reshape(-1)
        return torch.cat([S.t * q[:n] + (1.0 - S.t) * q[self.partner_unknown], q[n:] - v[S.gp]])

    def gmres(self, b, tol=1e-13, most=400):
        beta = torch.linalg.norm(b)
        V = torch.empty((most + 1, b.numel()), dtype=F64, device=b.device)
        H = np.zeros((most + 1, most))
        V[0] = b / beta
        for j in range(most):
            w = self.operator(V[j])
            hj = torch.zeros(j + 1, dtype=F64, device=b.device)
            for _ in range(2):
                c = V[:j + 1] @ w
                w = w - c @ V[:j + 1]
                hj += c
            hn = float(torch.linalg.norm(w))
            H[:j + 1, j], H[j + 1, j] = hj.cpu().numpy(), hn
            V[j + 1] = w / hn
            if j % 8 == 7 or j + 1 == most:
                e = np.zeros(j + 2)
                e[0] = 1.0
                y, _, _, _ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
                if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) < tol:
                    break
        return beta * (torch.as_tensor(y, dtype=F64, device=b.device) @ V[:j + 1])

    def solve(self, f, g):
        S, direct = self.sets, self.case["layer"] == "direct"
        up = self.volume(f)
        b = torch.cat([g, up.reshape(-1)[S.gp]]) if direct else g - S.closure(up)
        q = self.gmres(b)
        u = torch.where(S.nplus, up + self.conv(self.rho(q)), torch.zeros_like(up)).reshape(-1)
        if direct:
            u[S.gm] = q[:S.gm.numel()]
        return q, u.reshape((S.N,) * 3)


def _box_particular(case, seed):
    """The 7-point problem with zero values on the layers 0 and N: odd extension and the periodic FFT."""
    N, h = case["N"], _h(case)
    S = _Sets(_phi(case, seed), h)
    f = _source(case, seed)[0]
    r = torch.where(S.inside, h * h * f, torch.zeros_like(f))
    for ax in range(3):
        zero = torch.zeros_like(r.narrow(ax, 0, 1))
        r = torch.cat([zero, r.narrow(ax, 1, N - 1), zero, -r.narrow(ax, 1, N - 1).flip(ax)], ax)
    c = torch.cos(math.pi * torch.arange(2 * N, dtype=F64, device=r.device) / N)
    d = (6.0 + case["kappa2"] * h * h) - 2 * (c.view(-1, 1, 1) + c.view(1, -1, 1) + c[:N + 1].view(1, 1, -1))
    x = torch.fft.rfftn(r) * torch.where(d.abs() > 1e-13, 1 / d, torch.zeros_like(d))
    return torch.fft.irfftn(x, s=(2 * N,) * 3)[:N, :N, :N].contiguous()


def _cosine_spectrum(N, s):
    g = _lgf(N, s)
    k = torch.arange(N + 1, dtype=F64, device=g.device)
    n = torch.arange(N, dtype=F64, device=g.device)
    C = 2 * torch.cos(math.pi * torch.remainder(k[:, None] * n[None, :], 2 * N) / N)
    C[:, 0] = 1.0
    return torch.einsum("ai,ijk->ajk", C, torch.einsum("bj,ijk->ibk", C, g @ C.T)).contiguous()


def exact(case, seed):
    call = case["call"]
    if call == "spectrum":
        return _cosine_spectrum(case["N"], _kappa2_of(case, seed) * _h(case) ** 2)
    if call == "setup":
        S = _Sets(_phi(case, seed), _h(case))
        return S.points, (S.gm.numel(), S.gp.numel(), S.n_mp)
    if call == "box":
        return _box_particular(case, seed)
    m = _Method(case, seed, whole=call in ("potential", "particular"))
    if call == "operator":
        return m.operator(_density(m.n, seed))
    if call == "potential":
        return m.conv(m.rho(_density(m.n, seed)))
    if call == "particular":
        return m.volume(_source(case, seed)[0])
    f, g = _source(case, seed), _boundary_data(case, seed, m.sets.points)
    out = [m.solve(f[b], g[b]) for b in range(case["nrhs"])]
    if case["nrhs"] == 1:
        return out[0]
    return torch.stack([q for q, _ in out]), torch.stack([u for _, u in out])


# -------------------------------------------------------------------- work
def _fft_flops(extents):
    """One real convolution on the box padded to twice its extents: a forward and an inverse real transform (5/2 n
    log2 n each) and the product."""
    n = 8.0 * extents[0] * extents[1] * extents[2]
    return 5.0 * n * math.log2(n) + n


@functools.lru_cache(maxsize=64)
def _counts(items):
    case = dict(items)
    S = _Sets(_phi(case, 1), _h(case))
    ext = []
    for ax in range(3):
        on = torch.nonzero(S.nplus.any(dim=(ax + 1) % 3, keepdim=True).any(dim=(ax + 2) % 3, keepdim=True).reshape(-1))
        ext.append(int(on.max()) - int(on.min()) + 3)
    return S.gm.numel(), S.gp.numel(), S.n_mp, tuple(ext)


def work(case):
    N, call = case["N"], case["call"]
    n3 = N ** 3
    if call == "spectrum":   # a cosine transform of the (N + 1)^3 table; the table itself has no input
        n = (N + 1.0) ** 3
        return dict(bytes=8 * n, flops=2.5 * 3 * n * math.log2(2 * N))
    n_gm, n_gp, n_mp, ext = _counts(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    n = n_gm + (n_gp if case["layer"] == "direct" else 0)
    if call == "setup":   # the samples in, the boundary points out
        return dict(bytes=8 * (n3 + 3 * n_gm), flops=20.0 * n3)
    if call == "operator":
        return dict(bytes=16 * n, flops=_fft_flops(ext))
    if call == "potential":
        return dict(bytes=8 * (n + n3), flops=_fft_flops((N, N, N)))
    if call in ("particular", "box"):
        return dict(bytes=8 * (n_mp + n3), flops=_fft_flops((N, N, N)))
    # a solve: f on the body and g in, u and the density out; about a dozen operator applies at the default tolerance
    return dict(bytes=8 * case["nrhs"] * (n_mp + n_gm + n3 + n), flops=12 * case["nrhs"] * _fft_flops(ext))
