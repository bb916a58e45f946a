"""The work that is measured: calls of the public API over the sizes and options it is used at.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same
ranges.  ``prepare`` makes what a user's program holds before the call (a
context for one u-v coverage, the data, the iteration state), ``run`` is one
pass through the public entry points, ``work`` the bytes and operations of one
pass and ``exact`` its result in 64 bits from plain torch.

Kinds of case:
  phi    y = Phi x and x = Phi^H v: the measurement operator and its adjoint
         (gridding an observation, predicting visibilities, an outer solver)
  sara   Psi^H x, its reweighted soft threshold, Psi of that (the prior step)
  cg     the x-update: CG steps on (Phi^H Phi + 2I) x = b
  solve  one call that runs the whole method (state, iterations, image)
  sdmm   a kept state: load the data, iterate, reweight, iterate, read the image
         (data stored as complex64 or bf16, SARA or TV prior, one ball or several)
  batch  several uneven problems advanced together
  diff   unrolled SDMM, forward and backward (gradients of both weight sets)
"""
import math

import numpy as np
import torch

from paper_1307_4370_gb300 import autodiff, binding

SIDES = (64, 96, 128, 192, 256, 384, 512, 768, 1024)  # image sides: 2n = 2^a or 3 2^a, four wavelet levels
ISNR_DB = 30.0


def listed():
    return [
        # the smallest image of the tests: launch latency of one operator pair
        {"name": "phi_64", "kind": "phi", "n": 64, "M": 2048, "J": 4, "arcs": 0, "kernel": "kb", "beam": False},
        # an ordinary ragged observation on a 3 2^a grid, with a primary beam
        {"name": "phi_384", "kind": "phi", "n": 384, "M": 250327, "J": 6, "arcs": 0, "kernel": "kb", "beam": True},
        # the largest workload: half of the points on tracks, two per pixel
        {"name": "phi_1024", "kind": "phi", "n": 1024, "M": 2097152, "J": 6, "arcs": 200, "kernel": "kb",
         "beam": False},
        # the prior step on the largest image, all nine bases
        {"name": "sara_1024", "kind": "sara", "n": 1024},
        # ... and on an ordinary 3 2^a one
        {"name": "sara_192", "kind": "sara", "n": 192},
        # the x-update of the 256 x 256 workload
        {"name": "cg_256", "kind": "cg", "n": 256, "M": 65536, "J": 6, "arcs": 0, "kernel": "kb", "iters": 10},
        # a small image solved by the one-call form
        {"name": "solve_64", "kind": "solve", "n": 64, "M": 2048, "J": 4, "arcs": 0, "kernel": "kb", "iters": 50},
        # the 256 x 256 workload, one reweighting
        {"name": "sdmm_256", "kind": "sdmm", "n": 256, "M": 65536, "J": 6, "arcs": 0, "kernel": "kb", "iters": 10,
         "rounds": 2, "data": "c64", "prior": "sara", "blocks": 0},
        # the 1024 x 1024 workload
        {"name": "sdmm_1024", "kind": "sdmm", "n": 1024, "M": 2097152, "J": 6, "arcs": 200, "kernel": "kb",
         "iters": 5, "rounds": 1, "data": "c64", "prior": "sara", "blocks": 0},
        # the TV prior, four data blocks, bf16-stored data, the Gaussian kernel
        {"name": "tv_512", "kind": "sdmm", "n": 512, "M": 235293, "J": 4, "arcs": 0, "kernel": "gauss", "iters": 6,
         "rounds": 1, "data": "bf16", "prior": "tv", "blocks": 4},
        # uneven problems side by side
        {"name": "batch_6", "kind": "batch", "sides": "128,512,192,384,256,128", "M_per_pixel": 0.9, "J": 6,
         "arcs": 0, "kernel": "kb", "iters": 5},
        # gradients of an unrolled solve
        {"name": "diff_256", "kind": "diff", "n": 256, "M": 65536, "J": 6, "arcs": 0, "kernel": "kb", "iters": 6,
         "checkpoint": 3},
    ]


def draw(rng):
    kind = rng.choice(["phi", "phi", "sara", "cg", "solve", "sdmm", "sdmm", "batch", "diff"])
    if kind == "batch":
        count = rng.randint(2, 6)
        return {"kind": kind, "sides": ",".join(str(rng.choice((128, 192, 256, 384, 512))) for _ in range(count)),
                "M_per_pixel": round(rng.uniform(0.2, 1.0), 3), "J": rng.choice((4, 6)), "arcs": 0, "kernel": "kb",
                "iters": rng.randint(2, 4)}
    largest = {"phi": 1024, "sara": 1024, "cg": 768, "solve": 256, "sdmm": 512, "diff": 256}[kind]
    sides = [s for s in SIDES if s <= largest]
    n = rng.choice(sides)
    if kind == "sara":
        return {"kind": kind, "n": n}
    M = int(n * n * math.exp(rng.uniform(math.log(0.2), math.log(2.0))))
    case = {"kind": kind, "n": n, "M": M, "J": rng.choice((2, 4, 4, 6, 6, 6, 8)),
            "arcs": rng.choice((0, n // 5)) if n >= 256 else 0, "kernel": rng.choice(("kb", "kb", "gauss"))}
    if kind == "phi":
        case["beam"] = rng.random() < 0.3
    elif kind == "cg":
        case["iters"] = rng.randint(3, 12)
    elif kind == "solve":
        case["iters"] = rng.randint(5, 40)
    elif kind == "sdmm":
        case.update(iters=rng.randint(2, 6), rounds=rng.choice((1, 2)), data=rng.choice(("c64", "bf16")),
                    prior=rng.choice(("sara", "sara", "tv")), blocks=rng.choice((0, 0, 5)))
    else:
        case.update(iters=rng.randint(2, 4), checkpoint=rng.choice((1, 2, 4)))
    return case


# ---------------------------------------------------------------------------
# Inputs (from the seed alone)
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1307 + int(seed))


def _coverage(case, g):
    """M float32 frequencies in [-pi, pi)^2: a Gaussian variable density without the origin's cell, and
    with ``arcs`` half of the points on circular tracks, in random order."""
    M, n, arcs = case["M"], case["n"], case["arcs"]
    m_arc = M // 2 if arcs else 0
    parts, have = [], 0
    while have < M - m_arc:
        u = torch.randn(2 * (M - m_arc - have) + 64, 2, generator=g, device="cuda", dtype=torch.float64) * (math.pi / 4)
        u = u[(u.abs() < math.pi).all(1) & (u.norm(dim=1) >= 2 * math.pi / n)][:M - m_arc - have]
        parts.append(u)
        have += u.shape[0]
    if m_arc:
        p = torch.rand(3, arcs, generator=g, device="cuda", dtype=torch.float64)
        rad, start, ext = 2 * math.pi / n + p[0] * (math.pi - 2 * math.pi / n), 2 * math.pi * p[1], 0.5 * math.pi * p[2]
        i = torch.arange(m_arc, device="cuda")
        a, per = i % arcs, -(-m_arc // arcs)
        t = start[a] + ext[a] * ((i // arcs) + 0.5) / per
        parts.append(torch.stack([rad[a] * t.cos(), rad[a] * t.sin()], 1))
    u = torch.cat(parts)
    if m_arc:
        u = u[torch.randperm(M, generator=g, device="cuda")]
    top = float(np.nextafter(np.float32(math.pi), np.float32(0)))
    return u.float().clamp(-top, top).contiguous()


def _observe(uv, n, g):
    """Visibilities of a sky of Gaussian sources (their transform in closed form) with noise at 30 dB, complex64,
    and the bound of the l2 ball."""
    K, M = 40, uv.shape[0]
    p = torch.rand(6, K, generator=g, device="cuda", dtype=torch.float64)
    pos = (0.1 + 0.8 * p[:2]) * n - n // 2
    sa, ratio, ang, amp = 1.0 + 5.0 * p[2], 0.3 + 0.7 * p[3], math.pi * p[4], 10.0 ** (-3.0 * p[5])
    sb, ca, sn = sa * ratio, ang.cos(), ang.sin()
    y = torch.empty(M, dtype=torch.complex128, device="cuda")
    for b in range(0, M, 1 << 18):
        u = uv[b:b + (1 << 18)].double()
        q = (u[:, :1] * ca + u[:, 1:] * sn) ** 2 * sa ** 2 + (u[:, 1:] * ca - u[:, :1] * sn) ** 2 * sb ** 2
        mag = amp * sa * sb * (2 * math.pi) * torch.exp(-0.5 * q) / (2 * n)
        y[b:b + (1 << 18)] = torch.polar(mag, -(u @ pos)).sum(1)
    sigma = float(y.norm()) / math.sqrt(M) * 10.0 ** (-ISNR_DB / 20.0)
    y = y + (sigma * math.sqrt(0.5)) * torch.randn(M, 2, generator=g, device="cuda",
                                                    dtype=torch.float64).view(-1, 2).contiguous().view(torch.complex128)[:, 0]
    return y.to(torch.complex64), math.sqrt((2.0 * M + 4.0 * math.sqrt(M)) * sigma * sigma / 2.0)


def _beam(n):
    c = (torch.arange(n, device="cuda", dtype=torch.float64) - n // 2) / n
    return torch.exp(-(c[:, None] ** 2 + c[None, :] ** 2) / (2 * 0.4 ** 2)).float()


def _randc(count, g):
    return torch.randn(count, 2, generator=g, device="cuda").view(torch.complex64)[:, 0].contiguous()


def _members(case):
    """The problems of a batch: one phi-like description each, visibilities uneven."""
    out = []
    for k, side in enumerate(int(s) for s in case["sides"].split(",")):
        M = int(case["M_per_pixel"] * (1.0 - 0.1 * (k % 5)) * side * side) + k
        out.append(dict(n=side, M=M, J=case["J"], arcs=case["arcs"], kernel=case["kernel"]))
    return out


def _inputs(case, seed):
    """Everything random of one case: arrays on the GPU."""
    g = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        out = []
        for m in _members(case):
            uv = _coverage(m, g)
            out.append((uv, *_observe(uv, m["n"], g)))
        return out
    n = case["n"]
    if kind == "sara":
        d = {"x": _randc(n * n, g).reshape(n, n)}
        d["w"] = torch.rand(9, n, n, generator=g, device="cuda")
        return d
    d = {"uv": _coverage(case, g)}
    if kind == "phi":
        d["x"] = _randc(n * n, g).reshape(n, n)
        d["v"] = _randc(case["M"], g)
    elif kind == "cg":
        d["b"] = _randc(n * n, g).reshape(n, n)
        d["x0"] = _randc(n * n, g).reshape(n, n)
    else:
        d["y"], d["eps"] = _observe(d["uv"], n, g)
        if kind == "diff":
            d["wv"] = 1.0 + 0.1 * (2.0 * torch.rand(case["M"], generator=g, device="cuda") - 1.0)
            d["omega"] = 0.5 + torch.rand(9, n, n, generator=g, device="cuda")
            d["gx"] = _randc(n * n, g).reshape(n, n)
    return d


def _blocks(case, eps):
    """Consecutive uneven blocks of the visibilities, each with its share of the bound."""
    R, M = case["blocks"], case["M"]
    off = [M * b * (b + 1) // (R * (R + 1)) for b in range(R + 1)]
    sigma = eps / math.sqrt((2.0 * M + 4.0 * math.sqrt(M)) / 2.0)
    e = [sigma * math.sqrt((2.0 * m + 4.0 * math.sqrt(m)) / 2.0) for m in (off[i + 1] - off[i] for i in range(R))]
    return off, e


GAMMA_SARA = 0.1  # threshold of the stand-alone prior step


# ---------------------------------------------------------------------------
# What is timed
# ---------------------------------------------------------------------------
def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        parts = []
        for m, (uv, y, eps) in zip(_members(case), d):
            ctx = binding.Context(m["n"], uv, J=m["J"], kernel=m["kernel"])
            st = ctx.sdmm_state()
            st.init(y, eps)
            parts.append((st, y, eps))
        return {"case": case, "parts": parts, "batch": binding.Batch([p[0] for p in parts])}
    if kind == "sara":
        uv = torch.zeros(16, 2, device="cuda")
        d["ctx"] = binding.Context(case["n"], uv, J=4)
    else:
        d["ctx"] = binding.Context(case["n"], d["uv"], J=case["J"], kernel=case["kernel"])
    d["case"] = case
    if case.get("beam"):
        d["ctx"].set_beam(_beam(case["n"]))
    if kind == "sdmm":
        st = d["st"] = d["ctx"].sdmm_state()
        st.set_prior(case["prior"])
        if case["blocks"]:
            st.set_blocks(*_blocks(case, d["eps"]))
    if kind == "diff":
        d["wv"].requires_grad_(True)
        d["omega"].requires_grad_(True)
        d["gamma"] = autodiff.penalty(d["ctx"], d["y"], d["wv"])
    return d


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        for st, y, eps in state["parts"]:
            st.init(y, eps)
        state["batch"].step(case["iters"])
        return [st.get_image() for st, _, _ in state["parts"]]
    ctx = state["ctx"]
    if kind == "phi":
        return ctx.phi(state["x"]), ctx.phi_adj(state["v"])
    if kind == "sara":
        alpha = ctx.sara_analysis(state["x"])
        thr = ctx.prox_l1_reweighted(alpha, state["w"], GAMMA_SARA)
        return alpha, thr, ctx.sara_synthesis(thr)
    if kind == "cg":
        return ctx.cg_solve(state["b"], state["x0"], case["iters"])[0]
    if kind == "solve":
        return ctx.sdmm_solve(state["y"], state["eps"], max_iters=case["iters"])[0]
    if kind == "sdmm":
        st = state["st"]
        st.init(state["y"], state["eps"])
        if case["data"] == "bf16":
            st.set_data_bf16(state["y"])
        for r in range(case["rounds"]):
            if r > 0:
                st.reweight(r)
            for _ in range(case["iters"]):
                st.step()
        return st.get_image()
    wv, omega = state["wv"], state["omega"]
    x = autodiff.sdmm_unrolled(ctx, state["y"], state["eps"], wv, omega, K=case["iters"],
                               checkpoint=case["checkpoint"], gamma=state["gamma"])
    gw, go = torch.autograd.grad(x, (wv, omega), state["gx"])
    return x.detach(), gw, go


# ---------------------------------------------------------------------------
# Bytes and operations of one pass
# ---------------------------------------------------------------------------
def _phi_flops(n, M, J):
    """One Phi (or Phi^H): a 2-D FFT of a 2n grid and J^2 real-by-complex terms per visibility."""
    L = 2 * n
    return 5.0 * L * L * math.log2(L * L) + 4.0 * M * J * J


def _psi_flops(n):
    """One Psi^H (or Psi): eight filter pairs along both axes, the levels a geometric series."""
    return sum(4.0 * n * n * 2 * 2 * p for p in range(1, 9)) * 4.0 / 3.0


def _sdmm_work(n, M, J, iters, k=10, prior="sara"):
    """Per iteration: k CG steps over x, r, p, s, w; the prior's dual and weights; the data branch's y, z2, u-v."""
    N = n * n
    D = 9 * N if prior == "sara" else N
    by = iters * (k * 10 * 8.0 * N + 20.0 * D + 32.0 * M)
    fl = iters * ((2 * k + 2) * _phi_flops(n, M, J) + (2 * _psi_flops(n) if prior == "sara" else 20 * 40.0 * N))
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_sdmm_work(m["n"], m["M"], m["J"], case["iters"]) for m in _members(case)]
        return {"bytes": sum(a for a, _ in w), "flops": sum(b for _, b in w)}
    n = case["n"]
    N = n * n
    if kind == "sara":
        return {"bytes": 8.0 * N + 9 * N * (8.0 + 4.0 + 8.0) + 8.0 * N, "flops": 2 * _psi_flops(n) + 9 * N * 10.0}
    M, J = case["M"], case["J"]
    if kind == "phi":
        return {"bytes": 16.0 * N + 24.0 * M, "flops": 2 * _phi_flops(n, M, J)}
    if kind == "cg":
        return {"bytes": 24.0 * N + 8.0 * M + case["iters"] * 80.0 * N, "flops": (2 * case["iters"] + 2) * _phi_flops(n, M, J)}
    if kind in ("solve", "sdmm"):
        by, fl = _sdmm_work(n, M, J, case["iters"] * case.get("rounds", 1), prior=case.get("prior", "sara"))
        return {"bytes": by, "flops": fl}
    # the forward once, once more from the checkpoints, and the reverse (about as much again)
    by, fl = _sdmm_work(n, M, J, 3 * case["iters"])
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# The same in 64 bits, from the definitions
# ---------------------------------------------------------------------------
class _Phi64:
    """Phi = G F D Z B with J x J taps of the Kaiser-Bessel (or Gaussian) kernel on the 2n grid."""

    def __init__(self, n, uv, J, kernel, beam=None):
        L = self.L = 2 * n
        self.n, self.J = n, J
        kappa = uv.double() * (L / (2 * math.pi))
        k0 = torch.floor(kappa) - J // 2 + 1
        f = (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) / L
        if kernel == "gauss":
            b = math.pi * 1.5 / (2.0 * (J / 2.0))
            def g(t):
                return torch.where(t.abs() <= J / 2, torch.exp(-b * t * t), torch.zeros_like(t))
            gh = math.sqrt(math.pi / b) * torch.exp(-(math.pi * f) ** 2 / b)
        else:
            beta = math.pi * math.sqrt((J / 2.0) ** 2 * 2.25 - 0.8)
            i0b = torch.special.i0(torch.tensor(beta, dtype=torch.float64, device="cuda"))
            def g(t):
                s = 1.0 - (2.0 * t / J) ** 2
                return torch.where(s >= 0, torch.special.i0(beta * s.clamp(min=0).sqrt()) / i0b, torch.zeros_like(t))
            a = torch.sqrt(beta ** 2 - (math.pi * J * f) ** 2)
            gh = J * torch.sinh(a) / (i0b * a)
        self.w = [g(kappa - (k0 + a)) for a in range(J)]
        self.k = [((k0 + a) % L).long() for a in range(J)]
        self.dz = 1.0 / (gh[:, None] * gh[None, :])
        if beam is not None:
            self.dz = self.dz * beam.double()
        self.rows = (torch.arange(n, device="cuda") - n // 2) % L

    def _cells(self):
        for a in range(self.J):
            for b in range(self.J):
                yield self.k[a][:, 0] * self.L + self.k[b][:, 1], self.w[a][:, 0] * self.w[b][:, 1]

    def fwd(self, x):
        L = self.L
        grid = torch.zeros(L, L, dtype=torch.complex128, device="cuda")
        grid = grid.index_put((self.rows[:, None], self.rows[None, :]), x * self.dz)
        X = (torch.fft.fft2(grid) / L).reshape(-1)
        y = 0
        for cell, w in self._cells():
            y = y + w * X[cell]
        return y

    def adj(self, y):
        L = self.L
        X = torch.zeros(L * L, 2, dtype=torch.float64, device="cuda")
        for cell, w in self._cells():
            X = X.index_add(0, cell, torch.view_as_real(w * y)) if X.requires_grad or y.requires_grad \
                else X.index_add_(0, cell, torch.view_as_real(w * y))
        x = torch.fft.ifft2(torch.view_as_complex(X).reshape(L, L)) * L
        return x[self.rows[:, None], self.rows[None, :]] * self.dz


def _db(p):
    """Daubechies-p low-pass and high-pass filters by spectral factorisation."""
    z = []
    if p > 1:
        for y in np.roots([math.comb(p - 1 + k, k) for k in range(p)][::-1]):
            c = 2.0 - 4.0 * y
            r = np.sqrt(c * c - 4.0 + 0j)
            z.append(min((c + r) / 2, (c - r) / 2, key=abs))
    h = np.real(np.poly(np.concatenate([-np.ones(p), np.array(z, dtype=complex)])))
    h *= math.sqrt(2.0) / h.sum()
    return h, (-1.0) ** np.arange(2 * p) * h[::-1]


def _split(s, h, g, dim):
    L = s.shape[dim]
    i = 2 * torch.arange(L // 2, device="cuda")
    a = d = 0
    for m in range(len(h)):
        v = s.index_select(dim, (i + m) % L)
        a, d = a + h[m] * v, d + g[m] * v
    return torch.cat([a, d], dim)


def _join(c, h, g, dim):
    L = c.shape[dim]
    i = 2 * torch.arange(L // 2, device="cuda")
    a, d = c.narrow(dim, 0, L // 2), c.narrow(dim, L // 2, L // 2)
    s = torch.zeros_like(c)
    for m in range(len(h)):
        s = s.index_add(dim, (i + m) % L, h[m] * a + g[m] * d)
    return s


def _psi_adj(x, levels=4):
    out = [x]
    for p in range(1, 9):
        h, g = _db(p)
        c, L = x, x.shape[0]
        for _ in range(levels):
            blk = _split(_split(c[:L, :L], h, g, 1), h, g, 0)
            c = blk if L == x.shape[0] else torch.cat([torch.cat([blk, c[:L, L:]], 1), c[L:]], 0)
            L //= 2
        out.append(c)
    return torch.stack(out) / 3.0


def _psi(alpha, levels=4):
    n = alpha.shape[1]
    x = alpha[0]
    for p in range(1, 9):
        h, g = _db(p)
        c = alpha[p]
        for lev in reversed(range(levels)):
            L = n >> lev
            blk = _join(_join(c[:L, :L], h, g, 0), h, g, 1)
            c = blk if L == n else torch.cat([torch.cat([blk, c[:L, L:]], 1), c[L:]], 0)
        x = x + c
    return x / 3.0


def _soft(a, lam):
    mag = a.abs()
    on = mag > lam
    return torch.where(on, a * (1.0 - lam / torch.where(on, mag, torch.ones_like(mag))), torch.zeros_like(a))


def _cg(q, b, x, iters):
    r = b - q(x)
    p, rho = r, (r.conj() * r).sum().real
    for _ in range(iters):
        if float(rho) == 0.0:
            break
        v = q(p)
        alpha = rho / (p.conj() * v).sum().real
        x, r = x + alpha * p, r - alpha * v
        rho, old = (r.conj() * r).sum().real, rho
        p = r + (rho / old) * p
    return x


def _grad(x):
    z = torch.zeros_like(x)
    return torch.cat([x[1:] - x[:-1], z[:1]], 0), torch.cat([x[:, 1:] - x[:, :-1], z[:, :1]], 1)


def _tv_prox(b, lam, w, iters=20):
    def op(p, q):
        out = torch.zeros_like(b)
        out[:-1] += p[:-1]
        out[:, :-1] += q[:, :-1]
        out[1:] -= p[:-1]
        out[:, 1:] -= q[:, :-1]
        return out
    p = torch.zeros_like(b)
    q, r, s, t = p, p, p, 1.0
    for _ in range(iters):
        g1, g2 = _grad(b - lam * op(r, s))
        pn, qn = r - g1 / (8 * lam), s - g2 / (8 * lam)
        mag = (pn.abs() ** 2 + qn.abs() ** 2).sqrt()
        f = torch.where(mag > w, w / mag.clamp(min=1e-300), torch.ones_like(mag))
        pn, qn = pn * f, qn * f
        pn[-1], qn[:, -1] = 0, 0
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        c = (t - 1.0) / tn
        r, s, p, q, t = pn + c * (pn - p), qn + c * (qn - q), pn, qn, tn
    return b - lam * op(p, q)


def _sdmm64(P, y, eps, iters, k=10, prior="sara", blocks=None, omega=None, wv=None, gamma=None, rounds=1):
    """Algorithm 1 with a warm-started k-step CG; blocks: (offsets, bounds) of several balls."""
    n = P.n
    tv = prior == "tv"
    wv = torch.ones_like(y.real) if wv is None else wv
    y = wv * y
    fwd, adj = (lambda x: wv * P.fwd(x)), (lambda v: P.adj(wv * v))
    psi_adj, psi = ((lambda x: x), (lambda a: a)) if tv else (_psi_adj, _psi)

    def feature(x):
        return torch.sqrt(sum(d.abs() ** 2 for d in _grad(x))) if tv else psi_adj(x).abs()
    if gamma is None:
        gamma = 1e-3 * float(feature(adj(y)).max())
    zero = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
    w = omega if omega is not None else torch.ones(zero.shape if tv else (9, n, n), dtype=torch.float64, device="cuda")
    off, e = blocks if blocks else ([0, len(y)], [eps])
    size = torch.tensor([off[i + 1] - off[i] for i in range(len(e))], device="cuda")
    bounds = torch.tensor(e, dtype=torch.float64, device="cuda")
    x, x1, x2, x3, z3 = zero, zero, zero, zero, zero
    z1, z2 = psi_adj(zero), torch.zeros_like(y)
    for rnd in range(rounds):
        if rnd > 0:
            a = feature(x)
            delta = max(10.0 ** -rnd, 1e-6) * float(a.max())
            w = delta / (delta + a)
        for _ in range(iters):
            x = _cg(lambda v: adj(fwd(v)) + 2.0 * v, x1 + x2 + x3, x, k)
            a1 = psi_adj(x) + z1
            r1 = _tv_prox(a1, gamma, w) if tv else _soft(a1, gamma * w)
            z1, x1 = a1 - r1, psi(2 * r1 - a1)
            a2 = fwd(x) + z2
            d = a2 - y
            nd = torch.stack([t.abs().square().sum() for t in d.split(size.tolist())]).sqrt()
            f = torch.where(nd > bounds, bounds / nd, torch.ones_like(nd)).repeat_interleave(size, output_size=len(y))
            r2 = y + f * d
            z2, x2 = a2 - r2, adj(2 * r2 - a2)
            a3 = x + z3
            r3 = torch.complex(a3.real.clamp(min=0), torch.zeros_like(a3.real))
            z3, x3 = a3 - r3, 2 * r3 - a3
    return x


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    c128 = torch.complex128
    if kind == "batch":
        return [_sdmm64(_Phi64(m["n"], uv, m["J"], m["kernel"]), y.to(c128), eps, case["iters"])
                for m, (uv, y, eps) in zip(_members(case), d)]
    if kind == "sara":
        alpha = _psi_adj(d["x"].to(c128))
        thr = _soft(alpha, float(np.float32(GAMMA_SARA)) * d["w"].double())
        return alpha, thr, _psi(thr)
    P = _Phi64(case["n"], d["uv"], case["J"], case["kernel"], _beam(case["n"]) if case.get("beam") else None)
    if kind == "phi":
        return P.fwd(d["x"].to(c128)), P.adj(d["v"].to(c128))
    if kind == "cg":
        return _cg(lambda v: P.adj(P.fwd(v)) + 2.0 * v, d["b"].to(c128), d["x0"].to(c128), case["iters"])
    y = d["y"].to(c128)
    if kind == "solve":
        return _sdmm64(P, y, d["eps"], case["iters"])
    if kind == "sdmm":
        return _sdmm64(P, y, d["eps"], case["iters"], prior=case["prior"], rounds=case["rounds"],
                       blocks=_blocks(case, d["eps"]) if case["blocks"] else None)
    wv = d["wv"].double().requires_grad_(True)
    om = d["omega"].double().requires_grad_(True)
    with torch.no_grad():
        gamma = 1e-3 * float(_psi_adj(P.adj(wv * wv * y)).abs().max())
    x = _sdmm64(P, y, d["eps"], case["iters"], omega=om, wv=wv, gamma=gamma)
    gw, go = torch.autograd.grad(x, (wv, om), d["gx"].to(c128))
    return x.detach(), gw, go
