"""Performance cases of the ACAT step: what a program that uses the library has
it do, through the binding's public calls (Context.acat_step, Context.acat_run,
adjoint.run), over the sizes of the test problems and of the benchmark.

A case is a dict of plain values:
  kind   "step" (one step, with its dt and order codes), "run" (consecutive
         steps in place), "grad" (forward run and gradient of a misfit)
  data   "riemann", "burgers", "wave", "pulse" (1D), "batch" (a ragged batch of
         1D Riemann problems), "quadrants", "smooth", "wave2d" (2D)
  n, ny  cells (batch: the largest instance); inst: instances of a batch
  P, f32, steps, and the options rect, lo (F^lo) and mod (psi~^2).

exact() restates the method in plain torch float64 operations.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

from paper_2007_01416_gb300 import acat, adjoint

GAMMA = 1.4
FLUX = {"riemann": acat.EULER1D, "batch": acat.EULER1D, "pulse": acat.EULER1D, "burgers": acat.BURGERS,
        "wave": acat.LINEAR, "quadrants": acat.EULER2D, "smooth": acat.EULER2D, "wave2d": acat.LINEAR}
PERIODIC = ("burgers", "wave", "pulse", "smooth", "wave2d")
TWO_D = ("quadrants", "smooth", "wave2d")
NVARS = {acat.LINEAR: 1, acat.BURGERS: 1, acat.EULER1D: 3, acat.EULER2D: 4}


def _case(name, kind, data, n, P, steps, f32=False, ny=1, inst=0, rect=False, lo=0, mod=False):
    c = dict(kind=kind, data=data, n=n, ny=ny, P=P, steps=steps, f32=f32, inst=inst, rect=rect, lo=lo, mod=mod)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one step of a coarse shock-tube grid, as a host code that drives the
        # time loop itself calls it (dt and the selected orders come back)
        _case("step_p4_450", "step", "riemann", 450, 4, 1),
        # a whole run of the paper's Burgers test, 400 cells to past shock formation
        _case("run_burgers_p2_400", "run", "burgers", 400, 2, 300),
        # a block of steps between two outputs of a long shock-tube run: the
        # highest order in FP64, the lowest, and the highest in FP32
        _case("run_p4_16384", "run", "riemann", 16384, 4, 48),
        _case("run_p2_16384", "run", "riemann", 16384, 2, 48),
        _case("run_p4_16384_f32", "run", "riemann", 16384, 4, 48, f32=True),
        # ragged ensembles: a few hundred members in FP64, thousands in FP32
        _case("batch_p3_256", "run", "batch", 16384, 3, 2, inst=256),
        _case("batch_p3_4096_f32", "run", "batch", 16384, 3, 2, f32=True, inst=4096),
        # 2D Riemann problems: production size in FP32, ragged and small in FP64
        _case("quadrants_p2_4096_f32", "run", "quadrants", 4096, 2, 2, f32=True, ny=4096),
        _case("quadrants_p2_500x411", "run", "quadrants", 500, 2, 2, ny=411),
        # high-order 2D: smooth flow with a contact on square stencils in FP64,
        # four quadrants on rectangular stencils in FP32
        _case("smooth_p3_256", "run", "smooth", 256, 3, 2, ny=256),
        _case("quadrants_rect_p4_512_f32", "run", "quadrants", 512, 4, 2, f32=True, ny=512, rect=True),
        # gradient of a final-time misfit with respect to the initial state
        _case("grad_p2_8192", "grad", "pulse", 8192, 2, 128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "run1d", "run1d", "batch", "quadrants", "smooth", "grad"])
    f32, P = rng.random() < 0.5, rng.choice([2, 3, 4])
    lo, mod = (2, True) if rng.random() < 0.25 else (0, False)
    if kind == "step":
        return _case(None, "step", "riemann", _log(rng, 64, 40000), P, 1, f32=f32, lo=lo, mod=mod)
    if kind == "run1d":
        data = rng.choice(["riemann", "riemann", "burgers", "wave"])
        return _case(None, "run", data, _log(rng, 200, 40000), P, rng.randint(8, 60), f32=f32, lo=lo, mod=mod)
    if kind == "batch":
        return _case(None, "run", "batch", _log(rng, 300, 16384), P, rng.randint(1, 2), f32=f32,
                     inst=_log(rng, 8, 1024 if f32 else 64), lo=lo, mod=mod)
    if kind == "grad":
        return _case(None, "grad", "pulse", _log(rng, 256, 8192), rng.choice([2, 3]), rng.randint(16, 100), f32=f32)
    top = (2048 if P == 2 else 512) if f32 else (512 if P == 2 else 192)
    data = kind if P == 2 or kind == "smooth" else "wave2d"
    rect = kind == "quadrants" and P > 2
    return _case(None, "run", "quadrants" if rect else data, _log(rng, 48, top), P, rng.randint(1, 2), f32=f32,
                 ny=_log(rng, 48, top), rect=rect, lo=lo, mod=mod)


# ---- inputs -----------------------------------------------------------------
def _sizes(case, seed):
    """Instance sizes of a batch: the case fixes them, the seed their order."""
    if case["data"] != "batch":
        return None
    lo = min(256, case["n"])
    sizes = np.random.default_rng([case["n"], case["inst"]]).integers(lo, case["n"] + 1, size=case["inst"])
    return np.random.default_rng([seed, 7]).permutation(sizes).astype(np.int64)


def _centres(n, a, b):
    return a + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * ((b - a) / n)


def _euler1d(rho, u, p):
    return torch.stack([rho, rho * u, p / (GAMMA - 1.0) + 0.5 * rho * u * u])


def _euler2d(rho, u, v, p):
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)])


def _riemann(x, left, w, k):
    """Seeded Riemann data with an entropy wave in the density; w[0..5] the
    left and right (rho, u, p), k the wave number (numbers, or one per cell)."""
    side = [torch.where(left, w[q], w[q + 3]) for q in range(3)]
    return _euler1d(side[0] * (1.0 + 0.2 * torch.sin(k * x)), side[1], side[2])


def _state(case, seed):
    """The initial state in float64, [s, n] or [s, ny, n], on the GPU."""
    rng, d, n, ny = np.random.default_rng([seed, 3]), case["data"], case["n"], case["ny"]
    dev = dict(dtype=torch.float64, device="cuda")
    if d in ("riemann", "batch"):
        B = case["inst"] if d == "batch" else 1
        w = np.stack([rng.uniform(*r, size=B) for r in ((0.1, 1), (-0.5, 0.5), (0.1, 1)) * 2 + ((4.0, 8.0),)])
        w = torch.tensor(w, **dev)
        if d == "batch":
            sizes = torch.tensor(_sizes(case, seed), device="cuda")
            w = torch.repeat_interleave(w, sizes, dim=1)
            nb = torch.repeat_interleave(sizes, sizes).to(torch.float64)
            off = torch.repeat_interleave(torch.cumsum(sizes, 0) - sizes, sizes)
            x = (torch.arange(int(sizes.sum()), device="cuda") - off + 0.5) / nb
        else:
            x = _centres(n, 0.0, 1.0)
        return _riemann(x, x < 0.5, w[:6], w[6])
    if d == "burgers":
        a, b, phi = rng.uniform(0.2, 0.5), rng.uniform(0.5, 1.0), rng.uniform(0.0, 2.0 * math.pi)
        return (a + b * torch.sin(math.pi * _centres(n, -1.0, 1.0) + phi))[None].contiguous()
    if d == "wave":  # a smooth wave and a step
        k, xc = rng.integers(1, 4), rng.uniform(0.3, 0.7)
        x = _centres(n, 0.0, 1.0)
        return (torch.sin(2 * math.pi * int(k) * x) + 0.5 * (x > xc))[None].contiguous()
    if d == "pulse":
        xc, w = rng.uniform(0.3, 0.7), rng.uniform(0.02, 0.08)
        rho = 1.0 + 0.01 * torch.exp(-((_centres(n, 0.0, 1.0) - xc) ** 2) / (w * w))
        return _euler1d(rho, torch.zeros_like(rho), rho ** GAMMA / GAMMA)
    x, y = _centres(n, 0.0, 1.0)[None, :], _centres(ny, 0.0, 1.0)[:, None]
    if d == "quadrants":
        q = torch.where(x > 0.5, torch.where(y > 0.5, 0, 3), torch.where(y > 0.5, 1, 2))
        st = [[rng.uniform(*r) for _ in range(4)] for r in ((0.1, 1.5), (-0.8, 0.8), (-0.8, 0.8), (0.1, 1.5))]
        return _euler2d(*(torch.tensor(s, **dev)[q] for s in st)).contiguous()
    a, xc, phi = rng.uniform(0.1, 0.3), rng.uniform(0.4, 0.7), rng.uniform(0.0, 2.0 * math.pi)
    tp = 2 * math.pi
    if d == "wave2d":
        return (1.0 + a * torch.sin(tp * x) * torch.sin(tp * y) + 0.3 * (x + 0 * y > xc))[None].contiguous()
    rho = 1.0 + a * torch.sin(tp * x) * torch.sin(tp * y) + 0.3 * (x + 0 * y > xc)
    return _euler2d(rho, 0.3 + 0.1 * torch.cos(tp * y) + 0 * x, -0.2 + 0.1 * torch.sin(tp * x) + 0 * y,
                    1.0 + 0.1 * torch.cos(tp * (x + y) + phi)).contiguous()


def _params(case):
    d = case["data"]
    x0 = -1.0 if d == "burgers" else 0.0
    return dict(flux=FLUX[d], P=case["P"], nx=case["n"], ny=case["ny"], cfl=0.5 if d == "burgers" else 0.4, x0=x0,
                x1=1.0, y0=0.0, y1=1.0, gamma=GAMMA, adv=(1.0, 0.7), lo_flux=case["lo"], psi2_mod=int(case["mod"]),
                rect_2d=int(case["rect"]), bc=acat.PERIODIC if d in PERIODIC else acat.TRANSMISSIVE,
                precision=acat.PREC_F32 if case["f32"] else acat.PREC_F64)


def prepare(case, seed):
    u0 = _state(case, seed)
    sizes = _sizes(case, seed)
    ctx = acat.Context(sizes=None if sizes is None else sizes.tolist(), **_params(case))
    layout = acat.to_pair if case["f32"] else (lambda v: v)
    s = {"case": case, "ctx": ctx, "u0": layout(u0)}
    if case["kind"] == "grad":
        s["target"] = _state(case, seed + 1000003)
        s["u0"].requires_grad_(True)
    else:
        s["u"] = torch.empty_like(s["u0"])
    if case["kind"] == "step":
        s["dt"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["orders"] = torch.zeros(case["n"] + 1, dtype=torch.int8, device="cuda")
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["kind"] == "step":
        ctx.acat_step(s["u0"], s["u"], dt_out=s["dt"], orders_out=s["orders"])
        return {"u": s["u"], "dt": s["dt"], "orders": s["orders"]}
    if case["kind"] == "grad":
        uN = adjoint.run(s["u0"], ctx, case["steps"])
        value = acat.from_pair(uN) if case["f32"] else uN
        loss = 0.5 * ((value - s["target"]) ** 2).sum() / case["n"]
        (g,) = torch.autograd.grad(loss, s["u0"])
        return {"u": uN.detach(), "loss": loss.detach(), "grad": g}
    s["u"].copy_(s["u0"])
    ctx.acat_run(s["u"], case["steps"])
    return {"u": s["u"]}


# ---- work -------------------------------------------------------------------
def _cells(case):
    if case["data"] == "batch":
        return case["inst"] * (min(256, case["n"]) + case["n"]) // 2
    return case["n"] * case["ny"]


def work(case):
    """The state in and out once; the flops of the method with running Taylor
    sums, every interface at order 2P, no boundary or indicator work."""
    flux, n = FLUX[case["data"]], 2 * case["P"]
    S, cells = NVARS[flux], _cells(case)
    phi = {acat.LINEAR: 1, acat.BURGERS: 2, acat.EULER1D: 10, acat.EULER2D: 19}[flux]
    if case["data"] in TWO_D:
        node = phi + (n - 1) * (4 * n * S + (n - 1) * (6 * S + phi) + 8 * S)
        flops = cells * n * n * node
    else:
        flops = cells * (n * phi + (n - 1) * (2 * n * n * S + n * (n - 1) * (4 * S + phi) + 4 * n * S))
    passes = 3.0 if case["kind"] == "grad" else 1.0  # forward, and the reverse sweep
    return {"bytes": 2.0 * cells * S * 8, "flops": passes * case["steps"] * flops}


# ---- the method in plain float64 ---------------------------------------------
def _fd(nodes, k, at):
    """Weights of the k-th derivative at `at` on the integer nodes (exact)."""
    n, h = len(nodes), [Fraction(x) - at for x in nodes]
    A = [[h[j] ** i for j in range(n)] + [Fraction(math.factorial(k) if i == k else 0)] for i in range(n)]
    for i in range(n):
        piv = next(r for r in range(i, n) if A[r][i] != 0)
        A[i], A[piv] = A[piv], A[i]
        A[i] = [v / A[i][i] for v in A[i]]
        for r in range(n):
            if r != i and A[r][i] != 0:
                A[r] = [a - A[r][i] * b for a, b in zip(A[r], A[i])]
    return [float(A[i][n]) for i in range(n)]


_WEIGHTS: dict = {}


def _weights(p):
    if p not in _WEIGHTS:
        nodes = list(range(-p + 1, p + 1))
        d1, gh, s = _fd(list(range(-p, p + 1)), 1, Fraction(0)), [], 0.0
        for m in range(2 * p):
            s -= d1[m]
            gh.append(s)
        _WEIGHTS[p] = ([_fd(nodes, 1, Fraction(j)) for j in nodes], [_fd(nodes, k, Fraction(0)) for k in range(2 * p)],
                       gh, _fd(nodes, 2 * p - 1, Fraction(1, 2)))
    return _WEIGHTS[p]


class _Exact:
    def __init__(self, case, seed):
        self.case, self.kw = case, _params(case)
        self.flux, self.P = FLUX[case["data"]], case["P"]
        self.S, self.G = NVARS[self.flux], max(case["P"], 2)
        self.sizes = _sizes(case, seed)
        self.two_d = case["data"] in TWO_D
        self.speed_max = {}

    # physics in direction `dr`
    def prim(self, u):
        v = [m / u[0] for m in u[1:-1]]
        return v, (GAMMA - 1.0) * (u[-1] - 0.5 * u[0] * sum(w * w for w in v))

    def f(self, u, dr=0):
        if self.flux == acat.LINEAR:
            return [self.kw["adv"][dr] * u[0]]
        if self.flux == acat.BURGERS:
            return [0.5 * u[0] * u[0]]
        v, p = self.prim(u)
        out = [u[1 + dr]] + [m * v[dr] for m in u[1:-1]] + [v[dr] * (u[-1] + p)]
        out[1 + dr] = out[1 + dr] + p
        return out

    def eig(self, u, dr=0):
        if self.flux == acat.LINEAR:
            a = torch.full_like(u[0], self.kw["adv"][dr])
            return a, a
        if self.flux == acat.BURGERS:
            return u[0], u[0]
        v, p = self.prim(u)
        c = torch.sqrt(GAMMA * p / u[0])
        return v[dr] - c, v[dr] + c

    def radius(self, u, dr=0):
        if self.flux in (acat.LINEAR, acat.BURGERS):
            a = self.eig(u, dr)[0]
            return torch.where(a < 0, -a, a)
        v, p = self.prim(u)
        return torch.where(v[dr] < 0, -v[dr], v[dr]) + torch.sqrt(GAMMA * p / u[0])

    # order of the interfaces of line[c] ([K, 2G], cell i in column G - 1)
    def orders(self, line):
        ic, eps = self.G - 1, 1e-12
        ps = torch.ones(line[0].shape[0], dtype=torch.int64, device=line[0].device)
        for p in range(2, self.P + 1):
            best = None
            for q in line:
                d = [q[:, ic + 1 + j] - q[:, ic + j] for j in range(-p + 1, p)]  # j = -p+1 .. p-1
                D = math.factorial(2 * p - 1) * sum(w * q[:, ic + j - p + 1] for j, w in enumerate(_weights(p)[3]))
                tau = D * D
                IL, IR = sum(x * x for x in d[:p - 1]) + eps, sum(x * x for x in d[p:]) + eps
                if p == 2 and self.case["mod"]:
                    splits = ((IL, IR + d[1] * d[1]), (IL + d[1] * d[1], IR))
                else:
                    splits = ((IL, IR),)
                psi = None
                for a, b in splits:
                    I = a * b / (a + b)
                    v = I / (I + tau)
                    psi = v if psi is None else torch.maximum(psi, v)
                best = psi if best is None else torch.minimum(best, psi)
            ps = torch.where(best >= 0.9, torch.full_like(ps, p), ps)
        return ps

    # CAT flux of blocks ub[c] ([K, n2, n1]); p2 = 0: a 1D stencil (n2 = 1)
    def cat(self, ub, p1, p2, lx, ly, dr):
        pm = max(p1, p2)
        n1, n = 2 * p1, 2 * pm
        z1, z2 = p1 - 1, max(p2 - 1, 0)
        ps = p2 if dr else p1
        col = lambda g: torch.tensor(g, dtype=torch.float64, device=ub[0].device)  # noqa: E731
        gx, gk, gh = col(_weights(p1)[0]), _weights(pm)[1], col(_weights(ps)[2])
        gy = col(_weights(p2)[0]) if p2 else None
        total = lambda h: ((h[:, :, z1] if dr else h[:, z2, :]) * gh).sum(-1)  # noqa: E731
        f, g = self.f(ub, 0), (self.f(ub, 1) if p2 else None)
        out = [total(h) for h in (g if dr else f)]
        args = [list(ub) for _ in range(n)]
        kf = 1.0
        f0, g0 = f, g
        for k in range(2, n + 1):
            kf *= k
            U = [-lx * sum(h[:, :, r:r + 1] * gx[:, r] for r in range(n1)) for h in f]
            if p2:
                U = [a - ly * sum(h[:, r:r + 1, :] * gy[:, r][:, None] for r in range(2 * p2)) for a, h in zip(U, g)]
            f = [gk[k - 1][pm - 1] * h for h in f0]
            g = [gk[k - 1][pm - 1] * h for h in g0] if p2 else None
            for r in range(n):
                j = r - pm + 1
                if j == 0:
                    continue
                w = float(j) ** (k - 1) / math.factorial(k - 1)
                args[r] = [a + w * x for a, x in zip(args[r], U)]
                f = [a + gk[k - 1][r] * b for a, b in zip(f, self.f(args[r], 0))]
                if p2:
                    g = [a + gk[k - 1][r] * b for a, b in zip(g, self.f(args[r], 1))]
            if k <= 2 * ps:
                out = [a + total(h) / kf for a, h in zip(out, g if dr else f)]
        return out

    def limiter(self, line, dr):
        ic = self.G - 1
        one = torch.ones_like(line[0][:, 0])

        def superbee(upw, loc):
            zero = loc == 0
            inf = torch.where(upw > 0, one * math.inf, -one * math.inf)
            r = torch.where(zero, torch.where(upw == 0, one, inf), upw / torch.where(zero, one, loc))
            a, b = torch.where(2 * r < 1, 2 * r, one), torch.where(r < 2, r, 2 * one)
            m = torch.where(a > b, a, b)
            return torch.where(m > 0, m, 0 * one)

        if self.S == 1:
            um, u0, u1, u2 = (line[0][:, ic + d] for d in (-1, 0, 1, 2))
            if self.flux == acat.LINEAR:
                a = self.kw["adv"][dr] * one
            else:
                same = u0 == u1
                a = torch.where(same, u0, (0.5 * u1 * u1 - 0.5 * u0 * u0) / torch.where(same, one, u1 - u0))
            return superbee(torch.where(a > 0, u0 - um, u2 - u1), u1 - u0)
        best = 2 * one
        for q in line:
            loc = q[:, ic + 1] - q[:, ic]
            for upw in (q[:, ic] - q[:, ic - 1], q[:, ic + 2] - q[:, ic + 1]):
                v = superbee(upw, loc)
                best = torch.where(v < best, v, best)
        return best

    def lo(self, ul, ur, dr):
        fl, fr = self.f(ul, dr), self.f(ur, dr)
        if self.case["lo"] == acat.LO_HLL:
            (al, bl), (ar, br) = self.eig(ul, dr), self.eig(ur, dr)
            sl, sr = torch.where(ar < al, ar, al), torch.where(br > bl, br, bl)
            den = torch.where(sr == sl, torch.ones_like(sl), sr - sl)
            mid = [(sr * a - sl * b + sl * sr * (y - x)) / den for a, b, x, y in zip(fl, fr, ul, ur)]
            return [torch.where(sl >= 0, a, torch.where(sr <= 0, b, m)) for a, b, m in zip(fl, fr, mid)]
        a, b = self.radius(ul, dr), self.radius(ur, dr)
        alpha = torch.where(b > a, b, a)
        return [0.5 * (a + b) - 0.5 * alpha * (y - x) for a, b, x, y in zip(fl, fr, ul, ur)]

    # fluxes at interfaces: `gather(sel, p1, p2)` gives the block of nodes
    def fluxes(self, line, other, gather, lx, ly, dr):
        with torch.no_grad():
            ps = self.orders(line)
            cross = ps if self.two_d else torch.zeros_like(ps)
            if self.two_d and self.case["rect"]:
                cross = torch.where(ps > 1, self.orders(other), ps)
        out = [torch.zeros(ps.shape[0], dtype=torch.float64, device=ps.device) for _ in range(self.S)]
        at = lambda v, sel: v[sel][:, None, None] if torch.is_tensor(v) else v  # noqa: E731
        for key in torch.unique(ps * 8 + cross).tolist():
            p, q = key // 8, key % 8
            sel = torch.nonzero(ps * 8 + cross == key)[:, 0]
            p1, p2 = (q, p) if dr else (p, q)
            F = self.cat(gather(sel, p1, p2), p1, p2, at(lx, sel), at(ly, sel), dr)
            if p == 1:
                ls = [v[sel] for v in line]
                w = self.limiter(ls, dr)
                lo = self.lo([v[:, self.G - 1] for v in ls], [v[:, self.G] for v in ls], dr)
                F = [w * a + (1.0 - w) * b for a, b in zip(F, lo)]
            out = [o.index_copy(0, sel, v) for o, v in zip(out, F)]
        return out, ps

    def wrap(self, i, n):
        return torch.remainder(i, n) if self.kw["bc"] == acat.PERIODIC else torch.minimum(i.clamp(min=0), n - 1)

    def step1d(self, u, dt=None):
        """One 1D step of u [S, M]; the instances of a batch side by side."""
        dev, G, length = u.device, self.G, self.kw["x1"] - self.kw["x0"]
        sizes = torch.tensor(self.sizes if self.sizes is not None else [u.shape[1]], device=dev)
        B = sizes.shape[0]
        inst = torch.repeat_interleave(torch.arange(B, device=dev), sizes)
        dx = length / sizes.to(torch.float64)
        if dt is None:
            sp = torch.zeros(B, dtype=torch.float64, device=dev)
            sp = sp.scatter_reduce(0, inst, self.radius(list(u.detach())), "amax")
            dt = self.kw["cfl"] * dx / sp
        off = torch.cumsum(sizes, 0) - sizes
        iface = torch.repeat_interleave(torch.arange(B, device=dev), sizes + 1)  # interface -> instance
        first = off + torch.arange(B, device=dev)
        m = torch.arange(iface.shape[0], device=dev) - first[iface]
        lam, F, codes = dt / dx, [], []
        for part in torch.split(torch.arange(iface.shape[0], device=dev), 1 << 20):
            b = iface[part]
            cell = m[part][:, None] + torch.arange(2 * G, device=dev) - G
            line = [v[off[b][:, None] + self.wrap(cell, sizes[b][:, None])] for v in u]
            gather = lambda sel, p1, p2: [v[sel][:, None, G - p1:G + p1] for v in line]  # noqa: E731
            f, ps = self.fluxes(line, None, gather, lam[b], 0.0, 0)
            F.append(torch.stack(f))
            codes.append(ps)
        F = torch.cat(F, 1)
        left = torch.arange(u.shape[1], device=dev) + inst
        return u + lam[inst] * (F[:, left] - F[:, left + 1]), dt, torch.cat(codes)

    def step2d(self, u):
        S, ny, nx = u.shape
        G, dev = self.G, u.device
        dx, dy = 1.0 / nx, 1.0 / ny
        sx, sy = (float(self.radius(list(u), d).max()) for d in (0, 1))
        dt = 0.5 * self.kw["cfl"] * min(dx / sx, dy / sy)
        nxt, nyt = torch.tensor(nx, device=dev), torch.tensor(ny, device=dev)
        flat = u.reshape(S, -1)
        span = lambda p: torch.arange(-p + 1, p + 1, device=dev)  # noqa: E731
        res = []
        for dr in (0, 1):
            w, h = (nx + 1, ny) if dr == 0 else (nx, ny + 1)
            F = []
            for part in torch.split(torch.arange(w * h, device=dev), (1 << 24) // (4 * self.P * self.P)):
                x, y = part % w - (1 - dr), part // w - dr
                pick = lambda xx, yy: self.wrap(yy, nyt) * nx + self.wrap(xx, nxt)  # noqa: E731
                ix = pick(x[:, None] + span(G), y[:, None])
                iy = pick(x[:, None], y[:, None] + span(G))
                lines = [[v[i] for v in flat] for i in (ix, iy)]

                def gather(sel, p1, p2):
                    i = pick(x[sel][:, None, None] + span(p1), y[sel][:, None, None] + span(p2)[:, None])
                    return [v[i] for v in flat]

                F.append(torch.stack(self.fluxes(lines[dr], lines[1 - dr], gather, dt / dx, dt / dy, dr)[0]))
            res.append(torch.cat(F, 1).reshape(S, h, w))
        F, Gy = res
        return u + dt / dx * (F[:, :, :-1] - F[:, :, 1:]) + dt / dy * (Gy[:, :-1] - Gy[:, 1:])


def _pair(u):
    hi = u.to(torch.float32).to(torch.float64)
    return torch.stack([hi, u - hi])


def exact(case, seed):
    u = _state(case, seed)
    if case["f32"]:
        u = _held(u)
    E, layout = _Exact(case, seed), (_pair if case["f32"] else (lambda v: v))
    if case["kind"] == "step":
        un, dt, codes = E.step1d(u)
        return {"u": layout(un), "dt": dt, "orders": codes.to(torch.int8)}
    if case["kind"] == "run":
        for _ in range(case["steps"]):
            u = E.step2d(u) if E.two_d else E.step1d(u)[0]
        return {"u": layout(u)}
    seen = []
    for _ in range(case["steps"]):
        un, dt, _ = E.step1d(u)
        seen.append((u, dt))
        u = un
    diff = u - _state(case, seed + 1000003)
    g = diff / case["n"]
    for v, dt in reversed(seen):
        v = v.detach().requires_grad_(True)
        (g,) = torch.autograd.grad(E.step1d(v, dt)[0], v, grad_outputs=g)
    return {"u": layout(u), "loss": 0.5 * (diff ** 2).sum() / case["n"],
            "grad": torch.stack([g, g]) if case["f32"] else g}


def _held(u):
    """The value hi + lo that the compensated FP32 layout holds of u."""
    hi = u.to(torch.float32)
    return hi.to(torch.float64) + (u - hi.to(torch.float64)).to(torch.float32).to(torch.float64)
