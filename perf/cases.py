"""Performance cases: the calls that a user of this library makes, over the sizes they make them at.

Kinds of a case (``kind``):

* ``sweeps``   -- a new problem in an existing handle: ``reset`` (initial plan),
  domain-decomposition sweeps, score, both marginals and the dual read back.
* ``batch``    -- sweeps of many independent problems in one batch, continuing.
* ``sinkhorn`` -- the global unbalanced Sinkhorn (the warm start and comparator).
* ``gap``      -- the primal-dual certificate of a handle.
* ``grad``     -- the adjoint: gradients in mu, nu and the source positions.
* ``score``    -- the differentiable score, forward and backward.

``eps_px`` is eps in squared pixels, eps = eps_px / N^2.  ``err < 0`` is the
library's fixed-budget mode (exactly ``maxit`` iterations).  Results of the
modes that compute in single precision (FP32 cells, MIXED Sinkhorn, FP32
adjoint) are kept in float32, as a program that chose those modes keeps them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_08859_gb300 import domdec as dd
from paper_2410_08859_gb300 import inputs

F64 = torch.float64
PRECISION = {"fp32": dd.FP32, "fp64": dd.FP64, "mixed": dd.MIXED}


# ------------------------------------------------------------------ the cases
def _sweeps(N, s, **kw):
    c = dict(kind="sweeps", N=N, s=s, field="blobs", eps_px=1.0, lam=1.0, precision="fp32", strategy="staggered",
             ti=0, err=-1.0, maxit=20, sweeps=2, start="duals")
    c.update(kw)
    return c


def listed():
    return [
        # small double-precision solve from the product plan: the paper's tolerance, at most 100 iterations
        _sweeps(32, 4, name="mix32_fp64", field="mix", precision="fp64", err=2e-5, maxit=100, start="product"),
        # the 256 x 256 workload of blob images: warm start, then sweeps in FP32 at eps = h^2
        _sweeps(256, 8, name="blobs256", sweeps=4),
        # the translation step with the line search on each staggered sub-batch
        _sweeps(256, 8, name="line256", strategy="staggered_line", ti=1),
        # odd sizes, weak marginal penalty, one step size for the whole partition
        _sweeps(210, 7, name="swift210", field="lognormal", eps_px=2.0, lam=0.1, strategy="swift", sweeps=3),
        # the largest workload: log-normal fields at 1024 x 1024
        _sweeps(1024, 16, name="lognormal1024", field="lognormal", eps_px=4.0, maxit=8, sweeps=8),
        # many small and middling problems at once
        dict(name="batch16", kind="batch", count=16, side_lo=64, side_hi=256, s=8, eps_px=4.0, maxit=10, sweeps=2),
        # the warm start of the solver: eps-scaling from 1, float while eps is coarse
        dict(name="warm256_mixed", kind="sinkhorn", N=256, eps_px=2.0, lam=1.0, precision="mixed", err=-1.0,
             maxit=20, noalloc=False),
        # a small global solve in double precision to the paper's tolerance
        dict(name="sinkhorn64_fp64", kind="sinkhorn", N=64, eps_px=4.0, lam=1.0, precision="fp64", err=2e-5,
             maxit=1000, noalloc=False),
        # the certificate that ends a solve, at the largest size
        dict(name="gap1024", kind="gap", N=1024, s=16, eps_px=4.0, lam=1.0),
        # the backward pass at 512 x 512, and a small odd one with single-precision sums
        dict(name="grad512_fp64", kind="grad", N=512, eps_px=4.0, lam=1.0, precision="fp64"),
        dict(name="grad150_fp32", kind="grad", N=150, eps_px=4.0, lam=1.0, precision="fp32"),
        # one evaluation of the differentiable score and its gradients, handle and warm start included
        dict(name="score64", kind="score", N=64, s=8, eps_px=4.0, lam=1.0, maxit=20, sweeps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweeps", "sweeps", "sweeps", "batch", "sinkhorn", "gap", "grad", "score"])
    lam = round(math.exp(rng.uniform(math.log(0.1), math.log(10.0))), 3)
    eps_px = round(rng.uniform(1.0, 4.0), 2)
    if kind == "sweeps":
        if rng.random() < 0.25:
            s = rng.randint(2, 4)
            N = 2 * s * max(2, _log_int(rng, 16, 40) // (2 * s))
            return _sweeps(N, s, field="mix", eps_px=eps_px, lam=lam, precision="fp64", err=2e-5, maxit=100,
                           start="product", sweeps=rng.randint(1, 2))
        s = rng.randint(4, 16)
        N = 2 * s * max(4, _log_int(rng, 96, 640) // (2 * s))
        strategy, ti = rng.choice([("staggered", 0), ("staggered", 0), ("staggered", 1), ("swift", 0),
                                   ("staggered_line", 1)])
        return _sweeps(N, s, field=rng.choice(["blobs", "lognormal"]), eps_px=eps_px, lam=lam, strategy=strategy,
                       ti=ti, maxit=rng.randint(5, 20), sweeps=rng.randint(1, 4))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 20), side_lo=rng.choice([32, 64]),
                    side_hi=rng.choice([128, 192, 256]), s=rng.choice([4, 8]), eps_px=eps_px,
                    maxit=rng.randint(5, 15), sweeps=rng.randint(1, 3))
    if kind == "sinkhorn":
        precision, N = rng.choice(["mixed", "fp64", "fp32"]), _log_int(rng, 32, 300)
        return dict(kind="sinkhorn", N=N, eps_px=round(2 * eps_px, 2), lam=lam, precision=precision, err=-1.0,
                    maxit=rng.randint(5, 15), noalloc=precision != "mixed" and N <= 256 and rng.random() < 0.3)
    if kind == "gap":
        s = rng.randint(4, 16)
        return dict(kind="gap", N=2 * s * max(4, _log_int(rng, 96, 900) // (2 * s)), s=s, eps_px=eps_px, lam=lam)
    if kind == "grad":
        return dict(kind="grad", N=_log_int(rng, 40, 640), eps_px=eps_px, lam=lam,
                    precision=rng.choice(["fp64", "fp32"]))
    s = rng.randint(4, 8)
    return dict(kind="score", N=2 * s * rng.randint(4, 8), s=s, eps_px=round(2 * eps_px, 2), lam=lam,
                maxit=rng.randint(10, 20), sweeps=2 * rng.randint(1, 3))


# ------------------------------------------------------------------- the work
def work(case):
    """Bytes of the inputs and outputs; operations of the separable
    log-sum-exp terms within e^-36 of their target (four operations each:
    exponent, shift, exponential, sum)."""
    px = case["eps_px"]
    win = 2.0 * math.sqrt(36.0 * px) + 1.0

    def glob(N, p):   # one separable log-sum-exp over the grid
        return 2.0 * N * N * min(N, 2.0 * math.sqrt(36.0 * p) + 1.0) * 4.0

    def cells(N, s, maxit, sweeps):   # cell iterations of `sweeps` partition sweeps
        x, y = 2 * s, min(N, 2 * s + win)
        terms = x * y * min(x, win) + y * y * min(x, win) + y * x * min(y, win) + x * x * min(y, win)
        return sweeps * (N / (2 * s)) ** 2 * maxit * terms * 4.0

    def stages(N, px_end, maxit):
        return sum(2 * maxit * glob(N, px_end * 2.0 ** k) for k in range(int(math.log2(N * N / px_end)) + 1))

    kind = case["kind"]
    if kind == "batch":
        sides = _sides(case)
        return {"bytes": sum(8.0 * 6 * N * N for N in sides),
                "flops": sum(cells(N, case["s"], case["maxit"], case["sweeps"]) for N in sides)}
    N = case["N"]
    n = float(N) * N
    if kind == "sweeps":
        it = case["maxit"] if case["err"] < 0 else 50
        return {"bytes": 8.0 * 7 * n, "flops": cells(N, case["s"], it, case["sweeps"])}
    if kind == "sinkhorn":
        return {"bytes": 8.0 * 4 * n, "flops": stages(N, px, case["maxit"] if case["err"] < 0 else 20)}
    if kind == "gap":
        return {"bytes": 8.0 * 6 * n, "flops": glob(N, px)}
    if kind == "grad":
        return {"bytes": 8.0 * 8 * n, "flops": 2 * glob(N, px)}
    return {"bytes": 8.0 * 4 * n,
            "flops": stages(N, 2 * px, case["maxit"]) + cells(N, case["s"], case["maxit"], case["sweeps"])}


# ----------------------------------------------------------------- the inputs
def _sides(case):
    """Grid sides of a batch: spread evenly over the logarithm of the range, whole cells."""
    k, lo, hi, c = case["count"], case["side_lo"], case["side_hi"], 2 * case["s"]
    return [max(4, round(lo * (hi / lo) ** (i / max(1, k - 1)) / c)) * c for i in range(k)]


def _image_pair(field, N, seed):
    seed = 1000 + 17 * seed
    if field == "mix":
        mu, nu = inputs.mixture_small(N=N, seed=seed)
    elif field == "blobs":
        mu, nu = inputs.mixture_blobs(N=N, seed=seed)
    else:
        mu, nu = inputs.lognormal_field(N=N, seed=seed)
    return tuple(torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda() for a in (mu, nu))


def _duals(mu, nu, N, eps, lam, precision="mixed", maxit=10):
    """Warm-start potentials at eps: a few iterations at each stage of the eps-scaling."""
    a, b = torch.empty_like(mu), torch.empty_like(mu)
    dd.domdec_full_sinkhorn(mu, nu, N, eps, lam, eps_start=max(eps, 0.125), precision=PRECISION[precision],
                            maxit=maxit, err=-1.0, alpha=a, beta=b)
    return a, b


def _handle(case, N, mu, nu, lam, a=None, b=None):
    eps = case["eps_px"] / N ** 2
    more = {} if a is None else dict(alpha0=a, beta0=b, eps_init=2 * eps)
    return dd.DomDec(mu, nu, eps, lam, case["s"], precision=case.get("precision", "fp32"),
                     strategy=case.get("strategy", "staggered"), cell_ti=case.get("ti", 0),
                     err=case.get("err", -1.0), maxit=case.get("maxit", 2000), **more)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        lams = (0.5, 1.0, 5.0)
        st = {"case": case, "handles": [], "out": [], "problems": []}
        for i, N in enumerate(_sides(case)):
            mu, nu = _image_pair("blobs", N, 100 * seed + i)
            lam = lams[i % 3]
            a, b = _duals(mu, nu, N, 2 * case["eps_px"] / N ** 2, lam)
            st["handles"].append(_handle(case, N, mu, nu, lam, a, b))
            st["out"].append([torch.empty_like(mu) for _ in range(3)])
            st["problems"].append((N, mu, nu, lam, a, b))
        st["batch"] = dd.DomDecBatch(st["handles"])
        return st
    N = case["N"]
    lam = case["lam"]
    eps = case["eps_px"] / N ** 2
    mu, nu = _image_pair(case.get("field", "blobs"), N, seed)
    st = {"case": case, "mu": mu, "nu": nu, "eps": eps}
    if kind == "sweeps":
        st["a0"], st["b0"] = (None, None) if case["start"] == "product" else _duals(mu, nu, N, 2 * eps, lam)
        st["handle"] = _handle(case, N, mu, nu, lam, st["a0"], st["b0"])
        st["out"] = [torch.empty_like(mu) for _ in range(3)]
    elif kind == "sinkhorn":
        st["out"] = [torch.empty_like(mu) for _ in range(2)]
    elif kind == "gap":
        st["a0"], st["b0"] = _duals(mu, nu, N, 2 * eps, lam, "fp64", 4)
        st["handle"] = _handle(case, N, mu, nu, lam, st["a0"], st["b0"])
        st["out"] = torch.empty_like(mu)
    elif kind == "grad":
        st["a"], st["b"] = _duals(mu, nu, N, eps, lam, "fp64", 4)
        st["out"] = [torch.empty_like(mu), torch.empty_like(mu), torch.empty(2 * N * N, dtype=F64, device="cuda")]
    else:
        st["mu"], st["nu"] = mu.float(), nu.float()
    return st


# ------------------------------------------------------------------- the pass
def _read(h, out, single):
    """Both marginals and the stitched dual of a handle, on the device."""
    dd.domdec_plan_marginals(h.h, out[0], out[1])
    dd.domdec_duals(h.h, out[2])
    return [t.float() if single else t for t in out]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "sweeps":
        h, single = st["handle"], case["precision"] == "fp32"
        h.reset(st["mu"], st["nu"], st["a0"], st["b0"], 0.0 if st["a0"] is None else 2 * st["eps"])
        h.iterate(case["sweeps"])
        h.sync()
        score = h.score()[:5]
        return [score.astype(np.float32) if single else score] + _read(h, st["out"], single)
    if kind == "batch":
        st["batch"].iterate(case["sweeps"])
        st["batch"].sync()
        return [_read(h, out, True) for h, out in zip(st["handles"], st["out"])]
    if kind == "sinkhorn":
        N, single = case["N"], case["precision"] != "fp64"
        alpha, beta = st["out"]
        solve = dd.domdec_full_sinkhorn_noalloc if case["noalloc"] else dd.domdec_full_sinkhorn
        it, _, primal, dual, _ = solve(st["mu"], st["nu"], N, st["eps"], case["lam"], eps_start=1.0,
                                       precision=PRECISION[case["precision"]], maxit=case["maxit"],
                                       err=case["err"], check_every=10, alpha=alpha, beta=beta)
        value = np.array([primal, dual], dtype=np.float32 if single else np.float64)
        return [it, value] + [t.float() if single else t for t in (alpha, beta)]
    if kind == "gap":
        out = dd.domdec_pd_gap(st["handle"].h, st["out"])
        return list(out) + [st["out"]]
    if kind == "grad":
        single = case["precision"] == "fp32"
        g_mu, g_nu, g_x = st["out"]
        value = dd.domdec_uot_gradients(st["mu"], st["nu"], st["a"], st["b"], case["N"], st["eps"], case["lam"],
                                        precision=PRECISION[case["precision"]], grad_mu=g_mu, grad_nu=g_nu,
                                        grad_x=g_x)
        value = np.array(value, dtype=np.float32 if single else np.float64)
        return [value] + [t.float() if single else t for t in (g_mu, g_nu, g_x)]
    from paper_2410_08859_gb300.autograd import uot_score
    mu, nu = st["mu"].clone().requires_grad_(True), st["nu"].clone().requires_grad_(True)
    score = uot_score(mu, nu, st["eps"], case["lam"], s=case["s"], gap=0.0, max_sweeps=case["sweeps"],
                      cell_err=-1.0, cell_maxit=case["maxit"], warm_err=-1.0, warm_maxit=case["maxit"])
    score.backward()
    return [score.detach(), mu.grad, nu.grad]


# ------------------------------------------------ the same in plain 64-bit torch
def _lse_grid(f, q):
    """log sum_y exp(f(y) - q |x - y|^2) for every pixel x of the grid (f: N x N)."""
    N = f.shape[0]
    t = torch.arange(N, device=f.device, dtype=F64)
    K = -q * (t[:, None] - t[None, :]) ** 2
    rows = max(1, (1 << 25) // (N * N))
    for _ in range(2):
        f = torch.cat([torch.logsumexp(f[i:i + rows, None, :] + K[None], 2) for i in range(0, N, rows)]).T
    return f


def _sinkhorn(mu, nu, N, eps_start, eps, lam, maxit, err, every=10):
    mu, nu = mu.view(N, N), nu.view(N, N)
    lmu, lnu = mu.log(), nu.log()
    alpha, beta, total = torch.zeros_like(mu), torch.zeros_like(mu), 0
    e = max(eps_start, eps)
    while True:
        kap, q = e / (1 + e / lam), 1.0 / (N * N * e)
        w = _lse_grid(beta / e + lnu, q)
        for it in range(1, maxit + 1):
            alpha = -kap * w
            z = _lse_grid(alpha / e + lmu, q)
            beta = -kap * z
            w = _lse_grid(beta / e + lnu, q)
            if it % every == 0 or it == maxit:
                px, ref = mu * (alpha / e + w).exp(), mu * (-alpha / lam).exp()
                pd = float((px * (px / ref).log() - px + ref).sum())
                if err >= 0 and pd <= err * float(mu.sum()):
                    break
        total += it
        if e <= eps:
            break
        e = max(eps, 0.5 * e)
    dual = float(eps * mu.sum() * nu.sum() - eps * (nu * (beta / eps + z).exp()).sum()
                 - lam * (((-alpha / lam).exp() - 1) * mu).sum() - lam * (((-beta / lam).exp() - 1) * nu).sum())
    return total, dual + lam * pd, dual, alpha.reshape(-1), beta.reshape(-1)


def _kl(p, m):
    return (torch.special.xlogy(p, p / m) - p + m).sum()


class _Plan:
    """The domain-decomposition state in 64 bits: dense basic-cell marginals."""

    def __init__(self, N, s, mu, nu, eps, lam, thr=1e-15):
        self.N, self.s, self.eps, self.lam, self.thr = N, s, eps, lam, thr
        self.mu, self.nu, self.nb = mu.view(N, N), nu.view(N, N), N // s
        self.lmu, self.lnu = self.mu.log(), self.nu.log()
        self.t = torch.arange(N, device=mu.device, dtype=F64)
        self.mass = self.mu.view(self.nb, s, self.nb, s).sum((1, 3)).reshape(-1)
        self.swept = 0

    def tighten(self):
        """Row and column range of every basic-cell marginal's support."""
        on = self.V > 0
        r, c = on.any(2), on.any(1)
        last = lambda m: self.N - m.flip(1).int().argmax(1)  # noqa: E731
        empty = ~r.any(1)
        box = torch.stack([r.int().argmax(1), last(r), c.int().argmax(1), last(c)], 1)
        box[empty] = torch.tensor([self.N, 0, self.N, 0], device=box.device)
        self.box = box
        self.PY = self.V.sum(0)

    def product(self):
        m, h2 = self.nu.sum(), 1.0 / self.N ** 2
        self.V = self.mass[:, None, None] * self.nu
        self.V[self.V < self.thr] = 0
        t = self.t
        c1 = (self.nu * ((t[:, None, None, None] - t[None, None, :, None]) ** 2
                         + (t[None, :, None, None] - t[None, None, None, :]) ** 2)).sum((2, 3)) * self.mu * h2
        self.C = c1.view(self.nb, self.s, self.nb, self.s).sum((1, 3)).reshape(-1)
        self.H = torch.zeros_like(self.C)
        self.PX, self.alpha = self.mu * m, torch.zeros_like(self.mu)
        self.tighten()

    def duals(self, a0, b0, eps0):
        N, s, nb = self.N, self.s, self.nb
        a0, b0 = a0.view(N, N) / eps0, b0.view(N, N) / eps0
        q = 1.0 / (N * N * eps0)
        t = self.t
        K = -q * (t[:, None] - t[None, :]) ** 2
        n = nb * nb
        self.V = torch.zeros(n, N, N, dtype=F64, device=a0.device)
        self.C, self.H = torch.zeros(n, dtype=F64, device=a0.device), torch.zeros(n, dtype=F64, device=a0.device)
        moments = []
        for i in range(n):
            r, c = slice(i // nb * s, (i // nb + 1) * s), slice(i % nb * s, (i % nb + 1) * s)
            v, cost, ent = _marginal(a0[r, c], self.lmu[r, c], K[:, r], K[:, c], b0, self.lnu, q)
            self.V[i] = torch.where(v < self.thr, 0.0, v)
            moments.append((v, cost, ent))
            if len(moments) == 16 or i == n - 1:   # the box is known once the marginal is
                lo = i + 1 - len(moments)
                on = self.V[lo:i + 1] > 0
                inside = (on.any(2).flip(1).cumsum(1).flip(1) > 0) & (on.any(2).cumsum(1) > 0)
                insidec = (on.any(1).flip(1).cumsum(1).flip(1) > 0) & (on.any(1).cumsum(1) > 0)
                for k, (v, cost, ent) in enumerate(moments):
                    m = (inside[k][:, None] & insidec[k][None, :]).double()
                    self.C[lo + k] = (m * cost).sum() / N ** 2
                    self.H[lo + k] = (m * ent).sum() - (m * cost).sum() * q - (m * v).sum() \
                        + self.mass[lo + k] * self.nu.sum()
                moments = []
        self.PX = self.mu * (a0 + _lse_grid(b0 + self.lnu, q)).exp()
        self.alpha = a0 * eps0
        self.tighten()

    def score(self, C=None, H=None, PX=None, PY=None):
        C, H, PX, PY = (x if x is not None else y for x, y in zip((C, H, PX, PY), (self.C, self.H, self.PX, self.PY)))
        loc = float(C.sum() + self.eps * H.sum())
        kx, ky = self.lam * float(_kl(PX, self.mu)), self.lam * float(_kl(PY.clamp(min=0), self.nu))
        return [loc + kx + ky, loc, kx, ky, float(PY.sum())]

    def sweep(self, strategy, ti, err, maxit):
        off = self.swept % 2
        self.swept += 1
        nc = self.nb // 2 + off
        cells = [(P, Q) for P in range(nc) for Q in range(nc)]
        groups = [[c for c in cells if 2 * (c[0] % 2) + c[1] % 2 == k] for k in range(4)]
        for g in (groups if strategy.startswith("staggered") else [cells]):
            if g:
                self.step([(2 * P - off, 2 * Q - off) for P, Q in g], strategy, ti, err, maxit)

    def step(self, corners, strategy, ti, err, maxit):
        """One batch of cells, `corners` their first basic cell (may lie outside the grid)."""
        N, s, nb, dev = self.N, self.s, self.nb, self.mu.device
        eps, lam = self.eps, self.lam
        q, sl, kap = 1.0 / (N * N * eps), eps / lam, eps / (1 + eps / lam)
        members = [[(i + a) * nb + j + b if 0 <= i + a < nb and 0 <= j + b < nb else -1 for a in (0, 1)
                    for b in (0, 1)] for i, j in corners]
        B, first = len(corners), torch.tensor(corners, device=dev) * s
        mem = torch.tensor(members, device=dev)
        x = torch.arange(2 * s, device=dev)
        xr, xc = first[:, :1] + x, first[:, 1:] + x
        inx = ((xr >= 0) & (xr < N))[:, :, None] & ((xc >= 0) & (xc < N))[:, None, :]
        gr, gc = xr.clamp(0, N - 1)[:, :, None], xc.clamp(0, N - 1)[:, None, :]
        bx = self.box[mem.clamp(min=0)]
        none = (mem < 0)[:, :, None]
        lo = torch.where(none, N, bx[:, :, 0::2]).amin(1)
        hi = torch.where(none, 0, bx[:, :, 1::2]).amax(1)
        Hm, Wm = (hi - lo).amax(0).tolist()
        yr, yc = lo[:, :1] + torch.arange(Hm, device=dev), lo[:, 1:] + torch.arange(Wm, device=dev)
        iny = (yr < hi[:, :1])[:, :, None] & (yc < hi[:, 1:])[:, None, :]
        hr, hc = yr.clamp(0, N - 1)[:, :, None], yc.clamp(0, N - 1)[:, None, :]
        inf = float("inf")
        lmu, mu = torch.where(inx, self.lmu[gr, gc], -inf), torch.where(inx, self.mu[gr, gc], 0.0)
        lnu, nu = torch.where(iny, self.lnu[hr, hc], -inf), self.nu[hr, hc]
        old = torch.where(iny[:, None] & (mem >= 0)[:, :, None, None],
                          self.V[mem.clamp(min=0)[:, :, None, None], hr[:, None], hc[:, None]], 0.0)
        rho = torch.where(iny, (self.PY[hr, hc] - old.sum(1)).clamp(min=0) / nu, 0.0)
        lrho, background = rho.log(), (rho * nu).sum((1, 2))
        Kr = -q * (yr[:, :, None] - xr[:, None, :]).double() ** 2   # B, H, 2s
        Kc = -q * (yc[:, :, None] - xc[:, None, :]).double() ** 2   # B, W, 2s
        alpha = torch.where(inx, self.alpha[gr, gc], 0.0)
        done = torch.zeros(B, dtype=torch.bool, device=dev)
        b, w = torch.zeros_like(rho), torch.zeros_like(alpha)
        for it in range(maxit):
            f = alpha / eps + lmu
            T = torch.logsumexp(f[:, :, None, :] + Kc[:, None], 3)
            z = torch.logsumexp(T[:, None] + Kr[:, :, :, None], 2)
            nb_ = _root(lrho, -sl * z, sl) - z
            U = torch.logsumexp((nb_ + lnu)[:, :, :, None] + Kc[:, None], 2)
            nw = torch.logsumexp(U[:, :, None, :] + Kr[:, :, :, None], 1)
            b, w = torch.where(done[:, None, None], b, nb_), torch.where(done[:, None, None], w, nw)
            if err >= 0:
                px, ref = mu * (alpha / eps + w).exp(), mu * (-alpha / lam).exp()
                gap = (torch.special.xlogy(px, torch.where(inx, px / ref, 1.0)) - px + ref).sum((1, 2))
                done = done | (gap <= err * mu.sum((1, 2)))
                if bool(done.all()):
                    break
            if it == maxit - 1:
                break
            new = -kap * w
            if ti:
                A = (mu * (-new / lam).exp()).sum((1, 2))
                Bn = torch.where(iny, nu * (-sl * b).exp(), 0.0).sum((1, 2))
                u = (background + (background ** 2 + 4 * A * Bn).sqrt()) / (2 * Bn)
                new = new + lam * u.log()[:, None, None]
            alpha = torch.where(done[:, None, None], alpha, new)
        px = mu * (alpha / eps + w).exp()
        nut, Ct, Ht = torch.zeros_like(old), torch.zeros(B, 4, dtype=F64, device=dev), \
            torch.zeros(B, 4, dtype=F64, device=dev)
        for k in range(4):
            r, c = slice(k // 2 * s, (k // 2 + 1) * s), slice(k % 2 * s, (k % 2 + 1) * s)
            have = mem[:, k] >= 0
            v, cost, ent = _marginal(alpha[:, r, c] / eps, lmu[:, r, c], Kr[:, :, r], Kc[:, :, c], b, lnu, q)
            keep = have[:, None, None] & iny
            v, cost, ent = (torch.where(keep, y, 0.0) for y in (v, cost, ent))
            nut[:, k] = v
            Ct[:, k] = cost.sum((1, 2)) / N ** 2
            Ht[:, k] = ent.sum((1, 2)) - cost.sum((1, 2)) * q - v.sum((1, 2)) \
                + self.mass[mem[:, k].clamp(min=0)] * self.nu.sum()
        C1, H1, PX1, PY1 = self.C.clone(), self.H.clone(), self.PX.clone(), self.PY.clone()
        ok = mem >= 0
        C1[mem[ok]], H1[mem[ok]] = Ct[ok], Ht[ok]
        PX1[gr.expand_as(px)[inx], gc.expand_as(px)[inx]] = px[inx]
        dpy = torch.where(iny, (nut - old).sum(1), 0.0)
        PY1.view(-1).index_add_(0, (hr * N + hc).reshape(-1), dpy.reshape(-1))
        now = (self.C, self.H, self.PX, self.PY)
        mixed = lambda th: [(1 - th) * x + th * y for x, y in zip(now, (C1, H1, PX1, PY1))]  # noqa: E731
        safe = 1.0 / B
        if strategy.endswith("line"):
            theta = _line(now, (C1, H1, PX1, PY1), self.mu, self.nu, eps, lam, safe)
        else:
            E0 = self.score()[0]
            theta = 1.0 if self.score(*mixed(1.0))[0] <= self.score(*mixed(safe))[0] + 1e-12 * abs(E0) else safe
        self.C, self.H, self.PX, _ = mixed(theta)
        self.alpha[gr.expand_as(px)[inx], gc.expand_as(px)[inx]] = alpha[inx]
        new = (1 - theta) * old + theta * nut
        new = torch.where(new < self.thr, 0.0, new)
        for j in range(B):
            h, wd = int(hi[j, 0] - lo[j, 0]), int(hi[j, 1] - lo[j, 1])
            for k in range(4):
                if members[j][k] >= 0:
                    self.V[members[j][k], lo[j, 0]:hi[j, 0], lo[j, 1]:hi[j, 1]] = new[j, k, :h, :wd]
        self.tighten()


def _marginal(a, lmu, Kr, Kc, b, lnu, q):
    """Of the plan exp(a + b - c/eps) mu nu over a block of X: per y its mass, its
    transport cost in squared pixels, and its sum of pi (a + b); separably."""
    f = (a + lmu).unsqueeze(-2) + Kc.unsqueeze(-3)                     # r, W, c
    T = torch.logsumexp(f, -1)
    p = torch.where(torch.isfinite(T)[..., None], (f - T[..., None]).exp(), 0.0)
    Ma = (p * a.unsqueeze(-2)).sum(-1)
    Md = (p * (-Kc / q).unsqueeze(-3)).sum(-1)
    g = T.unsqueeze(-3) + Kr.unsqueeze(-1)                             # H, r, W
    P = torch.logsumexp(g, -2)
    p = torch.where(torch.isfinite(P).unsqueeze(-2), (g - P.unsqueeze(-2)).exp(), 0.0)
    v = (b + lnu + P).exp()
    ma = (p * Ma.unsqueeze(-3)).sum(-2)
    md = (p * (Md.unsqueeze(-3) + (-Kr / q).unsqueeze(-1))).sum(-2)
    return v, v * md, v * (ma + b)


def _root(lrho, c0, s):
    """u with log(rho + e^u) + s u + c0 = 0, by Newton from the left of the two linear bounds' roots."""
    u = -c0 / (1 + s)
    u = torch.where(torch.isfinite(lrho), torch.minimum(u, -(lrho + c0) / s), u)
    for _ in range(60):
        la = torch.logaddexp(lrho, u)
        du = (la + s * u + c0) / ((u - la).exp() + s)
        u = u - du
        if float(du.abs().max()) <= 1e-14 * max(1.0, float(u.abs().max())):
            break
    return u


def _line(now, new, mu, nu, eps, lam, lo):
    """Minimiser over [lo, 1] of the convex tracked score along the mix (bisection on its derivative)."""
    d = [y - x for x, y in zip(now, new)]
    lin = d[0].sum() + eps * d[1].sum()

    def slope(z):
        g = lin
        for p, dp, m in ((now[2], d[2], mu), (now[3], d[3], nu)):
            on = dp != 0
            g = g + lam * (dp[on] * ((p[on] + z * dp[on]).clamp(min=1e-300) / m[on]).log()).sum()
        return float(g)

    if slope(1.0) <= 0:
        return 1.0
    if slope(lo) >= 0:
        return lo
    a, b = lo, 1.0
    for _ in range(52):
        m = 0.5 * (a + b)
        a, b = (a, m) if slope(m) > 0 else (m, b)
    return 0.5 * (a + b)


def _gradients(mu, nu, a, b, N, eps, lam):
    """Value terms and gradients of the dual at fixed potentials (N x N images)."""
    q = 1.0 / (N * N * eps)
    pen = lambda p: -lam * torch.expm1(-p / lam)  # noqa: E731
    rx, ry = (a / eps + _lse_grid(b / eps + nu.log(), q)).exp(), (b / eps + _lse_grid(a / eps + mu.log(), q)).exp()
    mx, my = float(mu.sum()), float(nu.sum())
    value = [eps * mx * my - eps * float((mu * rx).sum()) + float((pen(a) * mu).sum() + (pen(b) * nu).sum()),
             mx, my, float((mu * rx).sum()), float((nu * ry).sum())]
    # barycentric displacement, one axis at a time
    f = b / eps + nu.log()
    t = torch.arange(N, device=f.device, dtype=F64)
    d = t[None, :] - t[:, None]
    rows = max(1, (1 << 24) // (N * N))

    def axis(f, g):   # along the last axis: log-sum, mean displacement, mean of g
        L, M, G = [], [], []
        for i in range(0, N, rows):
            e = f[i:i + rows, None, :] - q * d[None] ** 2
            l = torch.logsumexp(e, 2)
            p = (e - l[..., None]).exp()
            L.append(l)
            M.append((p * d[None]).sum(2))
            if g is not None:
                G.append((p * g[i:i + rows, None, :]).sum(2))
        return torch.cat(L), torch.cat(M), torch.cat(G) if G else None

    A, m, _ = axis(f, None)
    _, M1, M2 = axis(A.T.contiguous(), m.T.contiguous())
    gx = -2.0 * (mu * rx)[..., None] / N * torch.stack([M1.T, M2.T], -1)
    return value, eps * my - eps * rx + pen(a), eps * mx - eps * ry + pen(b), gx


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sweeps", "score") and case["N"] > 400:
        return None   # the dense 64-bit state would take minutes
    if kind == "batch" and case["count"] * case["side_hi"] ** 2 * case["maxit"] * case["sweeps"] > 2.5e7:
        return None
    st = prepare(case, seed)
    if kind == "batch":
        outs = []
        for N, mu, nu, lam, a, b in st["problems"]:
            p = _Plan(N, case["s"], mu, nu, case["eps_px"] / N ** 2, lam)
            p.duals(a, b, 2 * p.eps)
            for _ in range(case["sweeps"]):
                p.sweep("staggered", 0, -1.0, case["maxit"])
            outs.append([x.reshape(-1) for x in (p.PX, p.PY, p.alpha)])
        return outs
    N, lam, eps, mu, nu = case["N"], case["lam"], st["eps"], st["mu"].double(), st["nu"].double()
    if kind == "sinkhorn":
        it, primal, dual, a, b = _sinkhorn(mu, nu, N, 1.0, eps, lam, case["maxit"], case["err"])
        return [it, np.array([primal, dual]), a, b]
    if kind == "grad":
        value, g_mu, g_nu, g_x = _gradients(*(x.view(N, N) for x in (mu, nu, st["a"], st["b"])), N, eps, lam)
        return [np.array(value), g_mu.reshape(-1), g_nu.reshape(-1), g_x.reshape(-1)]
    if kind == "gap":
        M, W = mu.view(N, N), nu.view(N, N)
        a, q, kap = st["a0"].view(N, N), 1.0 / (N * N * eps), eps / (1 + eps / lam)
        z = _lse_grid(a / eps + M.log(), q)
        b = -kap * z
        D = float(eps * M.sum() * W.sum() - eps * (W * (b / eps + z).exp()).sum()
                  - lam * (M * torch.expm1(-a / lam)).sum() - lam * (W * torch.expm1(-b / lam)).sum())
        px = M * (a / (2 * eps) + _lse_grid(st["b0"].view(N, N) / (2 * eps) + W.log(), q / 2)).exp()
        ex = float((px - M * (-a / lam).exp()).abs().sum())
        return [None, np.float64(D), None, np.float64(ex), None, b.reshape(-1)]
    if kind == "sweeps":
        p = _Plan(N, case["s"], mu, nu, eps, lam)
        if case["start"] == "product":
            p.product()
        else:
            p.duals(st["a0"], st["b0"], 2 * eps)
        for _ in range(case["sweeps"]):
            p.sweep(case["strategy"], case["ti"], case["err"], case["maxit"])
        return [np.array(p.score())] + [x.reshape(-1) for x in (p.PX, p.PY, p.alpha)]
    a, b = _sinkhorn(mu, nu, N, 1.0, 2 * eps, lam, case["maxit"], -1.0)[3:]
    p = _Plan(N, case["s"], mu, nu, eps, lam)
    p.duals(a, b, 2 * eps)
    for _ in range(case["sweeps"]):
        p.sweep("staggered", 0, -1.0, case["maxit"])
    z = _lse_grid(p.alpha / eps + p.lmu, 1.0 / (N * N * eps))
    _, g_mu, g_nu, _ = _gradients(p.mu, p.nu, p.alpha, -eps / (1 + eps / lam) * z, N, eps, lam)
    return [np.float64(p.score()[0]), g_mu.reshape(-1), g_nu.reshape(-1)]
