"""The tile and window kernels at the sizes where they can go wrong, against plain
64-bit torch: the separable Sinkhorn passes and the adjoint (edges of the
8-target tiles and of the 16-source blocks, eps so small that the table of
powers does not cover a window, eps so large that every source is kept), the
tile-wise box test of a dual-initialised plan,
and cells whose per-y arrays lie in a spill slot on one CTA and on a cluster."""
import numpy as np
import pytest

from oracle import domdec as odd
from paper_2410_08859_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2410_08859_gb300 import domdec
    return torch, domdec


def lse(torch, f, q):
    """log sum_y exp(f(y) - q |x - y|^2), f: N x N."""
    N = f.shape[0]
    t = torch.arange(N, device=f.device, dtype=torch.float64)
    K = -q * (t[:, None] - t[None, :]) ** 2
    for _ in range(2):
        f = torch.logsumexp(f[:, None, :] + K[None], 2).T
    return f


# tolerances: a potential's exponent f carries one rounding of |f| in every pass; in double that is
# ~1e-16 |pot| each (12 passes and the table's powers: 1e-12), in float ~1e-7 |pot| (5e-6)
@pytest.mark.parametrize("N", [1, 5, 8, 9, 31, 64, 128, 129, 200])
@pytest.mark.parametrize("eps_px", [0.2, 1.0, 4.0, 1e9])
@pytest.mark.parametrize("precision,tol", [(1, 1e-12), (0, 5e-6), (2, 5e-6)])
def test_separable_sinkhorn_edges(env, N, eps_px, precision, tol):
    torch, dd = env
    eps, lam = min(eps_px / N ** 2, 0.5), 0.8
    if precision == 0 and eps_px < 4.0:
        pytest.skip("single precision is for coarse eps")
    mu, nu = inputs.mixture_blobs(N=N, seed=7)
    mu, nu = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (mu, nu))
    a, b = torch.empty_like(mu), torch.empty_like(mu)
    dd.domdec_full_sinkhorn(mu, nu, N, eps, lam, eps_start=eps, precision=precision, maxit=3, err=-1.0,
                            check_every=2, alpha=a, beta=b)
    kap, q = eps / (1 + eps / lam), 1.0 / (N * N * eps)
    beta = torch.zeros_like(mu)
    for _ in range(3):
        alpha = -kap * lse(torch, beta / eps + nu.log(), q)
        beta = -kap * lse(torch, alpha / eps + mu.log(), q)
    for got, ref in ((a, alpha), (b, beta)):
        assert float((got - ref).abs().max()) <= tol * (float(ref.abs().max()) + eps)


@pytest.mark.parametrize("N", [1, 7, 16, 33, 129])
@pytest.mark.parametrize("eps_px", [0.3, 4.0])
def test_adjoint_edges(env, N, eps_px):
    torch, dd = env
    eps, lam = eps_px / N ** 2, 1.3
    rng = np.random.default_rng(N)
    mu, nu = inputs.mixture_blobs(N=N, seed=8)
    t = np.arange(N) / N
    # an expanding displacement plus noise, so that neighbouring targets take distant sources
    alpha = 0.05 * np.sin(6 * t[:, None] + 3 * t[None, :]) + 0.3 * (t[:, None] - 0.4) ** 2 + eps * rng.normal(size=(N, N))
    beta = -0.05 * np.cos(5 * t[None, :]) + eps * rng.normal(size=(N, N))
    d = [torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64).ravel()).cuda() for x in (mu, nu, alpha, beta)]
    n = N * N
    gm, gn, gx = (torch.empty(k * n, dtype=torch.float64, device="cuda") for k in (1, 1, 2))
    dd.domdec_uot_gradients(*d, N, eps, lam, precision=dd.FP64, grad_mu=gm, grad_nu=gn, grad_x=gx)
    m, w, a, b = (x.cpu().numpy() for x in d)
    I, J = np.divmod(np.arange(n), N)
    scale = {"m": float(gm.abs().max()), "n": float(gn.abs().max()), "x": float(gx.abs().max()) + 1e-300}
    for x in rng.choice(n, size=min(n, 25), replace=False):
        c = ((I - I[x]) ** 2 + (J - J[x]) ** 2) / N ** 2
        with np.errstate(over="ignore", invalid="ignore"):
            row = np.exp((a[x] + b - c) / eps) * w         # pi(x, .) / mu(x)
            col = np.exp((a + b[x] - c) / eps) * m
        if not (np.isfinite(row.sum()) and np.isfinite(col.sum())):
            continue   # beyond double: no reference
        g_mu = eps * w.sum() - eps * row.sum() - lam * np.expm1(-a[x] / lam)
        g_nu = eps * m.sum() - eps * col.sum() - lam * np.expm1(-b[x] / lam)
        # exponents of magnitude ~1/eps: one rounding of them is a relative 1e-16/eps of a term
        tol = 1e-11 + 4e-15 / eps
        assert abs(float(gm[x]) - g_mu) <= tol * max(scale["m"], eps * row.sum())
        assert abs(float(gn[x]) - g_nu) <= tol * max(scale["n"], eps * col.sum())
        for ax, P in ((0, I), (1, J)):
            ref = -2.0 * m[x] * float((row * (P - P[x])).sum()) / N
            assert abs(float(gx[2 * x + ax]) - ref) <= tol * max(scale["x"], abs(ref))


@pytest.mark.parametrize("N", [191, 192, 200, 401])
@pytest.mark.parametrize("eps_px", [0.2, 4.0, 1e4])
def test_adjoint_tiles_at_a_y_half(env, N, eps_px):
    """The double tile passes around the smallest grid they serve, at potentials of
    a plan: beta is the Y-half of a rough alpha, so every column has mass about 1;
    eps from below the range of the power table to every source kept."""
    torch, dd = env
    eps, lam = min(eps_px / N ** 2, 0.5), 0.9
    rng = np.random.default_rng(N)
    mu, nu = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in inputs.mixture_blobs(N=N, seed=11))
    t = np.arange(N) / N
    alpha = torch.from_numpy(0.02 * np.sin(7 * t[:, None] + 2 * t[None, :]) + 0.2 * (t[None, :] - 0.3) ** 2
                             + 0.5 * eps * rng.normal(size=(N, N))).cuda()
    q = 1.0 / (N * N * eps)
    beta = -eps / (1 + eps / lam) * lse(torch, alpha / eps + mu.log(), q)
    gm, gn, gx = (torch.empty(k * N * N, dtype=torch.float64, device="cuda") for k in (1, 1, 2))
    flat = [x.reshape(-1).contiguous() for x in (mu, nu, alpha, beta)]
    dd.domdec_uot_gradients(*flat, N, eps, lam, precision=dd.FP64, grad_mu=gm, grad_nu=gn, grad_x=gx)
    ry = (beta / eps + lse(torch, alpha / eps + mu.log(), q)).exp()
    rx = (alpha / eps + lse(torch, beta / eps + nu.log(), q)).exp()
    r_mu = eps * nu.sum() - eps * rx - lam * torch.expm1(-alpha / lam)
    r_nu = eps * mu.sum() - eps * ry - lam * torch.expm1(-beta / lam)
    # exponents of magnitude f = pot/eps: one rounding of them in each pass
    tol = 1e-12 + 1e-15 * float(max(alpha.abs().max(), beta.abs().max())) / eps
    assert float((gm - r_mu.reshape(-1)).abs().max()) <= tol * float(r_mu.abs().max() + eps * rx.abs().max())
    assert float((gn - r_nu.reshape(-1)).abs().max()) <= tol * float(r_nu.abs().max() + eps * ry.abs().max())
    # grad_x at sampled points, term by term
    I, J = torch.meshgrid(*(torch.arange(N, device="cuda", dtype=torch.float64),) * 2, indexing="ij")
    for x in rng.choice(N * N, size=12, replace=False):
        i, j = divmod(int(x), N)
        row = ((alpha[i, j] + beta) / eps - q * ((I - i) ** 2 + (J - j) ** 2)).exp() * nu
        for ax, P, p in ((0, I, i), (1, J, j)):
            ref = -2.0 * float(mu[i, j]) * float((row * (P - p)).sum()) / N
            bound = 2.0 * float(mu[i, j]) * float((row * (P - p).abs()).sum()) / N
            assert abs(float(gx[2 * x + ax]) - ref) <= 4 * tol * (bound + float(gx.abs().max()) * 1e-3)


@pytest.mark.parametrize("N,s", [(24, 3), (40, 4), (56, 7)])
def test_dual_initialised_boxes_match_oracle(env, N, s):
    """Grids that are no multiple of the box test's 16 x 16 tiles: boxes, values and costs."""
    torch, dd = env
    mu, nu = inputs.mixture_blobs(N=N, seed=9)
    mu, nu = mu.ravel(), nu.ravel()
    eps = 1.5 / N ** 2
    m, w = (torch.from_numpy(x.copy()).cuda() for x in (mu, nu))
    a, b = torch.empty_like(m), torch.empty_like(m)
    dd.domdec_full_sinkhorn(m, w, N, 2 * eps, 1.0, eps_start=1.0, maxit=20, err=-1.0, alpha=a, beta=b)
    geo = odd.Geometry(N, s)
    st = odd.init_from_duals(geo, mu, nu, a.cpu().numpy(), b.cpu().numpy(), 2 * eps, eps, 1.0)
    with dd.DomDec(mu, nu, eps, 1.0, s, alpha0=a, beta0=b, eps_init=2 * eps, precision="fp64") as g:
        box, vals = g.basic_marginals()
        pos = 0
        for i in range(geo.nbasic):
            k0, l0, H, W = box[i]
            assert (k0, l0) == tuple(st.lo[i]) and (k0 + H, l0 + W) == tuple(st.hi[i]), i
            assert np.abs(vals[pos:pos + H * W].reshape(H, W) - st.vals[i]).max() <= 1e-12 * st.vals[i].max()
            pos += H * W
        C, Hh = g.basic_costs()
        assert np.abs(C - st.Cc).max() <= 1e-9 * st.Cc.max()   # the oracle sums outside the box too (< 1e-15 each)
        assert np.abs(Hh - st.Hh).max() <= 1e-9 * np.abs(st.Hh).max()


@pytest.mark.parametrize("ctas", [1, 2, 4])
def test_boxes_beyond_shared_memory(env, ctas, precision="fp64", tol=1e-11):
    """192 x 192 boxes of a product plan: per-y arrays in the slot on one CTA (T, U and
    beta in shared memory where they fit) and on clusters; against a run on the
    largest cluster."""
    torch, dd = env
    N, s = 192, 8
    mu, nu = inputs.mixture_blobs(N=N, seed=10)
    eps = 16.0 / N ** 2
    out = []
    for c in (8, ctas):
        with dd.DomDec(mu, nu, eps, 1.0, s, precision=precision, cell_ctas=c, err=-1.0, maxit=3, strategy="safe",
                       spill_slots=144) as g:
            g.iterate(1)
            g.sync()
            out.append((*g.marginals(), g.duals(), g.cell_log()))
    ref, got = out
    assert (got[3][:, 7] >= 0).any()   # cells with a slot
    for k in range(2):
        assert np.abs(got[k] - ref[k]).sum() <= tol * np.abs(ref[k]).sum()
    assert np.abs(got[2] - ref[2]).max() <= tol * (1 + np.abs(ref[2]).max())


@pytest.mark.parametrize("ctas", [2, 4, 8])
@pytest.mark.parametrize("N,s", [(48, 4), (96, 8), (160, 16)])
def test_translation_step_on_clusters(env, N, s, ctas):
    """Cells with the translation step on a cluster against one CTA each, two sweeps (the
    second with the ragged boundary cells) of a fixed number of iterations.  In double the sums
    in another order differ by ~1e-16; t*/eps = log(u)/s amplifies that by 1/s (here up to 6.4e3)."""
    torch, dd = env
    mu, nu = inputs.mixture_blobs(N=N, seed=11)
    eps = 4.0 / N ** 2
    out = []
    for c in (1, ctas):
        with dd.DomDec(mu, nu, eps, 1.0, s, precision="fp64", cell_ctas=c, cell_ti=1, err=-1.0, maxit=4,
                       strategy="safe", spill_slots=100) as g:
            g.iterate(2)
            g.sync()
            out.append((*g.marginals(), g.duals()))
    ref, got = out
    for k in range(2):
        assert np.abs(got[k] - ref[k]).sum() <= 1e-11 * np.abs(ref[k]).sum()
    assert np.abs(got[2] - ref[2]).max() <= 1e-11 * (1 + np.abs(ref[2]).max())


def test_boxes_that_a_larger_cluster_holds_take_no_slot(env):
    """176 x 176 boxes fit the shared memory of four CTAs but not of two: with a launch on two and a
    single spill slot for many cells the sweep regroups to four."""
    torch, dd = env
    N, s = 176, 8
    mu, nu = inputs.mixture_blobs(N=N, seed=12)
    with dd.DomDec(mu, nu, 16.0 / N ** 2, 1.0, s, precision="fp32", err=-1.0, maxit=2, strategy="staggered",
                   spill_slots=1) as g:
        assert g.set_launch(2, 2.0) == 2
        g.iterate(1)
        g.sync()
        assert g.stats()["cluster_regroups"] >= 1
        PX, PY = g.marginals()
    assert abs(PX.sum() - PY.sum()) <= 1e-5 * PX.sum()
