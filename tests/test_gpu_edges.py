"""Rarely met paths of the kernels, each where it can go wrong: the stop on a
tolerance of cells on clusters, windows in the adjoint at very small eps,
values far outside the usual range, large grids, several host threads."""
import numpy as np
import pytest

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


# ---------------------------------------------------- stop on a tolerance on clusters
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("N,s", [(16, 2), (32, 4), (64, 8), (64, 16)])
@pytest.mark.parametrize("ctas", [2, 4, 8])
def test_stop_on_a_tolerance_on_clusters(env, N, s, ctas, precision):
    """Cells of uneven iteration counts on clusters, with most warps of a CTA idle in the
    small cells: every cell ends within the tolerance, and each of several runs gives the
    result of one CTA per cell (P_Y is accumulated by atomic additions, so runs differ by
    roundings)."""
    torch, dd = env
    mu, nu = inputs.mixture_blobs(N=N, seed=21)
    eps, err = 4.0 / N ** 2, 1e-4
    lam = 100.0 * eps   # the slowest mode of a cell contracts by 1/(1 + eps/lam): some hundred iterations
    out = []
    for c in (1, ctas, ctas, ctas):
        with dd.DomDec(mu, nu, eps, lam, s, precision=precision, cell_ctas=c, err=err, maxit=3000, strategy="safe",
                       spill_slots=100) as g:
            g.iterate(2)
            g.sync()
            out.append((g.cell_log(), *g.marginals()))
    m = np.pad(mu, s)   # the second sweep's cells are offset by s
    cell = m.reshape(m.shape[0] // (2 * s), 2 * s, -1, 2 * s).sum((1, 3)).max()
    one = out[0]
    for got in out:
        assert (got[0][:, 5] == 0).all()
        assert (got[0][:, 6] <= err * cell * (1 + 1e-6)).all()
        if precision == "fp64":   # sums in another order (1e-16) through hundreds of contracting iterations
            assert np.array_equal(got[0][:, :5], one[0][:, :5])
            for k in (1, 2):
                assert np.abs(got[k] - one[k]).sum() <= 1e-9 * np.abs(one[k]).sum()
        else:   # each side's P_X is within sqrt(2 gap |mu|) of its cells' limit (Pinsker), in both sweeps
            assert np.abs(got[1] - one[1]).sum() <= 4.0 * np.sqrt(2.0 * err) * mu.sum()


# ------------------------------------------------------ adjoint at very small eps
def lse(torch, f, q):
    """log sum_y exp(f(y) - q |x - y|^2), f: N x N."""
    N = f.shape[0]
    t = torch.arange(N, device=f.device, dtype=torch.float64)
    K = -q * (t[:, None] - t[None, :]) ** 2
    for _ in range(2):
        f = torch.cat([torch.logsumexp(f[i:i + 64, None, :] + K[None], 2) for i in range(0, N, 64)]).T
    return f


@pytest.mark.parametrize("N", [192, 259])
@pytest.mark.parametrize("eps_px", [0.005, 0.1, 0.5, 0.9, 0.95])
@pytest.mark.parametrize("rows", [0.0, 60.0])
@pytest.mark.parametrize("half", ["x", "y"])
def test_adjoint_windows_at_small_eps(env, N, eps_px, rows, half):
    """The double tile passes below eps = 0.93 h^2, where the table of powers is short, at
    potentials that jump by `rows` units of eps from row to row (every line's block maxima are
    its own).  One potential is the closed-form half of the other, so the ratio P/w that the
    gradient carries is e^{-pot/lam} in every pixel of that side."""
    torch, dd = env
    rng = np.random.default_rng(N)
    eps = eps_px / N ** 2
    lam = 500.0 * eps
    mu, nu = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in inputs.mixture_blobs(N=N, seed=12))
    t = np.arange(N) / N
    rough = torch.from_numpy(2.0 * eps * (np.sin(7 * t[:, None] + 2 * t[None, :]) + rng.normal(size=(N, N)))
                             + eps * rows * rng.uniform(-1, 1, size=(N, 1))).cuda()
    q, kap = 1.0 / (N * N * eps), eps / (1 + eps / lam)
    if half == "y":
        alpha = rough
        beta = -kap * lse(torch, alpha / eps + mu.log(), q)
    else:
        beta = rough
        alpha = -kap * lse(torch, beta / eps + nu.log(), q)
    flat = [x.reshape(-1).contiguous() for x in (mu, nu, alpha, beta)]
    g = [torch.empty(N * N, dtype=torch.float64, device="cuda") for _ in range(2)]
    dd.domdec_uot_gradients(*flat, N, eps, lam, precision=dd.FP64, grad_mu=g[0], grad_nu=g[1])
    ry = (beta / eps + lse(torch, alpha / eps + mu.log(), q)).exp()
    rx = (alpha / eps + lse(torch, beta / eps + nu.log(), q)).exp()
    # exponents of magnitude f = pot/eps: one rounding of them in each pass
    tol = 1e-12 + 1e-15 * float(max(alpha.abs().max(), beta.abs().max())) / eps
    if half == "y":
        ref, r, got = eps * mu.sum() - eps * ry - lam * torch.expm1(-beta / lam), ry, g[1]
    else:
        ref, r, got = eps * nu.sum() - eps * rx - lam * torch.expm1(-alpha / lam), rx, g[0]
    err = (got.view(N, N) - ref).abs()
    assert float((err / (ref.abs() + eps * r + eps)).max()) <= tol


@pytest.mark.parametrize("N", [200, 409])
def test_adjoint_tiles_summed_term_by_term(env, N):
    """Single pixels that stand 300 units of eps above their line: the sums of the tile's other
    targets leave the accepted range and are repeated term by term, by one lane of the group for
    all of its targets.  Equal in repeated calls and equal to plain torch."""
    torch, dd = env
    rng = np.random.default_rng(N)
    eps = 4.0 / N ** 2
    lam = 500.0 * eps
    mu, nu = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in inputs.mixture_blobs(N=N, seed=13))
    a = eps * rng.normal(size=(N, N))
    a[rng.integers(0, N, 40), rng.integers(0, N, 40)] += 300.0 * eps
    a[rng.integers(0, N, 40), rng.integers(0, N, 40)] -= 300.0 * eps
    alpha = torch.from_numpy(a).cuda()
    q = 1.0 / (N * N * eps)
    beta = -eps / (1 + eps / lam) * lse(torch, alpha / eps + mu.log(), q)
    flat = [x.reshape(-1).contiguous() for x in (mu, nu, alpha, beta)]
    out = []
    for _ in range(3):
        g = torch.empty(N * N, dtype=torch.float64, device="cuda")
        dd.domdec_uot_gradients(*flat, N, eps, lam, precision=dd.FP64, grad_nu=g)
        out.append(g.view(N, N))
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    ry = (beta / eps + lse(torch, alpha / eps + mu.log(), q)).exp()
    ref = eps * mu.sum() - eps * ry - lam * torch.expm1(-beta / lam)
    tol = 1e-12 + 1e-15 * float(max(alpha.abs().max(), beta.abs().max())) / eps
    assert float(((out[0] - ref).abs() / (ref.abs() + eps * ry + eps)).max()) <= tol


# ------------------------------------------------------ potentials of any magnitude
@pytest.mark.parametrize("shift", [1e3, 2e10])
def test_dual_initialised_plan_of_shifted_potentials(env, shift):
    """alpha0 + K, beta0 - K is the same plan for every K; K = shift eps costs it the roundings of
    exponents of that size (two in each of the sums over rows and columns)."""
    torch, dd = env
    N, s = 24, 3
    mu, nu = inputs.mixture_blobs(N=N, seed=9)
    eps = 1.5 / N ** 2
    a, b = np.empty((N, N)), np.empty((N, N))
    dd.domdec_full_sinkhorn(mu, nu, N, 2 * eps, 1.0, eps_start=1.0, maxit=20, err=-1.0, alpha=a, beta=b)
    out = []
    for k in (0.0, shift * 2 * eps):
        with dd.DomDec(mu, nu, eps, 1.0, s, alpha0=a + k, beta0=b - k, eps_init=2 * eps, precision="fp64") as g:
            out.append((*g.marginals(), g.basic_costs()[0]))
    tol = 8 * 2.0 ** -52 * shift + 1e-12
    for ref, got in zip(*out):
        assert np.abs(got - ref).sum() <= tol * np.abs(ref).sum()


# --------------------------------------------- separable passes with and without windows
@pytest.mark.parametrize("N", [16, 31, 200])
@pytest.mark.parametrize("reach", [5.0, 63.9, 64.1, 300.0])
@pytest.mark.parametrize("precision,tol", [(0, 5e-6), (1, 1e-12)])
def test_separable_passes_around_whole_rows(env, N, reach, precision, tol):
    """q2 (N - 1)^2 on both sides of 64, where the search for windows starts; beta = 0, and in double
    also a start whose exponents range over 200 (a potential is within one rounding of its
    exponents a pass; single precision accepts a previous value that the sum has left by up to
    2^30 as its shift, so its first iterations after such a start are coarse)."""
    torch, dd = env
    q2 = reach / (N - 1) ** 2
    q = q2 * np.log(2.0)
    eps, lam = 1.0 / (N * N * q), 0.8
    mu, nu = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in inputs.mixture_blobs(N=N, seed=7))
    t = torch.arange(N, device="cuda", dtype=torch.float64) / N
    for start in (None, eps * 200.0 * (t[:, None] * t[None, :] - 0.5).contiguous())[:1 + precision]:
        a, b = torch.empty_like(mu), torch.empty_like(mu)
        dd.domdec_full_sinkhorn(mu, nu, N, eps, lam, eps_start=eps, precision=precision, maxit=3, err=-1.0,
                                check_every=2, beta_in=start, alpha=a, beta=b)
        kap = eps / (1 + eps / lam)
        beta = torch.zeros_like(mu) if start is None else start
        for _ in range(3):
            alpha = -kap * lse(torch, beta / eps + nu.log(), q)
            beta = -kap * lse(torch, alpha / eps + mu.log(), q)
        for got, ref in ((a, alpha), (b, beta)):
            scale = float(ref.abs().max()) + (0.0 if start is None else float(start.abs().max()))
            assert float((got - ref).abs().max()) <= tol * (scale + eps)


# ------------------------------------------------------------------- large grids
@pytest.mark.parametrize("N,precision,tol", [(5600, 1, 1e-12), (8000, 1, 1e-12), (5600, 2, 1e-6), (8000, 0, 1e-6)])
def test_separable_sinkhorn_on_large_grids(env, N, precision, tol):
    """Rows that leave no room for a whole row of results: alpha of the first half-step at sampled
    pixels, from the sources within e^-60 of them (the tolerances are relative to the largest
    exponent, log nu)."""
    torch, dd = env
    free, _ = torch.cuda.mem_get_info()
    if free < 30 * N * N * 8:
        pytest.skip("not enough device memory")
    g = torch.Generator(device="cuda").manual_seed(N)
    mu = torch.rand(N, N, generator=g, device="cuda", dtype=torch.float64) + 0.5
    nu = torch.rand(N, N, generator=g, device="cuda", dtype=torch.float64) + 0.5
    mu, nu = mu / mu.sum(), nu / nu.sum()
    eps_px = 100.0 if precision == 0 else 4.0
    eps, lam = eps_px / N ** 2, 1.0
    a = torch.zeros_like(mu)
    dd.domdec_full_sinkhorn(mu, nu, N, eps, lam, eps_start=eps, precision=precision, maxit=1, err=-1.0, alpha=a)
    rng, w = np.random.default_rng(N), int((60 * eps_px) ** 0.5) + 1
    for i, j in [(0, 0), (N - 1, N - 1), (N // 2, N - 1)] + [tuple(rng.integers(0, N, 2)) for _ in range(60)]:
        i0, i1, j0, j1 = max(0, i - w), min(N, i + w + 1), max(0, j - w), min(N, j + w + 1)
        I = torch.arange(i0, i1, device="cuda", dtype=torch.float64)[:, None] - int(i)
        J = torch.arange(j0, j1, device="cuda", dtype=torch.float64)[None, :] - int(j)
        ref = -eps / (1 + eps / lam) * torch.logsumexp((nu[i0:i1, j0:j1].log() - (I * I + J * J) / eps_px).reshape(-1), 0)
        assert abs(float(a[i, j]) - float(ref)) <= tol * 20 * eps


def test_separable_sinkhorn_reports_rows_that_do_not_fit(env):
    """A row of 8300 doubles with its tables is beyond shared memory: an error, not untouched output;
    the library goes on working."""
    torch, dd = env
    N = 8300
    free, _ = torch.cuda.mem_get_info()
    if free < 30 * N * N * 8:
        pytest.skip("not enough device memory")
    mu = torch.full((N * N,), 1.0 / N ** 2, dtype=torch.float64, device="cuda")
    with pytest.raises(dd.DomDecError) as e:
        dd.domdec_full_sinkhorn(mu, mu, N, 4.0 / N ** 2, 1.0, precision=1, maxit=1, err=-1.0)
    assert e.value.code == dd.DOMDEC_ECUDA
    m = torch.full((1024,), 1.0 / 1024, dtype=torch.float64, device="cuda")
    assert dd.domdec_full_sinkhorn(m, m, 32, 0.01, 1.0, precision=1, maxit=5, err=-1.0)[0] == 5


# ------------------------------------------------------------------ several host threads
def test_threads_with_grids_of_different_sizes(env):
    """The same kernels launched from threads whose calls need different amounts of shared memory, each
    on its own stream: what one thread asks for must not shrink what another is about to
    launch with.  Every result equals the one of a thread alone."""
    import threading
    torch, dd = env
    jobs = []
    for N, prec in ((1200, dd.FP64), (2000, dd.FP64), (1600, dd.FP64), (1200, dd.MIXED)):
        g = torch.Generator(device="cuda").manual_seed(N)
        mu = torch.rand(N * N, generator=g, device="cuda", dtype=torch.float64) + 0.5
        mu /= mu.sum()
        jobs.append([N, prec, mu, torch.empty_like(mu), torch.empty_like(mu), torch.empty_like(mu), torch.empty_like(mu)])

    def solve(N, prec, mu, a, b, gm, gx, stream=None):
        eps = 4.0 / N ** 2
        dd.domdec_full_sinkhorn(mu, mu, N, eps, 1.0, eps_start=eps, precision=prec, maxit=4, err=-1.0, check_every=2,
                                alpha=a, beta=b, stream=stream)
        dd.domdec_uot_gradients(mu, mu, a, b, N, eps, 1.0, grad_mu=gm, grad_nu=gx, stream=stream)

    ref = []
    for j in jobs:
        solve(*j)
        ref.append([t.clone() for t in j[3:]])
        for t in j[3:]:
            t.zero_()
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            st = torch.cuda.Stream()
            for _ in range(6):
                solve(*jobs[k], stream=st)
        except Exception as e:   # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for j, r in zip(jobs, ref):
        for got, want in zip(j[3:], r):
            assert torch.equal(got, want)


# ------------------------------------------- single-precision cells beyond shared memory
# eps/lam = 1/4, so a root amplifies a rounding four times at most; an exponent of magnitude
# below 50 costs 3e-6 a pass, and there are four passes in each of three iterations
FP32_TOL = 1e-4


def test_fp32_boxes_beyond_shared_memory(env):
    """192 x 192 boxes of a product plan in single precision: the list of slow roots, the tiles and
    the odd pitches with per-y arrays in a slot, on one CTA and on clusters, against double cells."""
    torch, dd = env
    N, s = 192, 8
    mu, nu = inputs.mixture_blobs(N=N, seed=10)
    eps = 16.0 / N ** 2
    out = []
    for precision, c in (("fp64", 8), ("fp32", 1), ("fp32", 2), ("fp32", 4), ("fp32", 8)):
        with dd.DomDec(mu, nu, eps, 4 * eps, s, precision=precision, cell_ctas=c, err=-1.0, maxit=3, strategy="safe",
                       spill_slots=144) as g:
            g.iterate(1)
            g.sync()
            out.append((*g.marginals(), g.duals(), g.cell_log()))
    ref = out[0]
    assert (out[1][3][:, 7] >= 0).any()   # cells with a slot
    for got in out[1:]:
        for k in range(2):
            assert np.abs(got[k] - ref[k]).sum() <= FP32_TOL * np.abs(ref[k]).sum()
        assert np.abs(got[2] - ref[2]).max() <= FP32_TOL * np.abs(ref[2]).max()


def test_fp32_regrouped_sweep_is_that_of_the_larger_cluster(env):
    """A sweep that regroups from clusters of two to four ends where one started on four does."""
    torch, dd = env
    N, s = 176, 8
    mu, nu = inputs.mixture_blobs(N=N, seed=12)
    eps = 16.0 / N ** 2
    out = []
    for first in (4, 2):
        with dd.DomDec(mu, nu, eps, 4 * eps, s, precision="fp32", err=-1.0, maxit=3, strategy="staggered",
                       spill_slots=1) as g:
            assert g.set_launch(first, 2.0) == first
            g.iterate(1)
            g.sync()
            assert (g.stats()["cluster_regroups"] >= 1) == (first == 2)
            out.append((*g.marginals(), g.duals()))
    for k in range(2):
        assert np.abs(out[1][k] - out[0][k]).sum() <= FP32_TOL * np.abs(out[0][k]).sum()
    assert np.abs(out[1][2] - out[0][2]).max() <= FP32_TOL * np.abs(out[0][2]).max()


@pytest.mark.parametrize("N,s", [(32, 4), (64, 8), (64, 16)])
@pytest.mark.parametrize("ctas", [2, 8])
def test_translation_step_stops_alike_on_clusters(env, N, s, ctas):
    """Double cells with the translation step that stop on a tolerance: the same iterations and
    marginals on clusters as on one CTA each (t*/eps amplifies a rounding by lam/eps = 100)."""
    torch, dd = env
    mu, nu = inputs.mixture_blobs(N=N, seed=22)
    eps = 4.0 / N ** 2
    out = []
    for c in (1, ctas):
        with dd.DomDec(mu, nu, eps, 100 * eps, s, precision="fp64", cell_ctas=c, cell_ti=1, err=1e-4, maxit=3000,
                       strategy="safe", spill_slots=100) as g:
            g.iterate(2)
            g.sync()
            out.append((g.cell_log(), *g.marginals()))
    one, got = out
    assert (got[0][:, 5] == 0).all() and np.array_equal(got[0][:, :5], one[0][:, :5])
    for k in (1, 2):
        assert np.abs(got[k] - one[k]).sum() <= 1e-9 * np.abs(one[k]).sum()


# --------------------------------------------------------------- capacity of a Y-box
@pytest.mark.parametrize("ctas", [0, 8])
def test_largest_boxes_without_spill_slots(env, ctas):
    """96 x 96 boxes of double cells at s = 16 fill the shared memory of eight CTAs to the last
    32 points: they run without a spill slot."""
    torch, dd = env
    N, s = 96, 16
    mu, nu = inputs.mixture_blobs(N=N, seed=23)
    eps = 16.0 / N ** 2
    out = []
    for slots in (16, -1):
        with dd.DomDec(mu, nu, eps, 1.0, s, precision="fp64", cell_ctas=ctas, err=-1.0, maxit=2, strategy="safe",
                       spill_slots=slots) as g:
            g.iterate(1)
            assert g.sync() == 0
            out.append(g.marginals())
    for k in range(2):
        assert np.abs(out[1][k] - out[0][k]).sum() <= 1e-11 * np.abs(out[0][k]).sum()
