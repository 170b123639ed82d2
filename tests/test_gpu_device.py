"""The library's own device functions (double 2^x, logarithm, reciprocal,
conversions, the Newton root and the log-sum-exp of the double cells, the
cells' block sums), compiled into a library of the tests and compared with
64-bit and longer arithmetic on the host."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def env(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_08859_gb300 import build as b
    so = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    subprocess.run([b.nvcc(), *b.ARCH, "-O3", "-std=c++17", "--expt-extended-lambda", "-Xcompiler", "-fPIC", "-shared",
                    "-I", os.path.join(b.ROOT, "include"), "-I", b.CSRC, os.path.join(HERE, "device_probe.cu"),
                    "-o", so, "-lcudart"], check=True, capture_output=True)
    return torch, ctypes.CDLL(so)


def dev(torch, x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def unary(env, kind, x):
    torch, lib = env
    a = dev(torch, x)
    y = torch.empty_like(a)
    assert lib.probe_unary(kind, ptr(a), ptr(y), a.numel()) == 0
    return y.cpu().numpy()


# ------------------------------------------------------------------ block sums
@pytest.mark.parametrize("K", [2, 4, 12])
def test_block_sums_keep_every_bit_of_a_double(env, K):
    """A single value among zeros comes back whole (also below the range of floats), every value
    from its own sum; sums of 512 terms err by at most nine roundings (a tree of 5 + 4 additions)."""
    torch, lib = env
    rng = np.random.default_rng(K)

    def sums(x):
        a, out = dev(torch, x), torch.empty(K, dtype=torch.float64, device="cuda")
        assert lib.probe_sums(K, ptr(a), ptr(out)) == 0
        return out.cpu().numpy()

    for t in (0, 1, 31, 32, 77, 255, 496, 511):
        x = np.zeros((K, 512))
        one = rng.uniform(1, 2, K) * 10.0 ** rng.integers(-60, 60, K) * rng.choice([-1, 1], K)
        x[:, t] = one
        assert np.array_equal(sums(x), one)
    for _ in range(5):
        x = rng.normal(size=(K, 512)) * 10.0 ** rng.uniform(-3, 3, (K, 512))
        ref = np.array([math.fsum(r) for r in x])
        assert (np.abs(sums(x) - ref) <= 9 * 2.0 ** -53 * np.abs(x).sum(1)).all()
    x = np.ones((K, 512))
    x[0, 3], x[1, 5] = np.inf, np.nan
    got = sums(x)
    assert got[0] == np.inf and np.isnan(got[1]) and (got[2:] == 512).all()


# ------------------------------------------------------- 2^x, reciprocal, conversions
def test_exp2(env):
    """Roundings of the table entry and of the result, the polynomial's remainder (2^-54) and the
    roundings of its small value (below 0.0055 of the result): 2.6 x 2^-53."""
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(-1021.9, 1021.9, 100000), rng.uniform(-70, 70, 100000), rng.uniform(-1, 1, 50000),
                        np.arange(-512, 513) / 64.0, (np.arange(-512, 513) + 0.5) / 64.0 * (1 + 1e-15), [0.0, -0.0]])
    y = unary(env, 0, x)
    ref = np.exp2(x.astype(np.longdouble))
    assert float((np.abs(y - ref) / ref).max()) <= 2.6 * 2.0 ** -53
    x = np.array([1023.5, 1024.0, 2000.0, np.inf, -1022.5, -1074.0, -1080.0, -2000.0, -np.inf, np.nan])
    with np.errstate(over="ignore", under="ignore"):
        y, ref = unary(env, 0, x), np.exp2(x)
    assert np.isnan(y[-1]) and (y[[1, 2, 3]] == np.inf).all() and (y[[6, 7, 8]] == 0.0).all()
    assert np.allclose(y[[0, 4, 5]], ref[[0, 4, 5]], rtol=4e-16, atol=5e-324)


def test_reciprocal(env):
    """Correctly rounded but for halfway cases within 2^-40: 0.51 ulp, i.e. 1.02 x 2^-53 relative."""
    rng = np.random.default_rng(2)
    x = np.concatenate([rng.uniform(1, 2, 100000), 2.0 ** rng.uniform(-1022, 1022, 100000), 2.0 ** np.arange(-1021, 1022),
                        np.array([2.0 ** -121, 2.0 ** 121, 2.0 ** -120, 2.0 ** 120]) * 1.999])
    x = np.concatenate([x, -x])
    y = unary(env, 2, x)
    ref = 1 / x.astype(np.longdouble)
    assert float((np.abs(y - ref) / np.abs(ref)).max()) <= 1.02 * 2.0 ** -53
    y = unary(env, 2, np.array([0.0, -0.0, np.inf, -np.inf, np.nan]))
    assert y[0] == np.inf and y[1] == -np.inf and y[2] == 0.0 and y[3] == 0.0 and np.isnan(y[4])


def test_conversions(env):
    """Rounded to nearest even where the result is a normal float; the general one for every input."""
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.normal(size=100000), 2.0 ** rng.uniform(-125.9, 127.9, 100000),
                        (1 + np.arange(4096) / 4096.0) * (1 + 2.0 ** -24),   # halfway between two floats
                        [2.0 ** -126, 1.0, np.nextafter(2.0, 1)]])
    x = np.concatenate([x, -x])
    ref = x.astype(np.float32).astype(np.float64)
    assert np.array_equal(unary(env, 3, x), ref)
    assert np.array_equal(unary(env, 4, x), ref)
    assert np.array_equal(unary(env, 3, np.array([0.0, 1e-60, -1e-300])), np.zeros(3))
    odd = np.array([0.0, 1e-60, -1e-300, 1e-40, 2.0 ** 128, -1e300, 3.4028235677973366e38, np.inf, -np.inf, np.nan])
    with np.errstate(over="ignore", under="ignore"):
        ref = odd.astype(np.float32).astype(np.float64)
    y = unary(env, 4, odd)
    y[np.abs(y) < 2.0 ** -126] = ref[np.abs(ref) < 2.0 ** -126] if (np.abs(y) < 2.0 ** -126).sum() == 4 else np.nan
    assert np.array_equal(y, ref, equal_nan=True)
    w = np.concatenate([np.float32(rng.uniform(1e-30, 1e30, 10000)).astype(np.float64), np.arange(1.0, 2000.0) ** 2])
    assert np.array_equal(unary(env, 5, w), w)
    # squares of distances: 0 stands as 2^-127, far below a rounding of any exponent
    assert unary(env, 5, np.zeros(1))[0] == 2.0 ** -127


# ------------------------------------------- logarithm of a quotient (the line search)
def test_log_of_a_quotient(env):
    """Half a unit in the last place of the result and two roundings of a table value (6e-17); next to
    a = b, where there is no table value, three units and the correction's 2^-44 x 2^-23."""
    torch, lib = env
    rng = np.random.default_rng(4)
    n = 100000

    def run(kind, a, b):
        y = torch.empty(a.size, dtype=torch.float64, device="cuda")
        assert lib.probe_binary(kind, ptr(dev(torch, a)), ptr(dev(torch, b)), ptr(y), a.size) == 0
        return y.cpu().numpy()

    for ratio in (1 + rng.choice([-1, 1], n) * 10 ** rng.uniform(-12, -1, n), rng.uniform(0.5, 2, n),
                  10 ** rng.uniform(-6, 6, n), 10 ** rng.uniform(-25, 20, n)):
        b = 10 ** rng.uniform(-9, -3, n)
        a = b * ratio
        A, B = a.astype(np.longdouble), b.astype(np.longdouble)
        ref = np.where(np.abs(ratio - 1) < 0.5, np.log1p((A - B) / B), np.log(A / B))
        size = np.abs(ref).astype(np.float64)
        tol = np.where(size > 1 / 257, 0.55 * np.spacing(size) + 6e-17, 3 * np.spacing(size) + 2e-20)
        assert float((np.abs(run(0, a, b) - ref) / tol).max()) <= 1.0
        d = (a - b) ** 2
        q = d.astype(np.longdouble) / A
        assert (np.abs(run(1, d, a) - q) <= 0.5001 * np.spacing(q.astype(np.float64))).all()
    # outside the fast path's range: as CUDA's
    a = np.array([1e-300, 1e-300, 1e300, 1e-40, 3.0, np.inf, np.nan])
    b = np.array([1e-5, 1e-200, 1e-5, 1e-310, 1e-310, 1e-3, 1.0])
    with np.errstate(over="ignore"):
        ref = np.log(a / b)
    got = run(0, a, b)
    assert np.allclose(got, ref, rtol=4e-16, atol=0, equal_nan=True)
    assert np.array_equal(run(1, np.array([0.0, 1e-320, 1e300]), np.array([2.0, 1e-5, 1e-60])), [0.0, 1e-320 / 1e-5, np.inf])


# --------------------------------------------------------- the root of a double cell
@pytest.mark.parametrize("s", [1e-6, 1e-3, 0.3, 20.0])
@pytest.mark.parametrize("scale", [1.0, 30.0, 1e4, 1e8])
def test_newton_root(env, s, scale):
    """g(u) = (1 + s) u + c0 + log(1 + e^(lr - u)) = 0 from good, bad and no previous roots: the error
    is a rounding of g's terms over g', plus the last step's cube (1e-15) and a rounding of u."""
    torch, lib = env
    rng = np.random.default_rng(int(1 / s) + int(scale))
    n = 4000
    lr = scale * rng.normal(size=n)
    lr[::7] = -np.inf
    c0 = scale * rng.normal(size=n)
    lo, hi = np.full(n, -1.0, np.longdouble), np.full(n, 1.0, np.longdouble)
    L, c = lr.astype(np.longdouble), c0.astype(np.longdouble)

    def g(u):
        t = L - u
        return (1 + np.longdouble(s)) * u + c + np.maximum(t, 0) + np.log1p(np.exp(-np.abs(t)))

    with np.errstate(over="ignore", under="ignore"):
        while (g(lo) > 0).any():
            lo = np.where(g(lo) > 0, lo * 4, lo)
        while (g(hi) < 0).any():
            hi = np.where(g(hi) < 0, hi * 4, hi)
        for _ in range(140):
            mid = (lo + hi) / 2
            up = g(mid) > 0
            hi, lo = np.where(up, mid, hi), np.where(up, lo, mid)
        ref = (lo + hi) / 2
        sig = 1 / (1 + np.exp(-np.where(np.isfinite(L), L - ref, -np.inf)))
    slope = (1 + s) - sig
    size = np.abs(c) + (1 + s) * np.abs(ref) + np.maximum(np.where(np.isfinite(L), L - ref, 0), 0) + 1
    tol = (8 * 2.0 ** -53 * size / slope + 1e-15 + 2.0 ** -52 * np.abs(ref)).astype(np.float64)
    r = ref.astype(np.float64)
    for uw in (np.full(n, np.inf), r, r + rng.normal(size=n), r + scale * rng.normal(size=n), r * (1 + 1e-9)):
        u = torch.empty(n, dtype=torch.float64, device="cuda")
        assert lib.probe_newton(ptr(dev(torch, lr)), ptr(dev(torch, c0)), ptr(dev(torch, uw)), ctypes.c_double(s), 30,
                                ptr(u), n) == 0
        e = np.abs(u.cpu().numpy() - r) / tol
        assert e.max() <= 1.0, (e.max(), int(e.argmax()))


# ------------------------------------------------ the log-sum-exp of the double cells
def lse_ref(f, q2, n):
    d = np.arange(n)[:, None] - np.arange(f.size)[None, :]
    with np.errstate(invalid="ignore", under="ignore", divide="ignore"):
        v = f.astype(np.longdouble)[None, :] - np.longdouble(q2) * d ** 2
        mx = np.where(np.isnan(f).any(), np.longdouble(np.nan), v.max(1))
        sh = np.where(np.isfinite(mx), mx, 0)
        return (sh + np.log2(np.exp2(v - sh[:, None]).sum(1))).astype(np.float64), mx.astype(np.float64)


def lse_dev(env, f, q2, n, P, prev=None):
    torch, lib = env
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    p = dev(torch, np.zeros(n) if prev is None else prev)
    assert lib.probe_lse(ptr(dev(torch, f)), f.size, ctypes.c_double(q2), ptr(p), int(prev is not None), P, ptr(out), n) == 0
    return out.cpu().numpy()


def test_lse_of_double_cells_with_special_sources(env):
    """-inf sources weigh nothing, a line of them gives -inf, a NaN source gives NaN everywhere."""
    rng = np.random.default_rng(5)
    for base in (0.0, -500.0, 500.0):
        f = base + rng.normal(size=32)
        f[[3, 4, 20]] = -np.inf
        ref, _ = lse_ref(f, 1.0, 32)
        for prev in (None, ref, ref + 50.0):
            assert (np.abs(lse_dev(env, f, 1.0, 32, 4, prev) - ref) <= 4 * 2.0 ** -53 * (np.abs(ref) + 70)).all()
        f[:] = -np.inf
        assert (lse_dev(env, f, 1.0, 32, 4) == -np.inf).all()
        f = base + rng.normal(size=32)
        f[9] = np.nan
        for prev in (None, np.full(32, base), np.full(32, np.nan)):
            assert np.isnan(lse_dev(env, f, 1.0, 32, 4, prev)).all()


@pytest.mark.parametrize("M", [1, 7, 32, 200])
@pytest.mark.parametrize("P", [1, 4, 32])
@pytest.mark.parametrize("q2", [1e-3, 1.0, 1e4, 1e8, 1e11])
def test_lse_of_double_cells(env, M, P, q2):
    """Sources from moderate to far larger than a float resolves (eps down to 1e-11 h^2), without a
    previous value, with the value itself, with one that is off by up to 40, and with a useless one.
    Each exponent carries two roundings of the magnitudes it is formed from."""
    rng = np.random.default_rng(M + P)
    n = 45
    for scale in (1.0, 100.0, 5.0 * q2):
        f = scale * rng.normal(size=M)
        ref, _ = lse_ref(f, q2, n)
        tol = 4 * 2.0 ** -53 * (np.abs(f).max() + np.abs(ref) + 70) + 1e-15
        for prev in (None, ref, ref + rng.uniform(-40, 40, n), ref + 1e4, np.full(n, -np.inf), np.full(n, np.nan)):
            got = lse_dev(env, f, q2, n, P, prev)
            assert (np.abs(got - ref) <= tol).all(), (scale, np.abs(got - ref).max())


# ------------------------------------------------------- cluster size of double cells
@pytest.mark.parametrize("N", [12, 20, 28, 32, 40, 48])
@pytest.mark.parametrize("strategy", ["staggered", "safe"])
def test_clusters_of_eight_for_few_double_cells(env, N, strategy):
    """Clusters of eight while the largest sub-batch has at most one cell per eight SMs."""
    torch, _ = env
    from paper_2410_08859_gb300 import domdec as dd
    from paper_2410_08859_gb300 import inputs
    s, nc = 2, N // 4 + 1
    cells = ((nc + 1) // 2) ** 2 if strategy == "staggered" else nc ** 2
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mu, nu = inputs.mixture_small(N=N, seed=5)
    with dd.DomDec(mu, nu, 1.0 / N ** 2, 1.0, s, precision="fp64", strategy=strategy) as g:
        got = g.set_launch(8, 2.0)
    # a layout that a box of few rows cannot use falls back to smaller clusters
    assert got == (8 if 8 * cells <= sms else 1) or (got == 1 and N < 16)
