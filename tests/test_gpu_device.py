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
