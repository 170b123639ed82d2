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
    small cells: every cell ends within the tolerance, two runs are equal to the last
    bit, and the result is that of one CTA per cell."""
    torch, dd = env
    mu, nu = inputs.mixture_blobs(N=N, seed=21)
    eps, err = 4.0 / N ** 2, 1e-4
    lam = 100.0 * eps   # the slowest mode of a cell contracts by 1/(1 + eps/lam): some hundred iterations
    out = []
    for c in (1, ctas, ctas):
        with dd.DomDec(mu, nu, eps, lam, s, precision=precision, cell_ctas=c, err=err, maxit=3000, strategy="safe",
                       spill_slots=100) as g:
            g.iterate(2)
            g.sync()
            log = g.cell_log()
            PX, PY = g.marginals()
            out.append((log, PX, PY, g.duals()))
    one, got, again = out
    assert (got[0][:, 5] == 0).all() and (one[0][:, 5] == 0).all()
    assert np.array_equal(got[0][:, :8], again[0][:, :8])
    for k in (1, 2, 3):
        assert np.array_equal(got[k], again[k])
    m = np.pad(mu, s)   # the second sweep's cells are offset by s
    cell = m.reshape(m.shape[0] // (2 * s), 2 * s, -1, 2 * s).sum((1, 3)).max()
    assert (got[0][:, 6] <= err * cell * (1 + 1e-6)).all()
    if precision == "fp64":   # sums in another order (1e-16) through hundreds of contracting iterations
        assert np.array_equal(got[0][:, :5], one[0][:, :5])
        for k in (1, 2):
            assert np.abs(got[k] - one[k]).sum() <= 1e-9 * np.abs(one[k]).sum()
    else:   # each side's P_X is within sqrt(2 gap |mu|) of its cells' limit (Pinsker), in both sweeps
        assert np.abs(got[1] - one[1]).sum() <= 4.0 * np.sqrt(2.0 * err) * mu.sum()
