"""The smoothed pair-distance histogram and its gradient at the edges of the
kernels' work split: bins per lane (1, 31, 33, 64, 129, 256 bins), particles
not filling a chunk, replicas of uneven size.  Against NumPy brute force; the
tolerance is the effect of the FP32 distances (|dr| <= 6e-7 from the rounding
of the FP32 offsets and their differences) plus 4e-6 of the summed terms (FP32
exponentials and sums)."""
import numpy as np
import pytest

from paper_2406_04210_gb300 import inputs

pytestmark = pytest.mark.gpu

DR, REL = 6e-7, 4e-6


@pytest.fixture(scope="module")
def ljmd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_04210_gb300 import build, ljmd as m
    build.build()
    m.load()
    return m


def _expected(s, nbins, rhist, width, rmax, coef):
    """(h, its tolerance, gradient, its tolerance)."""
    d = s.pos[:, None, :] - s.pos[None, :, :]
    d -= s.box * np.rint(d / s.box)
    r = np.sqrt(np.einsum("ijk,ijk->ij", d, d))
    np.fill_diagonal(r, np.inf)
    i, j = np.nonzero(r < rmax)
    d, r = d[i, j], r[i, j]
    x = (r[:, None] - (np.arange(nbins) + 0.5) * rhist / nbins) / width
    g = np.exp(-0.5 * x * x) / s.n
    h, tol = 0.5 * g.sum(0), 0.5 * ((np.abs(x) / width * DR + REL) * g).sum(0) + 1e-12
    D = -(x / width * g) @ coef                              # d/dr of sum_k coef_k g_k
    DD = ((x * x + 1) / width ** 2 * g) @ np.abs(coef) * DR + (np.abs(x) / width * g) @ np.abs(coef) * (REL + 2 * DR)
    grad, gtol = np.zeros((s.n, 3)), np.full(s.n, 1e-12)
    np.add.at(grad, i, (D / r)[:, None] * d)
    np.add.at(gtol, i, DD)
    return h, tol, grad, gtol


@pytest.mark.parametrize("nbins", [1, 31, 33, 64, 129, 256])
def test_histogram_and_gradient(ljmd, nbins):
    s = inputs.fcc_subset_system(997, 0.8, 0.7, seed=nbins)   # 7 chunks of 128 and one of 101
    rhist, rmax = 2.5, 2.7
    width = rhist / max(nbins, 8)
    coef = np.random.default_rng(nbins).normal(size=nbins)
    h, tol, grad, gtol = _expected(s, nbins, rhist, width, rmax, coef)
    b = ljmd.from_system(s)
    got, g = b.pair_hist(nbins, rhist, width, rmax, coef=coef)
    assert np.all(np.abs(got[0] - h) <= tol)
    assert np.all(np.linalg.norm(g - grad, axis=1) <= gtol)


def test_histogram_of_uneven_replicas(ljmd):
    ss = [inputs.fcc_subset_system(n, 0.8, 0.7, seed=n) for n in (200, 1153, 128, 513)]
    b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]), n=[s.n for s in ss])
    b.set_lj(1.0, 1.0, 2.2, 0.3)
    coef = np.random.default_rng(1).normal(size=(4, 40))
    got, g = b.pair_hist(40, 2.5, 0.06, 2.4, coef=coef)
    at = 0
    for r, s in enumerate(ss):
        h, tol, grad, gtol = _expected(s, 40, 2.5, 0.06, 2.4, coef[r])
        assert np.all(np.abs(got[r] - h) <= tol)
        assert np.all(np.linalg.norm(g[at:at + s.n] - grad, axis=1) <= gtol)
        at += s.n
