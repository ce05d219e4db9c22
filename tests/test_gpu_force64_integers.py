"""FP64 forces of one species, whose pair terms are 64-bit integers with common
exponents per particle: 16 and 4 threads per particle, only far pairs, pairs
too close for the exponents (they take FP64), rows of several scans, sigma well
off the spacing, small units, a changed layout and changed parameters.

Against the pair sum in extended precision.  Both sides fold positions of size
L: a separation is off by at most delta = 8 2^-53 L, a pair force by 14 delta /
r, so max |dF| / S_i <= 16 delta / r_min with S_i = sum_j |F_ij|, plus 1e-15
for the arithmetic; energy and virial the same, of their sums of magnitudes."""
import numpy as np
import pytest
from scipy.spatial import cKDTree

from paper_2406_04210_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ljmd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_04210_gb300 import build, ljmd as m
    build.build()
    m.load()
    return m


def _exact(box, pos, eps, sigma, rcut):
    p = cKDTree(np.mod(pos, box), boxsize=box).query_pairs(rcut, output_type="ndarray")
    i, j = p[:, 0], p[:, 1]
    x, L = pos.astype(np.longdouble), box.astype(np.longdouble)
    d = x[i] - x[j]
    d -= L * np.rint(d / L)
    r2 = (d * d).sum(1)
    eps, sigma, rcut = (np.longdouble(v) for v in (eps, sigma, rcut))
    s6, c6 = (sigma * sigma / r2) ** 3, (sigma / rcut) ** 6
    g = 24 * eps * s6 * (2 * s6 - 1)
    e = 4 * eps * s6 * (s6 - 1) - 4 * eps * c6 * (c6 - 1)
    fd = (g / r2)[:, None] * d
    f, S = np.zeros(x.shape, np.longdouble), np.zeros(len(x), np.longdouble)
    mag = abs(g) / np.sqrt(r2)
    for a, s in ((i, 1), (j, -1)):
        np.add.at(f, a, s * fd)
        np.add.at(S, a, mag)
    return f, S, e.sum(), g.sum(), (4 * eps * s6 * (s6 + 1)).sum(), abs(g).sum(), np.sqrt(r2.min()) if len(p) else rcut


def _check(b, box, pos, eps=1.0, sigma=1.0, rcut=2.5):
    f, S, e, w, es, ws, rmin = _exact(box, pos, eps, sigma, rcut)
    tol = 16 * 8 * 2.0 ** -53 * box.max() / rmin + 1e-15
    g, eg, wg = b.force()
    assert not g[S == 0].any()
    err = float((np.sqrt(((g - f) ** 2).sum(1))[S > 0] / S[S > 0]).max()) if S.any() else 0.0
    print(f"n {len(pos)} r_min {float(rmin):.3g}: max |dF|/S {err:.2e} (tolerance {float(tol):.2e}) "
          f"dE {float(abs(eg[0] - e) / es) if es else 0:.1e} dW {float(abs(wg[0] - w) / ws) if ws else 0:.1e}")
    assert err <= tol
    assert abs(eg[0] - e) <= tol * es and abs(wg[0] - w) <= tol * ws


def _box(ljmd, s, pos=None, scale=1.0, eps=1.0, sigma=1.0, rcut=2.5, skin=0.3):
    pos = (s.pos if pos is None else pos) * scale
    b = ljmd.Box(pos, s.box * scale, precision="fp64")
    b.set_lj(eps, sigma, rcut, skin, True)
    return b, s.box * scale, pos


@pytest.mark.parametrize("n,rho", [(500, 0.8442), (4863, 0.8442), (4865, 0.8442), (9001, 0.6), (4000, 1.2), (2000, 0.1)])
def test_sizes_and_densities(ljmd, n, rho):
    s = inputs.fcc_subset_system(n, rho, 0.7, seed=n)
    _check(*_box(ljmd, s))


@pytest.mark.parametrize("n", [1500, 6000])
@pytest.mark.parametrize("sigma,rcut,r", [(1.0, 2.5, 0.3), (1.0, 2.5, 0.112), (0.25, 2.5, 0.109), (0.25, 4.3, 0.15),
                                          (2.0, 2.5, 0.9), (1.0, 1.1, 1.0)])
def test_close_pairs_and_long_rows(ljmd, n, sigma, rcut, r):
    s = inputs.fcc_subset_system(n, 0.8442, 0.7, seed=n)
    pos = s.pos.copy()
    pos[11] = np.mod(pos[5] + r * np.array([0.6, 0.0, -0.8]), s.box)   # a neighbour's place or not: one close pair
    _check(*_box(ljmd, s, pos, sigma=sigma, rcut=rcut), sigma=sigma, rcut=rcut)


@pytest.mark.parametrize("n", [2000, 6000])
def test_small_units(ljmd, n):
    s, a = inputs.fcc_subset_system(n, 0.8442, 0.7, seed=n), 3.4e-4
    kw = dict(eps=1.65e-21, sigma=a, rcut=2.5 * a)
    _check(*_box(ljmd, s, scale=a, skin=0.3 * a, **kw), **kw)


def test_layout_parameters_and_steps(ljmd):
    s = inputs.fcc_subset_system(8000, 0.8442, 0.7, seed=1)
    b, box, pos = _box(ljmd, s)
    b.set_layout(cell_scale=1.2)
    _check(b, box, pos)
    b.set_lj(1.3, 0.9, 2.5, 0.3, True)
    _check(b, box, pos, 1.3, 0.9)
    b.set_lj(1.0, 1.0, 2.9, 0.4, True)
    _check(b, box, pos, rcut=2.9)
    b.integrate(0.004, 25)
    _check(b, box, b.get_state()[0], rcut=2.9)
