"""One species in FP32 forces with other units of length: lengths times sigma and
times times sigma leave velocities and energies as they are and divide forces by
sigma, so the FP64 oracle's results at sigma = 1 are scaled.  Tolerances are those
of the same quantities at sigma = 1 (test_gpu_force_items.py, test_gpu_allpairs.py,
test_gpu_adjoint_items.py)."""
import functools

import numpy as np
import pytest

import oracle
from forcecheck import pair_scale
from paper_2406_04210_gb300 import inputs

pytestmark = pytest.mark.gpu
SIGMAS = [2.0 ** -9, 1.0, 340.0, 1000.0]


@pytest.fixture(scope="module")
def ljmd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_04210_gb300 import build, ljmd as m
    build.build()
    m.load()
    return m


@functools.lru_cache(None)
def _fluid(n):
    """A fluid at sigma = 1, the oracle's forces, energy and virial, and S_i."""
    s = inputs.fcc_subset_system(n, 0.8, 0.7, seed=n, rcut=2.2)
    lj = oracle.LJ(s.eps, s.sigma, s.rcut, True)
    return s, oracle.forces(s.box, s.pos, lj, None), pair_scale(s.box, s.pos, lj)


def _box(ljmd, ss, sigma, prec="mixed_ds"):
    b = ljmd.Box(np.concatenate([s.pos for s in ss]) * sigma, np.stack([s.box for s in ss]) * sigma,
                 np.concatenate([s.vel for s in ss]), n=[s.n for s in ss], precision=prec)
    return b.set_lj(1.0, sigma, 2.2 * sigma, 0.3 * sigma)


# small work items and chunks, one replica and several
@pytest.mark.parametrize("sizes", [(1025,), (65537,), (200, 1153, 128), (200,) * 600])
@pytest.mark.parametrize("sigma", SIGMAS)
def test_forces(ljmd, sizes, sigma):
    b = _box(ljmd, [_fluid(n)[0] for n in sizes], sigma)
    f, e, w = b.force()
    at = 0
    for r, n in enumerate(sizes):
        _, (fo, eo, wo), S = _fluid(n)
        assert np.max(np.linalg.norm(f[at:at + n] * sigma - fo, axis=1) / np.maximum(S, 1e-3)) <= 1e-5
        assert abs(e[r] - eo) <= 1e-5 * abs(eo) and abs(w[r] - wo) <= 1e-5 * 0.5 * 2.2 * S.sum()
        at += n


# the force-only instances
@pytest.mark.parametrize("n", [1025, 65537])
@pytest.mark.parametrize("sigma", SIGMAS)
def test_steps_without_energies(ljmd, n, sigma):
    s = _fluid(n)[0]
    out = []
    for prec, unit in (("fp64", 1.0), ("mixed_ds", sigma)):
        b = _box(ljmd, [s], unit, prec)
        b.integrate(0.005 * unit, 10, thermo=False)
        x, v = b.get_state()[:2]
        out.append((x / unit, v))
    d = out[1][0] - out[0][0]
    assert np.max(np.abs(d - s.box * np.rint(d / s.box))) <= 1e-4


@pytest.mark.parametrize("sigma", SIGMAS)
def test_all_pairs(ljmd, sigma):
    s, _, _ = _fluid(1025)
    d = s.pos[:, None, :] - s.pos[None, :, :]
    d -= s.box * np.rint(d / s.box)
    r2 = np.einsum("ijk,ijk->ij", d, d)
    np.fill_diagonal(r2, np.inf)
    s6 = r2 ** -3
    f = 48 / r2 * s6 * (s6 - 0.5)
    fo, S = np.einsum("ij,ijk->ik", f, d), (np.abs(f) * np.sqrt(np.where(np.isinf(r2), 0, r2))).sum(1)
    b = ljmd.Box(s.pos * sigma, s.box * sigma)
    g, e, w = b.set_lj(1.0, sigma, np.inf, 0.3 * sigma).force()
    assert np.max(np.linalg.norm(g * sigma - fo, axis=1) / S) <= 1e-5
    eo = 2 * (s6 * (s6 - 1)).sum()
    assert abs(e[0] - eo) <= 1e-5 * abs(eo) and abs(w[0] - 24 * (s6 * (s6 - 0.5)).sum()) <= 1e-5 * S.sum() * s.box[0]


# (65,700 particles: chunks.  Beyond sigma ~ 940 the tables of several species overflow too.)
@pytest.mark.parametrize("n,nsteps,ckpt", [(1111, 6, 3), (65700, 3, 3)])
def test_gradient(ljmd, n, nsteps, ckpt):
    s = inputs.fcc_subset_system(n, 0.8, 0.7, seed=n, rcut=2.2)
    rng = np.random.default_rng(n)
    lx, lv = rng.normal(size=s.pos.shape), rng.normal(size=s.pos.shape)
    lj = oracle.LJ(s.eps, s.sigma, s.rcut)
    traj = oracle.run(s.box, s.pos, s.vel, lj, s.skin, s.dt, nsteps, traj=True)["traj"]
    want = oracle.adjoint(s.box, traj, lj, s.dt, lx, lv)
    for sigma in SIGMAS[:3] + [600.0]:
        b = _box(ljmd, [s], sigma)
        b.integrate(s.dt * sigma, nsteps, thermo=False, ckpt_every=ckpt)
        got = b.adjoint(lx / sigma, lv)
        for g, w, unit in zip(got, want, (sigma, 1.0, 1.0, sigma)):
            g, w = np.asarray(g) * unit, np.asarray(w)
            assert np.linalg.norm(g - w) / np.linalg.norm(w) <= 2e-4
