"""The adjoint's work split and its tape, against the FP64 oracle's adjoint with
test_gpu_adjoint.py's tolerance (2e-4 relative): boxes on either side of the
small-work-item rule (512 chunks), replicas of uneven size, lists rebuilt inside
a segment (the tape keeps them once per build), and graphs kept between calls."""
import numpy as np
import pytest

import oracle
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


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _expected(s, dt, nsteps, lx, lv):
    lj = oracle.LJ(s.eps, s.sigma, s.rcut)
    r = oracle.run(s.box, s.pos, s.vel, lj, s.skin, dt, nsteps, traj=True)
    return oracle.adjoint(s.box, r["traj"], lj, dt, lx, lv)


def _check(got, want):
    for g, w in zip(got, want):
        assert rel(np.asarray(g), np.asarray(w)) <= 2e-4


@pytest.mark.parametrize("n,nsteps,ckpt", [(1111, 6, 3), (65536, 3, 3), (65700, 3, 3)])
def test_sizes(ljmd, n, nsteps, ckpt):
    s = inputs.fcc_subset_system(n, 0.8, 0.7, seed=n)
    rng = np.random.default_rng(n)
    lx, lv = rng.normal(size=s.pos.shape), rng.normal(size=s.pos.shape)
    b = ljmd.from_system(s)
    b.integrate(s.dt, nsteps, thermo=False, ckpt_every=ckpt)
    _check(b.adjoint(lx, lv), _expected(s, s.dt, nsteps, lx, lv))


def test_replicas(ljmd):
    ss = [inputs.fcc_subset_system(n, 0.8, 0.7, seed=n) for n in (200, 1153, 640)]
    b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]),
                 np.concatenate([s.vel for s in ss]), n=[s.n for s in ss])
    b.set_lj()
    rng = np.random.default_rng(0)
    lx, lv = rng.normal(size=(b.n_total, 3)), rng.normal(size=(b.n_total, 3))
    b.integrate(0.005, 8, thermo=False, ckpt_every=4)
    gx, gv, ge, gs = b.adjoint(lx, lv)
    at, we, ws = 0, 0.0, 0.0
    for s in ss:
        k = slice(at, at + s.n)
        x, v, e, g = _expected(s, 0.005, 8, lx[k], lv[k])
        assert rel(gx[k], x) <= 2e-4 and rel(gv[k], v) <= 2e-4
        we, ws, at = we + e, ws + g, at + s.n
    assert rel(ge, we) <= 2e-4 and rel(gs, ws) <= 2e-4


def test_lists_rebuilt_inside_a_segment(ljmd):
    s = inputs.fcc_subset_system(1500, 0.8, 8.0, seed=4)
    rng = np.random.default_rng(4)
    lx, lv = rng.normal(size=s.pos.shape), rng.normal(size=s.pos.shape)
    b = ljmd.from_system(s)
    r0 = b.info().rebuilds
    b.integrate(0.002, 40, thermo=False, ckpt_every=40)
    assert b.info().rebuilds - r0 >= 3            # the checkpoint's and two on the way
    _check(b.adjoint(lx, lv), _expected(s, 0.002, 40, lx, lv))


def test_graphs_are_kept_between_calls_and_follow_changes(ljmd):
    s = inputs.fcc_subset_system(900, 0.8, 0.7, seed=6)
    rng = np.random.default_rng(6)
    lx, lv = rng.normal(size=s.pos.shape), rng.normal(size=s.pos.shape)
    b = ljmd.from_system(s)
    first = None
    for eps, dt, nsteps, ckpt in [(1.0, 0.004, 8, 4), (1.0, 0.004, 8, 4), (1.0, 0.002, 8, 4), (1.0, 0.002, 8, 8),
                                  (1.3, 0.002, 8, 8), (1.0, 0.004, 8, 4)]:
        b.set_lj(eps)
        b.set_state(s.pos, s.vel)
        b.integrate(dt, nsteps, thermo=False, ckpt_every=ckpt)
        got = b.adjoint(lx, lv)
        s.eps = np.full((1, 1), eps)
        _check(got, _expected(s, dt, nsteps, lx, lv))
        if (eps, dt, ckpt) == (1.0, 0.004, 4):
            first = first or got
            for x, y in zip(first, got):
                np.testing.assert_array_equal(x, y)
