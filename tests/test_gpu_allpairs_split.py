"""The FP32 all-pairs kernel at the edges of its split (groups of 32 particles,
staged tiles of 2,048, work items of 16 and whole chunks), against the FP64
oracle with test_gpu_allpairs.py's FP32 tolerance (max |dF| / S_i <= 1e-5); and
the thermostat's collisions drawn ahead of a graph's steps against those drawn
step by step."""
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


def _forces(s, i):
    """Forces on particles i, S_i, by NumPy."""
    d = s.pos[i][:, None, :] - s.pos[None, :, :]
    d -= s.box * np.rint(d / s.box)
    r2 = np.einsum("ijk,ijk->ij", d, d)
    r2[np.arange(len(i)), i] = np.inf
    e, g = s.eps[s.type[i]][:, s.type], s.sigma[s.type[i]][:, s.type]
    s6 = (g * g / r2) ** 3
    f = 48 * e / r2 * s6 * (s6 - 0.5)
    return np.einsum("ij,ijk->ik", f, d), (np.abs(f) * np.sqrt(np.where(np.isinf(r2), 0, r2))).sum(1)


def _box(ljmd, s):
    b = ljmd.Box(s.pos, s.box, s.vel, s.type)
    return b.set_lj(s.eps, s.sigma, np.full(s.eps.shape, np.inf), 0.3)


@pytest.mark.parametrize("n", [2, 33, 64, 127, 2047, 2049, 4130])
@pytest.mark.parametrize("species", [1, 2])
def test_forces(ljmd, n, species):
    s = inputs.fcc_subset_system(n, 0.7, 0.7, seed=n)
    if species == 2:
        s.eps, s.sigma, _ = inputs.binary_params()
        s.type = (np.arange(n) % 5 == 4).astype(np.int32)
    f, e, w = _box(ljmd, s).force()
    fo, S = _forces(s, np.arange(n))
    assert np.max(np.linalg.norm(f - fo, axis=1) / np.maximum(S, 1e-3)) <= 1e-5
    lj = oracle.LJ(s.eps, s.sigma, np.full(s.eps.shape, np.inf), True)
    _, eo, wo = oracle.forces_brute(s.box, s.pos, lj, s.type if species == 2 else None)
    assert abs(e[0] - eo) <= 1e-5 * abs(eo) + 1e-7 and abs(w[0] - wo) <= 1e-5 * S.sum() * s.box[0]


def test_replicas(ljmd):
    ss = [inputs.fcc_subset_system(n, 0.7, 0.7, seed=n) for n in (150, 31, 1100)]
    b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]), n=[s.n for s in ss])
    f = b.set_lj(1.0, 1.0, np.inf, 0.3).force()[0]
    at = 0
    for s in ss:
        fo, S = _forces(s, np.arange(s.n))
        assert np.max(np.linalg.norm(f[at:at + s.n] - fo, axis=1) / np.maximum(S, 1e-3)) <= 1e-5
        at += s.n


def test_whole_chunks(ljmd):
    s = inputs.fcc_subset_system(131201, 0.7, 0.7, seed=1)   # 1,026 chunks
    i = np.concatenate([np.arange(0, s.n, 2000), [s.n - 1]])
    fo, S = _forces(s, i)
    f = _box(ljmd, s).force()[0][i]
    assert np.max(np.linalg.norm(f - fo, axis=1) / S) <= 1e-5


@pytest.mark.parametrize("rate", [1.0, 150.0])
def test_collisions_drawn_ahead_equal_those_drawn_step_by_step(ljmd, rate):
    s = inputs.fcc_subset_system(30000, 0.8, 0.7, seed=2)   # 100 steps: beyond 64 MiB of draws
    out = []
    for calls, steps in ((1, 100), (10, 10)):
        b = ljmd.from_system(s).set_thermostat(1.3, rate, seed=5)
        for _ in range(calls):
            b.integrate(0.002, steps, thermo=False)
        out.append(b.get_state())
    np.testing.assert_allclose(out[1][1], out[0][1], rtol=0, atol=1e-9)


@pytest.mark.parametrize("calls", [(150,), (10, 150), (10, 140)])
def test_a_short_last_graph_draws_ahead_where_the_others_do_not(ljmd, calls):
    # 30,000 particles: 100 steps' draws exceed 64 MiB, those of the last 40 or 50 fit
    s = inputs.fcc_subset_system(30000, 0.8, 0.7, seed=3)
    out = []
    for steps in (calls, (10,) * (sum(calls) // 10)):
        b = ljmd.from_system(s).set_thermostat(1.3, 20.0, seed=6)
        for n in steps:
            b.integrate(0.002, n, thermo=False)
        out.append(b.get_state())
    np.testing.assert_allclose(out[1][1], out[0][1], rtol=0, atol=1e-9)
