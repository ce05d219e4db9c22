"""The two sizes of the FP32 list force's work items: 16 particles (boxes of up
to 512 chunks of 128) and chunks (larger boxes).  Both against the FP64 oracle
at ragged sizes, for one species, replicas and two species, with the tolerance
of test_gpu_md.py: max |dF| / S_i <= 1e-5, energies relative 1e-5; and a
trajectory on either side of the rule, with and without energies, against FP64."""
import numpy as np
import pytest

import oracle
from forcecheck import pair_scale
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


def _check(f, e, w, s):
    lj = oracle.LJ(s.eps, s.sigma, s.rcut, True)
    t = s.type if s.ntypes > 1 else None
    fo, eo, wo = oracle.forces(s.box, s.pos, lj, t)
    S = np.maximum(pair_scale(s.box, s.pos, lj, t), 1e-3)
    assert np.max(np.linalg.norm(f - fo, axis=1) / S) <= 1e-5
    assert abs(e - eo) <= 1e-5 * abs(eo) and abs(w - wo) <= 1e-5 * 0.5 * s.rcut.max() * S.sum()


@pytest.mark.parametrize("n", [200, 1025, 2943, 65537])
@pytest.mark.parametrize("prec", ["mixed_ds", "mixed_fp64"])
def test_one_species(ljmd, n, prec):
    s = inputs.fcc_subset_system(n, 0.8, 0.7, seed=n)
    f, e, w = ljmd.from_system(s, prec).force()
    _check(f, e[0], w[0], s)


@pytest.mark.parametrize("n", [1501, 65601])
def test_two_species(ljmd, n):
    s = inputs.fcc_subset_system(n, 1.1, 0.7, seed=9)
    s.eps, s.sigma, s.rcut = inputs.binary_params()
    s.type = (np.random.default_rng(1).random(n) < 0.2).astype(np.int32)
    f, e, w = ljmd.from_system(s).force()
    _check(f, e[0], w[0], s)


@pytest.mark.parametrize("sizes", [(200, 1153, 128, 513), (200,) * 259])
def test_replicas(ljmd, sizes):
    ss = [inputs.fcc_subset_system(n, 0.8, 0.7, seed=i, rcut=2.2) for i, n in enumerate(sizes)]
    b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]), n=list(sizes))
    b.set_lj(1.0, 1.0, 2.2, 0.3)
    f, e, w = b.force()
    at = 0
    for r, s in enumerate(ss):
        if r < 8 or r == len(ss) - 1:
            _check(f[at:at + s.n], e[r], w[r], s)
        at += s.n


@pytest.mark.parametrize("n", [65536, 65537])
def test_either_side_of_the_rule_follows_fp64(ljmd, n):
    s = inputs.fcc_subset_system(n, 0.8, 1.0, seed=3)
    ref = ljmd.from_system(s, "fp64")
    tr = ref.integrate(s.dt, 10)
    xr = ref.get_state()[0]
    for thermo in (True, False):
        b = ljmd.from_system(s)
        th = b.integrate(s.dt, 10, thermo=thermo)
        d = b.get_state()[0] - xr
        assert np.max(np.abs(d - s.box * np.rint(d / s.box))) <= 1e-4
        if thermo:
            np.testing.assert_allclose(th[:, 0, 0], tr[:, 0, 0], rtol=1e-5)
            np.testing.assert_allclose(th[:, 0, 1], tr[:, 0, 1], rtol=1e-5)
