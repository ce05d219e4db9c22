"""Two species choose their pair constants by selects, three and more read
tables: a mixture and the same mixture whose second species is split in two
equal ones give the same forces and energies bit for bit, in small work items
and in chunks, and the FP64 oracle's forces within 1e-5 of S_i = sum |F_ij| (the
FP32 tolerance of the force tests)."""
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


@pytest.mark.parametrize("n", [1000, 65600])
def test_selects_and_tables_agree(ljmd, n):
    s = inputs.binary_random_system(n, seed=n)
    three = s.type + ((s.type == 1) & (np.arange(n) % 3 == 0)).astype(np.int32)
    k = [0, 1, 1]
    two = ljmd.from_system(s)
    tab = ljmd.Box(s.pos, s.box, s.vel, three)
    tab.set_lj(s.eps[np.ix_(k, k)], s.sigma[np.ix_(k, k)], s.rcut[np.ix_(k, k)], s.skin, True)
    for x, y in zip(two.force(), tab.force()):
        np.testing.assert_array_equal(x, y)
    for x, y in zip(two.integrate(0.0005, 3, thermo=False) or (), tab.integrate(0.0005, 3, thermo=False) or ()):
        np.testing.assert_array_equal(x, y)
    for x, y in zip(two.get_state(), tab.get_state()):
        np.testing.assert_array_equal(x, y)
    if n <= 1000:
        b, lj = ljmd.from_system(s), oracle.LJ(s.eps, s.sigma, s.rcut, True)
        f, e, w = b.force()
        fo, eo, wo = oracle.forces_brute(s.box, s.pos, lj, s.type)
        assert np.max(np.linalg.norm(f - fo, axis=1) / pair_scale(s.box, s.pos, lj, s.type)) <= 1e-5
