"""The lane list kernel's two forms (four lanes per particle up to 2,048 cells,
one beyond) build exactly the FP64 neighbour sets: cells with fewer particles
than a pass and with several passes, rows longer than the lanes' buffers,
lists that outgrow the capacity, and the box sizes on either side of the rule."""
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


def _exact(s, rl):
    """Sorted neighbour sets by the definition |d|^2 < rl^2, d the minimum image in FP64."""
    pairs = cKDTree(np.mod(s.pos, s.box), boxsize=s.box).query_pairs(rl + 1e-6, output_type="ndarray")
    d = s.pos[pairs[:, 0]] - s.pos[pairs[:, 1]]
    d -= s.box * np.rint(d / s.box)
    pairs = pairs[np.sum(d * d, axis=1) < rl * rl]
    both = np.concatenate([pairs, pairs[:, ::-1]])
    return both[np.lexsort((both[:, 1], both[:, 0]))]


def _check(b, s, rl):
    c, nbr, _ = b.nlist()
    got = np.concatenate([np.stack([np.full(k, i), np.sort(nbr[i, :k])], axis=1) for i, k in enumerate(c)])
    np.testing.assert_array_equal(got, _exact(s, rl))


@pytest.mark.parametrize("n,rho,rcut", [(400, 0.05, 2.5), (3000, 0.8, 2.5), (3000, 1.1, 3.3), (30000, 0.3, 2.2),
                                        (41000, 0.85, 2.5), (46000, 0.85, 2.5)])
def test_lists_are_exact(ljmd, n, rho, rcut):
    s = inputs.fcc_subset_system(n, rho, 0.7, seed=n, rcut=rcut)
    _check(ljmd.from_system(s), s, rcut + 0.3)


def test_lists_regrow(ljmd):
    s = inputs.fcc_subset_system(2000, 0.9, 0.7, seed=1)
    b = ljmd.Box(s.pos, s.box)
    b.set_tuning(capacity=16)
    b.set_lj()
    _check(b, s, 2.8)
