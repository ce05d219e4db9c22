"""The launch grids chosen by size (a block per work item, or a few per SM) do
not change any bit: forces, energies and lists of the automatic grids against
fixed ones, at chunk counts around the SMs' blocks and for the mixture."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("species,n", [(1, 65537), (1, 116737), (1, 160001), (2, 70000)])
def test_grids_do_not_change_results(ljmd, species, n):
    s = inputs.fcc_subset_system(n, 0.8, 0.7, seed=n) if species == 1 else inputs.binary_random_system(n, seed=2)
    a, b = ljmd.from_system(s), ljmd.from_system(s)
    b.set_tuning(force_blocks_per_sm=3, list_blocks_per_sm=5)
    b.neighbour_update(True)
    for x, y in zip(a.force(), b.force()):
        np.testing.assert_array_equal(x, y)
    ca, na, _ = a.nlist()
    cb, nb, _ = b.nlist()
    np.testing.assert_array_equal(ca, cb)
    assert all((na[i, :c] == nb[i, :c]).all() for i, c in enumerate(ca))
    for x, y in zip(a.integrate(0.001, 5), b.integrate(0.001, 5)):
        np.testing.assert_array_equal(x, y)


def test_small_boxes_follow_the_set_grid(ljmd):
    # a quarter of a wave of small blocks per SM against all of them: the same forces, later
    s = inputs.fcc_subset_system(60000, 0.8, 0.7, seed=5)
    b = ljmd.from_system(s)
    forces, ms = [], []
    for per_sm in (0, 1):
        b.set_tuning(force_blocks_per_sm=per_sm)
        forces.append(b.force()[0])
        b.integrate(0.001, 5)
        b.set_profiling(True)
        b.integrate(0.001, 20)
        t, launches = b.profile()["force"]
        b.set_profiling(False)
        b.set_state(s.pos, s.vel)
        ms.append(t / launches)
    np.testing.assert_array_equal(*forces)
    assert ms[1] > 1.3 * ms[0]


def test_autotune_keeps_the_automatic_force_grid(ljmd):
    # a block per chunk, more than 32 per SM: no candidate is 2 % faster (they are 1 to 10 % slower)
    s = inputs.fcc_subset_system(1000000, 0.8442, 0.7, seed=6)
    b = ljmd.from_system(s)
    f0 = b.force()[0]
    t = b.autotune(reps=10, cache=False)
    assert t["force_blocks_per_sm"] == 0 == b.tuning()["force_blocks_per_sm"]
    assert np.abs(b.force()[0] - f0).max() <= 1e-4 * np.abs(f0).max()
