"""Velocities whose double-single words are subnormal FP32 numbers (or whose low
word is) come back as those words' sum, before and after a list build."""
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


def test_round_trip(ljmd):
    s = inputs.fcc_subset_system(500, 0.8, 0.7, seed=4)
    v = s.vel.copy()
    v.ravel()[:12] = [0.0, -0.0, 1e-39, -1.1754942e-38, 3e-42, 1.4e-45, -7e-46, 1.2e-38, 1e-35 * (1 + 2.0 ** -26),
                      -3e-37 * (1 + 2.0 ** -25), 1.0 + 2.0 ** -30, -2.0 ** -126]
    hi = v.astype(np.float32)
    lo = (v - hi.astype(np.float64)).astype(np.float32)
    want = hi.astype(np.float64) + lo.astype(np.float64)
    b = ljmd.from_system(s)
    b.set_state(s.pos, v)
    np.testing.assert_array_equal(b.get_state()[1], want)
    b.neighbour_update(True)
    np.testing.assert_array_equal(b.get_state()[1], want)
