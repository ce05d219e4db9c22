"""md_set_lj on a box that has already run: the step graphs captured with the
earlier parameters must not be replayed with them."""
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


@pytest.mark.parametrize("prec", ["mixed_ds", "mixed_fp64", "fp64"])
@pytest.mark.parametrize("again", [dict(eps=2.0), dict(sigma=0.9), dict(shift=False), dict(skin=0.2), dict(rcut=2.2)])
def test_run_after_a_change_of_parameters(ljmd, prec, again):
    s = inputs.fcc_subset_system(800, 0.8, 0.7, seed=1)
    a, b = (ljmd.Box(s.pos, s.box, s.vel, precision=prec) for _ in range(2))
    a.set_lj()
    a.integrate(0.004, 10)
    a.set_lj(**again)
    b.set_lj(**again)
    out = []
    for x in (a, b):
        x.set_state(s.pos, s.vel)
        out.append((x.integrate(0.004, 10), *x.get_state()[:2]))
    for x, y in zip(*out):
        np.testing.assert_allclose(x, y, rtol=1e-6, atol=1e-6)
