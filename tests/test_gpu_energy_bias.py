"""The FP32 list force's energy is w / 12 less a second sum; its constants are
rounded so that they do not shift the energy of all particles alike.  The tiled
kernel, which sums pair energies with constants that are exact at sigma = 1, has
no such shift: under pressure (w / 12 = 20 per particle) the two may differ by
what the rounding of the particles' sums (20 x 2^-24 each, of either sign) leaves
in the mean of 32,000, 7e-9, and not by 20 x 3e-8."""
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


# cell edges of 3, exact in FP32; small work items and chunks
@pytest.mark.parametrize("ncell,L", [(20, 27.0), (26, 36.0)])
def test_force_kernels_agree_in_the_mean(ljmd, ncell, L):
    s = inputs.fcc_system(ncell, rho=4 * ncell ** 3 / L ** 3, seed=3)
    e = []
    for kind in ("chunks", "tiles"):
        b = ljmd.from_system(s)
        b.force_kernel = kind
        e.append(b.force()[1][0] / s.n)
    assert abs(e[0] - e[1]) <= 1e-7
