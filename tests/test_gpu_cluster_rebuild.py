"""Small boxes bin, sort and gather in one cluster launch; with conditional
step graphs the same stages run as separate kernels.  Both must give the same
trajectories and energies bit for bit: one scan tile and two (over 2048
cells), several replicas of uneven size, the largest boxes on the cluster path
(49,152 slots) and the first beyond it, each precision."""
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
@pytest.mark.parametrize("sizes,rho,rcut", [((300,), 0.8, 2.5), ((32768,), 0.7, 2.2), ((32769,), 0.7, 2.2),
                                            ((49152,), 0.7, 2.2), ((49153,), 0.7, 2.2),
                                            ((500, 4001, 977), 0.8, 2.5)])
def test_cluster_and_separate_rebuilds_agree(ljmd, sizes, rho, rcut, prec):
    ss = [inputs.fcc_subset_system(n, rho, 2.0, seed=n, rcut=rcut) for n in sizes]
    out = []
    for cond in (True, False):
        b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]),
                     np.concatenate([s.vel for s in ss]), n=list(sizes), precision=prec)
        b.set_lj(1.0, 1.0, rcut, 0.3)
        b.graph_conditional = cond
        th = b.integrate(0.005, 30)
        out.append((*b.get_state(), th, b.info().rebuilds))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
    assert out[0][-1] > len(sizes) * 2   # lists were rebuilt on the way
