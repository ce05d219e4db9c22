"""md_force's reduction and output in one launch: forces to device and host
memory and not at all, energies and virial equal to the allocation-free call's
(separate kernels) bit for bit, for one to several reduction items, odd chunk
counts, replicas and each precision; a non-finite force is still reported."""
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


@pytest.mark.parametrize("sizes,prec", [((300,), "mixed_ds"), ((4000,), "fp64"), ((20000,), "mixed_fp64"),
                                        ((70001,), "mixed_ds"), ((500, 9001, 1300), "mixed_ds")])
def test_outputs_agree(ljmd, sizes, prec):
    import torch
    ss = [inputs.fcc_subset_system(n, 0.8, 0.7, seed=n) for n in sizes]
    b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]), n=list(sizes), precision=prec)
    b.set_lj()
    f, e, w = b.force()
    dev = torch.zeros((sum(sizes), 3), dtype=torch.float64, device="cuda")
    b.force(out=dev)
    np.testing.assert_array_equal(dev.cpu().numpy(), f)
    sep = torch.zeros_like(dev)
    e2, w2 = np.zeros(len(sizes)), np.zeros(len(sizes))
    assert b._lib.md_force_noalloc(b._h, sep.data_ptr(), e2.ctypes.data, w2.ctypes.data) == 0
    np.testing.assert_array_equal(sep.cpu().numpy(), f)
    np.testing.assert_array_equal(e2, e)
    np.testing.assert_array_equal(w2, w)
    e3 = np.zeros(len(sizes))
    assert b._lib.md_force(b._h, None, e3.ctypes.data, None) == 0   # energies alone
    np.testing.assert_array_equal(e3, e)
    assert np.abs(f).max() > 0


def test_non_finite_forces_are_reported(ljmd):
    s = inputs.fcc_subset_system(500, 0.8, 0.7, seed=3)
    pos = s.pos.copy()
    pos[7] = pos[8]
    b = ljmd.Box(pos, s.box)
    b.set_lj()
    with pytest.raises(ljmd.MDError, match="non-finite"):
        b.force()
