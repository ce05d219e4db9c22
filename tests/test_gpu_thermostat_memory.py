"""A thermostatted run whose buffer for collisions drawn ahead cannot be allocated
draws them in its steps: the same run, not an error."""
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


def test_refused_buffer(ljmd):
    import torch
    limit = [None]

    def alloc(nbytes, ctx):
        if limit[0] is not None and nbytes > limit[0]:
            return 0
        return int(torch.cuda.caching_allocator_alloc(int(nbytes)))

    def free(ptr, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    a, f = ljmd._ALLOC(alloc), ljmd._FREE(free)
    s = inputs.fcc_subset_system(2000, 0.8, 0.7, seed=8)
    out = []
    L = ljmd.load()
    L.md_set_allocator(a, f, None)
    try:
        for refuse in (False, True):
            limit[0] = None
            b = ljmd.from_system(s).set_thermostat(1.3, 20.0, seed=6)
            limit[0] = 1 << 19 if refuse else None   # 20 steps of 2,016 particles take 970 kB
            th = [b.integrate(0.002, n) for n in (20, 20, 5)]   # 5 steps (242 kB) fit
            out.append((np.concatenate(th), *b.get_state()[:2]))
            limit[0] = None
            b.close()
    finally:
        ljmd._install_torch_allocator(L)
    for x, y in zip(*out):
        np.testing.assert_allclose(y, x, rtol=0, atol=1e-9)
