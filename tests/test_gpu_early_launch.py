"""Step graphs with programmatic launches (all kernels of a step up to 64
chunks, the rebuild kernels beyond, the list build with one replica) give bit
for bit what profiled graphs, which have none, give: hot runs with several list
builds, both sides of the rule, every precision, mixture, replicas, all pairs."""
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


def _run(make, profiled, dt, steps):
    b = make()
    b.set_profiling(profiled)
    th = [b.integrate(dt, steps) for _ in range(2)]
    return [*th, *b.get_state()]


@pytest.mark.parametrize("n,prec", [(500, "mixed_ds"), (8192, "mixed_ds"), (8193, "mixed_ds"), (8192, "fp64"),
                                    (20000, "mixed_fp64"), (40000, "mixed_ds"),
                                    (49152, "mixed_ds"), (49153, "mixed_ds"), (140000, "mixed_ds")])
def test_one_box(ljmd, n, prec):
    s = inputs.fcc_subset_system(n, 0.8, 3.0, seed=n)
    for x, y in zip(*(_run(lambda: ljmd.from_system(s, prec), prof, 0.003, 30) for prof in (False, True))):
        np.testing.assert_array_equal(x, y)


def test_mixture_replicas_and_all_pairs(ljmd):
    s = inputs.binary_random_system(3000, seed=4)
    ss = [inputs.fcc_subset_system(n, 0.8, 2.0, seed=n) for n in (200, 640, 333)]

    def replicas():
        b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]),
                     np.concatenate([s.vel for s in ss]), n=[s.n for s in ss])
        b.set_lj()
        b.set_thermostat(np.full(3, 1.2), 0.5, 7)
        return b

    def pairs():
        b = ljmd.Box(ss[1].pos, ss[1].box, ss[1].vel)
        b.set_lj(1.0, 1.0, np.inf)
        return b

    for make in (lambda: ljmd.from_system(s), replicas, pairs):
        for x, y in zip(_run(make, False, 0.001, 20), _run(make, True, 0.001, 20)):
            np.testing.assert_array_equal(x, y)
