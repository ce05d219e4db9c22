"""The FP64 list-form force kernel at the edges of its work split: particles
ending inside a quarter of a chunk, rows longer than one scan (96 entries) and
than the queue's multiples, empty rows, two species, replicas.  Against the
FP64 oracle's brute force: max |dF| / S_i <= 1e-12, S_i = sum_j |F_ij| (the
tolerance of test_gpu_md.py), energies relative 1e-12."""
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


def _check(b, s, sl=slice(None), r=0):
    lj = oracle.LJ(s.eps, s.sigma, s.rcut, True)
    f, e, w = b.force()
    fo, eo, wo = oracle.forces_brute(s.box, s.pos, lj, s.type) if s.ntypes > 1 else oracle.forces_brute(s.box, s.pos, lj)
    S = np.maximum(pair_scale(s.box, s.pos, lj, s.type) if s.ntypes > 1 else pair_scale(s.box, s.pos, lj), 1e-30)
    assert np.max(np.linalg.norm(f[sl] - fo, axis=1) / S) <= 1e-12
    assert abs(e[r] - eo) <= 1e-12 * abs(eo) and abs(w[r] - wo) <= 1e-12 * 0.5 * s.rcut.max() * S.sum()


@pytest.mark.parametrize("n", [257, 383, 1000])
def test_ragged_sizes(ljmd, n):
    s = inputs.fcc_subset_system(n, 0.8, 0.7, seed=n)
    _check(ljmd.from_system(s, "fp64"), s)


@pytest.mark.parametrize("rcut,rho", [(2.5, 1.15), (3.2, 1.0), (4.3, 0.9)])
def test_long_rows(ljmd, rcut, rho):
    s = inputs.fcc_subset_system(1331, rho, 0.7, seed=3, rcut=rcut)   # ~110, ~180 and ~370 entries a row
    b = ljmd.from_system(s, "fp64")
    assert b.nlist()[0].max() > 96
    _check(b, s)


def test_two_species(ljmd):
    s = inputs.binary_random_system(1200, seed=4)
    _check(ljmd.from_system(s, "fp64"), s)


def test_replicas(ljmd):
    ss = [inputs.fcc_subset_system(n, 0.8, 0.7, seed=n) for n in (200, 640, 333)]
    b = ljmd.Box(np.concatenate([s.pos for s in ss]), np.stack([s.box for s in ss]), n=[s.n for s in ss],
                 precision="fp64")
    b.set_lj(1.0, 1.0, 2.5, 0.3)
    at = 0
    for r, s in enumerate(ss):
        _check(b, s, slice(at, at + s.n), r)
        at += s.n
