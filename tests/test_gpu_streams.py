"""Ordering of a box against the caller's stream: md_batch_create takes its
memory from the caller's pool, so everything it writes there must come after
the work already queued on the stream given at creation."""
import numpy as np
import pytest

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


def test_box_made_behind_queued_work_in_reused_memory(ljmd):
    """Tensors of the sizes a box allocates are written by kernels that are
    still queued when they are freed and the box is made in their memory."""
    import torch
    from paper_2406_04210_gb300 import inputs
    s = inputs.fcc_system(20, seed=11)
    pos, vel = (torch.tensor(a, device="cuda") for a in (s.pos, s.vel))
    torch.cuda.synchronize()
    ref = ljmd.Box(pos, s.box, vel).set_lj().force()
    for _ in range(3):
        slow = torch.ones(1 << 28, device="cuda")
        for _ in range(8):
            slow.mul_(1.0)                    # ~ms of work ahead of the writes below
        sizes = [64, 512, 4000, 8 * s.n, 16 * s.n, 24 * s.n, 1 << 20, 4 << 20]
        for t in [torch.empty(k, dtype=torch.uint8, device="cuda") for k in sizes * 3]:
            t.fill_(255)
        del t
        box = ljmd.Box(pos, s.box, vel).set_lj()
        f, e, w = box.force()
        assert np.array_equal(f, ref[0]) and np.array_equal(e, ref[1]) and np.array_equal(w, ref[2])


@pytest.mark.parametrize("side", [False, True])
def test_autograd_bridge_takes_transposed_tensors_on_any_stream(ljmd, side):
    """x0 and v0 stored by component, written on the current stream behind
    queued work, where the box was made on another one."""
    import torch
    from paper_2406_04210_gb300 import inputs
    s = inputs.fcc_system(6, seed=12)
    box = ljmd.from_system(s)
    one = torch.tensor(1.0, dtype=torch.float64)
    rng = np.random.default_rng(0)
    gx, gv = (torch.tensor(rng.normal(size=s.pos.shape), device="cuda") for _ in range(2))

    def run(x0, v0):
        x0, v0, e, g = (t.detach().requires_grad_() for t in (x0, v0, one, one))
        xT, vT = ljmd.TrajectoryFn.apply(x0, v0, e, g, box, s.dt, 4, 2)
        ((xT * gx).sum() + (vT * gv).sum()).backward()
        return [t.detach().cpu().numpy() for t in (xT, vT, x0.grad, v0.grad, e.grad, g.grad)]

    pos, vel = (torch.tensor(a, device="cuda") for a in (s.pos, s.vel))
    want = run(pos, vel)
    slow = torch.ones(1 << 28, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.current_stream()):
        for _ in range(8):
            slow.mul_(1.0)
        got = run(pos.t().contiguous().t(), vel.t().contiguous().t())
        torch.cuda.synchronize()
    for w, g in zip(want, got):
        np.testing.assert_array_equal(g, w)
