"""What a user of this library has it do, as cases that can be timed.

Every case goes through the public entry points (the Python binding and the C ABI calls
under it) with particle data on the GPU.  A case is a dict of plain values; ``kind`` says
what the program does:

* ``md``        one box: velocity-Verlet steps with the skin-rule list updates, then the
                state read out (one species, or the 80:20 binary mixture with ``species`` 2);
* ``replicas``  many boxes of uneven size advanced together, then the state read out;
* ``allpairs``  untruncated forces over all pairs with the Andersen-like thermostat;
* ``force``     one force/energy/virial call at the current positions (lists are current);
* ``evaluate``  new positions from outside, then forces (binning, list build, force);
* ``gradient``  a recorded trajectory, the pair-histogram loss and its gradient with
                respect to the initial state and both LJ parameters (torch.autograd).

Plain runs continue their trajectory from pass to pass, as a simulation does.  Results of
the FP32-force precisions are handed on in single precision (what those forces hold; the
library's arrays are FP64 whatever the precision), those of the FP64 precision in FP64.
Positions are returned unwrapped (position + image count x edge), as an analysis takes
them.  ``exact`` restates each computation in plain torch FP64.
"""
import math

import numpy as np
import torch

from paper_2406_04210_gb300 import ljmd

RHO, TEMP, DT, RC, SKIN = 0.8442, 0.722, 0.005, 2.5, 0.3
BINARY_EPS = [[1.0, 1.5], [1.5, 0.5]]
BINARY_SIGMA = [[1.0, 0.8], [0.8, 0.88]]
NBINS, RHIST, RMAX = 64, 2.5, 2.8
WIDTH = RHIST / NBINS
FCC = [[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]]


def listed():
    return [
        # one call on the smallest configuration (an external driver asking for forces): latency
        {"name": "force_4k", "kind": "force", "n": 4000, "rho": RHO, "T": TEMP, "precision": "mixed_ds"},
        # the N = 4000 fluid (fcc 10^3 x 4) as a default-precision run with energies every step:
        # many short launches
        {"name": "md_4k", "kind": "md", "n": 4000, "rho": RHO, "T": TEMP, "precision": "mixed_ds", "species": 1,
         "steps": 50, "thermo": True},
        # the same fluid by the plain all-FP64 method
        {"name": "md_4k_fp64", "kind": "md", "n": 4000, "rho": RHO, "T": TEMP, "precision": "fp64", "species": 1,
         "steps": 50, "thermo": True},
        # the truncated-force study's fluid of 10^5 particles, hot (frequent list updates)
        {"name": "md_100k_hot", "kind": "md", "n": 100000, "rho": RHO, "T": 1.5, "precision": "mixed_ds",
         "species": 1, "steps": 50, "thermo": True},
        # the large fluid (fcc 100^3 x 4): the throughput run
        {"name": "md_4m", "kind": "md", "n": 4000000, "rho": RHO, "T": TEMP, "precision": "mixed_ds", "species": 1,
         "steps": 20, "thermo": True},
        # all-FP64 reference run of a middling box
        {"name": "md_256k_fp64", "kind": "md", "n": 256000, "rho": RHO, "T": TEMP, "precision": "fp64", "species": 1,
         "steps": 10, "thermo": True},
        # FP32 forces over FP64 state, a ragged million, no energies (equilibration)
        {"name": "md_1m_fp64state", "kind": "md", "n": 1000003, "rho": RHO, "T": 1.0, "precision": "mixed_fp64",
         "species": 1, "steps": 20, "thermo": False},
        # the dense 80:20 mixture, two species (tables instead of constants)
        {"name": "binary_256k", "kind": "md", "n": 256000, "rho": 1.2, "T": 0.7, "precision": "mixed_ds",
         "species": 2, "steps": 20, "thermo": True},
        # 512 independent boxes, N log-uniform in [500, 20000], densities and temperatures of their own
        {"name": "replicas_512", "kind": "replicas", "nrep": 512, "nmin": 500, "nmax": 20000, "precision": "mixed_ds",
         "steps": 20},
        # the all-to-all workload: N = 2000, untruncated, thermostatted
        {"name": "allpairs_2k", "kind": "allpairs", "n": 2000, "rho": RHO, "T": TEMP, "rate": 1.0,
         "precision": "mixed_ds", "steps": 50},
        # positions of an outside program (a Monte Carlo move, a minimiser): list build + forces, ragged
        {"name": "evaluate_500k", "kind": "evaluate", "n": 500009, "rho": 0.75, "T": 1.0, "precision": "mixed_ds"},
        # the differentiable fluid (fcc 20^3 x 4): trajectory, histogram loss, gradients
        {"name": "gradient_32k", "kind": "gradient", "n": 32000, "rho": RHO, "T": TEMP, "steps": 40, "ckpt": 20},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["force", "md", "md", "md", "replicas", "allpairs", "evaluate", "gradient"])
    rho, T = round(rng.uniform(0.6, 0.95), 4), round(rng.uniform(0.5, 3.0), 3)
    prec = rng.choice(["mixed_ds", "mixed_ds", "mixed_fp64", "fp64"])
    if kind == "force":
        return {"kind": kind, "n": size(500, 1000000), "rho": rho, "T": T, "precision": prec}
    if kind == "md":
        two = rng.random() < 0.25
        n = size(500, 120000 if prec == "fp64" else 3000000)
        return {"kind": kind, "n": n, "rho": 1.2 if two else rho, "T": 0.7 if two else T, "precision": prec,
                "species": 2 if two else 1, "steps": rng.randint(8, 20) if n > 100000 else rng.randint(20, 50),
                "thermo": rng.random() < 0.7}
    if kind == "replicas":
        return {"kind": kind, "nrep": size(4, 400), "nmin": 500, "nmax": rng.randint(2000, 20000),
                "precision": rng.choice(["mixed_ds", "mixed_fp64"]), "steps": rng.randint(8, 20)}
    if kind == "allpairs":
        return {"kind": kind, "n": size(300, 8000), "rho": rho, "T": T, "rate": rng.choice([0.0, 0.5, 1.0, 4.0]),
                "precision": prec if prec != "fp64" else "mixed_ds", "steps": rng.randint(20, 50)}
    if kind == "evaluate":
        return {"kind": kind, "n": size(1000, 2000000), "rho": rho, "T": T, "precision": prec}
    ck = rng.choice([5, 10, 20])
    return {"kind": kind, "n": size(1000, 60000), "rho": round(rng.uniform(0.75, 0.9), 4), "T": TEMP,
            "steps": ck * rng.randint(1, 40 // ck), "ckpt": ck}


# ---- inputs: n sites of the smallest fcc lattice with at least n, jitter 0.05, Maxwell-Boltzmann velocities ----
def _fluid(n, rho, T, g):
    dev = g.device
    L = (n / rho) ** (1.0 / 3.0)
    m = max(1, int(round((n / 4.0) ** (1.0 / 3.0))))
    while 4 * m ** 3 < n:
        m += 1
    while m > 1 and 4 * (m - 1) ** 3 >= n:
        m -= 1
    pick = torch.randperm(4 * m ** 3, generator=g, device=dev)[:n].sort().values if 4 * m ** 3 > n else torch.arange(n, device=dev)
    cell, k = pick // 4, pick % 4
    corner = torch.stack([cell % m, (cell // m) % m, cell // (m * m)], dim=1).double()
    pos = (corner + torch.tensor(FCC, dtype=torch.float64, device=dev)[k]) * (L / m)
    pos = pos + (torch.rand((n, 3), generator=g, device=dev, dtype=torch.float64) * 2 - 1) * 0.05
    pos = pos - L * torch.floor(pos / L)
    vel = torch.randn((n, 3), generator=g, device=dev, dtype=torch.float64)
    vel -= vel.mean(dim=0, keepdim=True)
    vel *= torch.sqrt((3.0 * n - 3.0) * T / vel.square().sum())
    return pos.contiguous(), vel.contiguous(), L


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _dt(case):
    return 0.003 if case.get("species") == 2 else DT


def _inputs(case, seed):
    """Positions, velocities, edge of every replica, particles of every replica, species (int32 or None)."""
    g = _gen(seed)
    if case["kind"] == "replicas":
        h = torch.Generator().manual_seed(20000 + int(case["nrep"]))   # the sizes are the case's own
        u = torch.rand((case["nrep"], 3), generator=h, dtype=torch.float64).tolist()
        n = [int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** a[0])) for a in u]
        parts = [_fluid(k, 0.6 + 0.35 * a[1], 0.7 + 0.8 * a[2], g) for k, a in zip(n, u)]
        return torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts]), [p[2] for p in parts], n, None
    pos, vel, L = _fluid(case["n"], case["rho"], case["T"], g)
    types = None
    if case.get("species") == 2:
        types = torch.zeros(case["n"], dtype=torch.int32, device="cuda")
        types[torch.randperm(case["n"], generator=g, device="cuda")[: case["n"] // 5]] = 1
    return pos, vel, [L], [case["n"]], types


def _params(case):
    if case.get("species") == 2:
        s = np.array(BINARY_SIGMA)
        return np.array(BINARY_EPS), s, 2.5 * s
    return 1.0, 1.0, (math.inf if case["kind"] == "allpairs" else RC)


def _target(case, g):
    """A histogram to fit: the ideal gas's, with some structure."""
    c = (torch.arange(NBINS, dtype=torch.float64, device="cuda") + 0.5) * RHIST / NBINS
    ideal = 2.0 * math.pi * case["rho"] * c * c * WIDTH * math.sqrt(2.0 * math.pi)
    return ideal * (1.0 + 0.3 * torch.randn(NBINS, generator=g, dtype=torch.float64, device="cuda"))


def prepare(case, seed):
    pos, vel, L, n, types = _inputs(case, seed)
    prec = case.get("precision", "mixed_ds")
    torch.cuda.synchronize()   # the inputs are there before a box is made of them, as after loading a file
    box = ljmd.Box(pos, np.repeat(np.array(L)[:, None], 3, axis=1), vel, types, n=n, precision=prec)
    eps, sigma, rcut = _params(case)
    box.set_lj(eps, sigma, rcut, SKIN)
    s = {"case": case, "box": box, "pos": pos, "vel": vel,
         "edge": torch.tensor(np.repeat(L, n)[:, None], device="cuda")}
    if case["kind"] == "allpairs" and case["rate"] > 0:
        box.set_thermostat(case["T"], case["rate"], seed=int(seed))
    if case["kind"] == "evaluate":   # what the outside program moves to
        s["moved"] = pos + 0.03 * torch.randn(pos.shape, generator=_gen(seed + 1), dtype=torch.float64, device="cuda")
    if case["kind"] == "gradient":
        s["target"] = _target(case, _gen(seed + 2))
        s["eps"], s["sigma"] = (torch.tensor(1.0, dtype=torch.float64, device="cuda") for _ in range(2))
    return s


def _hand_on(case, out):
    """FP32-force results in single precision."""
    if case.get("precision", "mixed_ds") == "fp64":
        return out
    return {k: v.float() if isinstance(v, torch.Tensor) else v.astype(np.float32) for k, v in out.items()}


def run(s):
    case, box = s["case"], s["box"]
    kind = case["kind"]
    if kind == "gradient":
        x0, v0, eps, sigma = (t.detach().requires_grad_() for t in (s["pos"], s["vel"], s["eps"], s["sigma"]))
        xT, vT = ljmd.TrajectoryFn.apply(x0, v0, eps, sigma, box, DT, case["steps"], case["ckpt"])
        loss = ljmd.PairHistLossFn.apply(xT, box, s["target"], NBINS, RHIST, WIDTH, RMAX)
        loss.backward()
        return _hand_on(case, {"loss": loss.detach(), "vT": vT.detach(), "dx0": x0.grad, "dv0": v0.grad,
                               "deps": eps.grad, "dsigma": sigma.grad})
    if kind in ("force", "evaluate"):
        if kind == "evaluate":
            box.set_state(s["moved"])
        f, e, w = box.force(out=torch.empty_like(s["pos"]))
        return _hand_on(case, {"force": f, "epot": e, "virial": w})
    out = {}
    if case.get("thermo", True):
        log = torch.empty((case["steps"], box.nrep, 4), dtype=torch.float64, device="cuda")
        out["thermo"] = box.integrate(_dt(case), case["steps"], out=log)
    else:
        box.integrate(_dt(case), case["steps"], thermo=False)
    x, v = torch.empty_like(s["pos"]), torch.empty_like(s["pos"])
    img = torch.empty(x.shape, dtype=torch.int32, device="cuda")
    box._check(ljmd.load().md_get_state(box._h, x.data_ptr(), v.data_ptr(), img.data_ptr()), "md_get_state")
    out["x"], out["v"] = x + img * s["edge"], v
    return _hand_on(case, out)


# ---- the least a pass has to do ----
def work(case):
    """MD steps: offsets and velocities (24 B each) read and written once per particle and step, and every pair
    within the cutoff evaluated once (~25 operations).  A force call: positions read, forces written.  A
    gradient step: the forward step, and in reverse the same pairs' Hessian products (~50) and adjoint state."""
    kind = case["kind"]
    if kind == "replicas":
        lo, hi = case["nmin"], case["nmax"]
        n, rho = case["nrep"] * (hi - lo) / math.log(hi / lo), 0.775
    else:
        n, rho = case["n"], case["rho"]
    rc = 2.5 if case.get("species") != 2 else 2.2
    pairs = 0.5 * n * (n - 1) if kind == "allpairs" else 0.5 * n * rho * 4.18879 * rc ** 3
    if kind in ("force", "evaluate"):
        return {"bytes": n * (48.0 if kind == "force" else 48.0 + 24.0), "flops": 25.0 * pairs}
    if kind == "gradient":
        return {"bytes": case["steps"] * n * 192.0, "flops": case["steps"] * 75.0 * pairs + 64 * 12 * pairs}
    return {"bytes": case["steps"] * n * 96.0, "flops": case["steps"] * 25.0 * pairs}


# ---- the same computations in plain FP64 torch ----
class _Pairs:
    """All pairs i < j of every replica within `reach` (all of them for reach = inf), found by brute force
    (small replicas) or cells, kept while no particle has moved more than half the reach's margin over `need`."""

    def __init__(self, x, L, n, need, margin):
        self.L, self.n, self.need, self.margin = L, n, need, margin
        self.edge = torch.tensor(L, dtype=torch.float64, device=x.device)
        self.rep = torch.repeat_interleave(torch.arange(len(n), device=x.device), torch.tensor(n, device=x.device))
        self.at = None
        self.find(x)

    def current(self, x):
        if math.isfinite(self.need) and float((x - self.at).square().sum(1).max()) > (0.5 * self.margin) ** 2:
            self.find(x)

    def find(self, x):
        reach, off, got = self.need + self.margin, 0, []
        for L, n in zip(self.L, self.n):
            p = x[off:off + n]
            p = p - L * torch.floor(p / L)
            if n <= 12000:
                i, j = self._brute(p, L, reach)
            else:
                i, j = self._cells(p, L, reach)
            got.append((i + off, j + off))
            off += n
        self.i, self.j = torch.cat([a for a, _ in got]), torch.cat([b for _, b in got])
        self.at = x.clone()

    @staticmethod
    def _brute(p, L, reach):
        n = p.shape[0]
        if not math.isfinite(reach):
            return tuple(torch.triu_indices(n, n, 1, device=p.device))
        r2 = torch.zeros((n, n), dtype=torch.float64, device=p.device)
        for c in range(3):
            d = p[:, None, c] - p[None, :, c]
            d -= L * torch.round(d / L)
            r2 += d * d
        return tuple(torch.nonzero((r2 < reach * reach).triu_(1), as_tuple=True))

    @staticmethod
    def _cells(p, L, reach):
        dev, n = p.device, p.shape[0]
        m = int(L / reach)
        c = torch.clamp((p * (m / L)).long(), max=m - 1)
        order = torch.argsort(c[:, 0] + m * (c[:, 1] + m * c[:, 2]))
        cid = (c[:, 0] + m * (c[:, 1] + m * c[:, 2]))[order]
        count = torch.bincount(cid, minlength=m ** 3)
        first = torch.cumsum(count, 0) - count
        most = int(count.max())
        table = torch.full((m ** 3, most), -1, dtype=torch.long, device=dev)
        table[cid, torch.arange(n, device=dev) - first[cid]] = order
        far = torch.cat([p, torch.full((1, 3), 1e30, dtype=torch.float64, device=dev)])   # row -1: no particle
        cells = torch.arange(m ** 3, device=dev)
        cx, cy, cz = cells % m, (cells // m) % m, cells // (m * m)
        got = []
        for k in range(13, 27):
            dx, dy, dz = k % 3 - 1, (k // 3) % 3 - 1, k // 9 - 1
            nb = (cx + dx) % m + m * ((cy + dy) % m + m * ((cz + dz) % m))
            step = max(1, 40_000_000 // (most * most))
            for a in range(0, m ** 3, step):
                ia, jb = table[a:a + step], table[nb[a:a + step]]
                r2 = torch.zeros((ia.shape[0], most, most), dtype=torch.float64, device=dev)
                for q in range(3):
                    d = far[ia, q][:, :, None] - far[jb, q][:, None, :]
                    d -= L * torch.round(d / L)
                    r2 += d * d
                ok = (r2 < reach * reach) & (ia >= 0)[:, :, None] & (jb >= 0)[:, None, :]
                if k == 13:
                    ok &= torch.ones((most, most), dtype=torch.bool, device=dev).triu(1)
                w, u, v = torch.nonzero(ok, as_tuple=True)
                got.append((ia[w, u], jb[w, v]))
        return torch.cat([a for a, _ in got]), torch.cat([b for _, b in got])

    def vectors(self, x):
        L = self.edge[self.rep[self.i]][:, None]
        d = x[self.i] - x[self.j]
        d -= L * torch.round(d / L)
        return d, d.square().sum(1)


class _LJ:
    def __init__(self, case, types):
        t = lambda a: torch.as_tensor(np.atleast_2d(a), dtype=torch.float64, device="cuda")  # noqa: E731
        self.eps, self.sigma, self.rc = (t(a) for a in _params(case))
        self.types = types.long() if types is not None else None

    def of(self, pairs):
        if self.types is None:
            return self.eps[0, 0], self.sigma[0, 0], self.rc[0, 0]
        a, b = self.types[pairs.i], self.types[pairs.j]
        return self.eps[a, b], self.sigma[a, b], self.rc[a, b]


def _forces(x, pairs, lj):
    """Forces, E_pot and W per replica."""
    d, r2 = pairs.vectors(x)
    e, s, rc = lj.of(pairs)
    near = r2 < rc * rc
    r2 = torch.where(near, r2, torch.inf)
    s6 = (s * s / r2) ** 3
    f = 48.0 * e / r2 * s6 * (s6 - 0.5)
    c6 = (s / rc) ** 6
    u = torch.where(near, 4.0 * e * (s6 * (s6 - 1.0) - c6 * (c6 - 1.0)), 0.0)
    w = 48.0 * e * s6 * (s6 - 0.5)
    fd = f[:, None] * d
    F = torch.zeros_like(x).index_add_(0, pairs.i, fd).index_add_(0, pairs.j, fd, alpha=-1.0)
    z = torch.zeros(len(pairs.n), dtype=torch.float64, device=x.device)
    rep = pairs.rep[pairs.i]
    return F, z.index_add(0, rep, u), z.index_add(0, rep, w)


def _philox(c, key):
    """Philox4x32-10 on four arrays of 32-bit words (as uint64)."""
    m = np.uint64(0xFFFFFFFF)
    c = [np.asarray(a, dtype=np.uint64) for a in c]
    k0, k1 = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p, q = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(q >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), q & m, (p >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _collide(v, case, seed, step, dt):
    n = v.shape[0]
    u, z = np.arange(n, dtype=np.uint64), np.zeros(n, dtype=np.uint64)
    a = _philox([u, z + np.uint64(step), z, z], int(seed))
    hit = np.nonzero(a[0] < min(2 ** 32 - 1, math.floor(case["rate"] * dt * 2.0 ** 32)))[0]
    if not len(hit):
        return
    b = _philox([u, z + np.uint64(step), z, z + np.uint64(1)], int(seed))
    real = lambda w: (w[hit].astype(np.float64) + 0.5) / 2.0 ** 32  # noqa: E731
    r1, t1 = np.sqrt(-2.0 * np.log(real(a[1]))), 2.0 * np.pi * real(a[2])
    r2, t2 = np.sqrt(-2.0 * np.log(real(b[0]))), 2.0 * np.pi * real(b[1])
    g = math.sqrt(case["T"]) * np.stack([r1 * np.cos(t1), r1 * np.sin(t1), r2 * np.cos(t2)], axis=1)
    v[torch.from_numpy(hit).to(v.device)] = torch.from_numpy(g).to(v.device)


def _hessian(x, u, pairs, lj):
    """H u, and u . dF/deps, u . dF/dsigma (one species)."""
    d, r2 = pairs.vectors(x)
    e, s, rc = lj.of(pairs)
    r2 = torch.where(r2 < rc * rc, r2, torch.inf)
    s6 = (s * s / r2) ** 3
    f = 48.0 * e / r2 * s6 * (s6 - 0.5)
    A = e * s6 * (672.0 * s6 - 192.0) / (r2 * r2)
    uij = u[pairs.i] - u[pairs.j]
    du = (d * uij).sum(1)
    h = (A * du)[:, None] * d - f[:, None] * uij
    H = torch.zeros_like(x).index_add_(0, pairs.i, h).index_add_(0, pairs.j, h, alpha=-1.0)
    return H, (f / e * du).sum(), (e / s / r2 * s6 * (576.0 * s6 - 144.0) * du).sum()


def _histogram(x, pairs, n):
    d, r2 = pairs.vectors(x)
    keep = r2 < RMAX * RMAX
    d, r = d[keep], r2[keep].sqrt()
    c = (torch.arange(NBINS, dtype=torch.float64, device=x.device) + 0.5) * RHIST / NBINS
    g = torch.exp(-(r[:, None] - c).square() / (2.0 * WIDTH * WIDTH)) / n
    slope = -(r[:, None] - c) / (WIDTH * WIDTH) * g

    def gradient(coef):
        t = ((slope @ coef) / r)[:, None] * d
        return torch.zeros_like(x).index_add_(0, pairs.i[keep], t).index_add_(0, pairs.j[keep], t, alpha=-1.0)

    return g.sum(0), gradient


def exact(case, seed):
    pos, vel, L, n, types = _inputs(case, seed)
    lj, kind, dt = _LJ(case, types), case["kind"], _dt(case)
    if kind == "evaluate":
        pos = pos + 0.03 * torch.randn(pos.shape, generator=_gen(seed + 1), dtype=torch.float64, device="cuda")
    need = max(float(lj.rc.max()), RMAX) if kind == "gradient" else float(lj.rc.max())
    pairs = _Pairs(pos, L, n, need, 0.35)
    F, e, w = _forces(pos, pairs, lj)
    if kind in ("force", "evaluate"):
        return {"force": F, "epot": e, "virial": w}
    x, v = pos.clone(), vel.clone()
    dof = torch.tensor([3.0 * k - 3.0 for k in n], dtype=torch.float64, device="cuda")
    log, states = [], [x.clone()]
    for step in range(case["steps"]):
        v += 0.5 * dt * F
        x += dt * v
        pairs.current(x)
        F, e, w = _forces(x, pairs, lj)
        v += 0.5 * dt * F
        if kind == "allpairs" and case["rate"] > 0:
            _collide(v, case, seed, step, dt)
        if kind == "gradient":
            states.append(x.clone())
        else:
            k = torch.zeros_like(e).index_add(0, pairs.rep, 0.5 * v.square().sum(1))
            log.append(torch.stack([e, k, w, 2.0 * k / dof], dim=1))
    if kind != "gradient":
        out = {"thermo": torch.stack(log), "x": x, "v": v}
        if not case.get("thermo", True):
            del out["thermo"]
        return out
    hist, gradient = _histogram(x, pairs, n[0])
    off = hist - _target(case, _gen(seed + 2))
    loss = off.square().mean()
    lx, lv = gradient(2.0 * off / NBINS), torch.zeros_like(v)
    H, de, ds = _hessian(x, lv, pairs, lj)
    deps, dsigma = 0.5 * dt * de, 0.5 * dt * ds
    for step in range(case["steps"], 0, -1):
        lx = lx - 0.5 * dt * H
        lv = lv + dt * lx
        pairs.current(states[step - 1])
        H, de, ds = _hessian(states[step - 1], lv, pairs, lj)
        half = 0.5 if step == 1 else 1.0
        deps, dsigma = deps + half * dt * de, dsigma + half * dt * ds
        lx = lx - 0.5 * dt * H
    return {"loss": loss, "vT": v, "dx0": lx, "dv0": lv, "deps": deps, "dsigma": dsigma}
