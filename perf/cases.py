"""Workloads that the tree-code is timed on, each through its public entry points.

A case is a dict of plain values; ``kind`` says what one pass does:

* ``eval``: new bodies in, accelerations and potentials out (set_bodies,
  build, multipoles, forces), from device tensors or page-locked host
  arrays; with ``learned`` the theta = 1 walk with the network's correction
  and its judge (forces_learned);
* ``step``: one shared kick-drift-kick step and the new state in caller order;
* ``ensemble``: one such step of many independent systems at once;
* ``block``: one cycle of block time steps and the new state;
* ``sph``: neighbour counts and SPH densities on a built tree;
* ``train``: training of the correction's network from scratch on host rows;
* ``sort``: the allocation-free stable key sort.

Bodies are Plummer spheres in Henon units (or two of them, merging), drawn on
the GPU from the seed alone.
"""
import math

import numpy as np
import torch

import paper_1204_2280_gb300 as B
from paper_1204_2280_gb300 import learned as L

A_HENON = 3.0 * math.pi / 16.0   # Plummer scale length in Henon units
R_TRUNC = 10.0                   # truncation radius in scale lengths
DEV = "cuda"
KEY_BITS = 63


def listed():
    return [
        # A member of an ensemble, or a first try: every launch and call counts.
        dict(name="eval_4k", kind="eval", n=4096, theta=0.75, eps=0.01, ncrit=64, pack=0, host=False, learned=False,
             merger=False),
        # The smallest sphere of the paper's range, with packed groups of 32.
        dict(name="eval_32k", kind="eval", n=32768, theta=0.75, eps=0.002, ncrit=32, pack=1, host=False,
             learned=False, merger=False),
        # A host program's tree-code call: page-locked arrays in and out, a
        # merger of odd size, the accurate opening angle, the default groups.
        dict(name="eval_200k_host", kind="eval", n=200003, theta=0.5, eps=0.005, ncrit=64, pack=0, host=True,
             learned=False, merger=True),
        # An evaluation with the learned correction, judged by its direct sum.
        dict(name="eval_1m_learned", kind="eval", n=1 << 20, theta=1.0, eps=0.002, ncrit=64, pack=0, host=False,
             learned=True, merger=False),
        # Time stepping: an ordinary odd size, the benchmark's sphere and the
        # largest sphere of the repository's sweep.
        dict(name="step_100k", kind="step", n=100003, theta=0.75, eps=0.005, ncrit=32, pack=1, merger=False),
        dict(name="step_1m", kind="step", n=1 << 20, theta=0.75, eps=0.005, ncrit=32, pack=1, merger=False),
        dict(name="step_16m", kind="step", n=1 << 24, theta=0.75, eps=0.002, ncrit=32, pack=1, merger=False),
        # 64 systems of 2^12 to 2^18 bodies stepped together.
        dict(name="ensemble_64", kind="ensemble", nsys=64, lo_log2=12.0, span_log2=6.0, theta=0.75, eps=0.01,
             ncrit=32, pack=1),
        # Block time steps: 8 substeps, the benchmark's sphere.
        dict(name="block_1m", kind="block", n=1 << 20, theta=0.75, eps=0.005, ncrit=32, pack=1, max_level=3, eta=0.4,
             rebuild=1),
        # SPH density with about 48 neighbours per body.
        dict(name="sph_1m", kind="sph", n=1 << 20, neighbours=48, ncrit=32, pack=1),
        # The network's training: 16 snapshots' samples, one epoch.
        dict(name="train_64k", kind="train", n=65536, batch=4096, epochs=1),
        # Keys of a latency-critical caller that must not allocate.
        dict(name="sort_64k", kind="sort", n=65536),
    ]


def _size(rng, lo, hi):
    """Log-uniform, odd half of the time."""
    n = int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))
    return min(hi, n | 1) if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "step", "step", "ensemble", "block", "sph", "train", "sort"])
    ncrit, pack = rng.choice([(64, 0), (32, 1), (32, 0), (16, 0)])
    eps = rng.choice([0.002, 0.005, 0.01])
    if kind == "eval":
        lrn = rng.random() < 0.25
        return dict(kind=kind, n=_size(rng, 4096, 1 << 20 if lrn else 1 << 18),
                    theta=1.0 if lrn else rng.choice([0.5, 0.75, 1.0]), eps=eps, ncrit=64 if lrn else ncrit,
                    pack=0 if lrn else pack, host=rng.random() < 0.4, learned=lrn, merger=rng.random() < 0.4)
    if kind == "step":
        theta = rng.choice([0.5, 0.75, 1.0])
        return dict(kind=kind, n=_size(rng, 1 << 15, 1 << 24 if theta > 0.7 and ncrit == 32 else 1 << 22),
                    theta=theta, eps=eps, ncrit=ncrit, pack=pack, merger=rng.random() < 0.4)
    if kind == "ensemble":
        return dict(kind=kind, nsys=rng.randint(2, 64), lo_log2=12.0, span_log2=rng.uniform(1.0, 6.0), theta=0.75,
                    eps=eps, ncrit=ncrit, pack=pack)
    if kind == "block":
        return dict(kind=kind, n=_size(rng, 1 << 15, 1 << 20), theta=0.75, eps=0.005, ncrit=32, pack=rng.randint(0, 1),
                    max_level=rng.randint(1, 3), eta=rng.choice([0.2, 0.4]), rebuild=rng.choice([1, 1, 4]))
    if kind == "sph":
        return dict(kind=kind, n=_size(rng, 1 << 14, 1 << 20), neighbours=rng.randint(32, 64), ncrit=ncrit, pack=pack)
    if kind == "train":
        return dict(kind=kind, n=_size(rng, 8192, 1 << 17), batch=rng.choice([2048, 4096, 8192]), epochs=1)
    return dict(kind=kind, n=_size(rng, 1024, 65536))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _uniform(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _isotropic(g, n):
    c, p = _uniform(g, n, -1.0, 1.0), _uniform(g, n, 0.0, 2.0 * math.pi)
    s = torch.sqrt((1.0 - c * c).clamp_min(0.0))
    return torch.stack([s * torch.cos(p), s * torch.sin(p), c], 1)


def _sphere(g, n):
    """Positions and velocities (float64) of a truncated Plummer sphere of unit mass."""
    f = (R_TRUNC / math.sqrt(R_TRUNC * R_TRUNC + 1.0)) ** 3
    u = _uniform(g, n, 0.0, f).clamp_min(1e-300)
    r = A_HENON / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
    pos = _isotropic(g, n) * r[:, None]
    q = torch.zeros(n, device=DEV, dtype=torch.float64)
    todo = torch.arange(n, device=DEV)
    while todo.numel():              # von Neumann rejection on q^2 (1 - q^2)^(7/2)
        x1, x2 = _uniform(g, todo.numel()), _uniform(g, todo.numel(), 0.0, 0.1)
        ok = x2 < x1 * x1 * (1.0 - x1 * x1) ** 3.5
        q[todo[ok]] = x1[ok]
        todo = todo[~ok]
    vesc = math.sqrt(2.0) * (r * r + A_HENON * A_HENON) ** -0.25
    vel = _isotropic(g, n) * (q * vesc)[:, None]
    return pos - pos.mean(0), vel - vel.mean(0)


def _bodies(g, n, merger):
    """float32 positions, masses and velocities on the GPU."""
    if not merger:
        pos, vel = _sphere(g, n)
        mass = torch.full((n,), 1.0 / n, device=DEV)
    else:                            # two unit spheres at x = +-2, approaching at 0.5
        h = n // 2
        (p1, v1), (p2, v2) = _sphere(g, h), _sphere(g, n - h)
        p1[:, 0] += 2.0
        v1[:, 0] -= 0.25
        p2[:, 0] -= 2.0
        v2[:, 0] += 0.25
        pos, vel = torch.cat([p1, p2]), torch.cat([v1, v2])
        mass = torch.cat([torch.full((h,), 1.0 / h, device=DEV), torch.full((n - h,), 1.0 / (n - h), device=DEV)])
    return pos.float().contiguous(), mass, vel.float().contiguous()


def _sizes(case):
    """Sizes of an ensemble's systems: fixed by the case (log-uniform, evenly spread)."""
    k = case["nsys"]
    return [int(round(2.0 ** (case["lo_log2"] + case["span_log2"] * ((i * 0.6180339887498949) % 1.0)))) for i in range(k)]


def _smoothing(pos, n, neighbours):
    """Smoothing lengths for about `neighbours` bodies from the Plummer density at each radius."""
    r2 = pos.double().square().sum(1) / (A_HENON * A_HENON)
    density = n * 3.0 / (4.0 * math.pi * A_HENON ** 3) * (1.0 + r2) ** -2.5
    return ((3.0 * neighbours / (4.0 * math.pi * density)) ** (1.0 / 3.0)).float()


def _network(seed):
    """Weights and normalisation of a correction of about a hundredth of the force."""
    rng = np.random.default_rng(seed)
    h, i, o = B.MLP_H, B.MLP_IN, B.MLP_OUT
    parts = [rng.normal(0, math.sqrt(2 / i), h * i), rng.normal(0, 0.1, h), rng.normal(0, math.sqrt(2 / h), h * h),
             rng.normal(0, 0.1, h), rng.normal(0, 0.3 * math.sqrt(2 / h), o * h), np.zeros(o)]
    mu = [0.0, 0.0, 2.0, 3.5, 5.0, 5.5, 5.5, 8.0, 3.0, 0.7, 0.0, 3.0]
    sigma = [1.0, 0.5, 1.0, 1.0, 1.0, 1.5, 0.5, 3.0, 1.0, 0.3, 0.6, 0.6]
    return np.concatenate(parts).astype(np.float32), np.array(mu + sigma + [5e-3], np.float32)


def _rows(case, seed):
    """Feature rows and targets with the scales that the walk's samples have."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    X = rng.normal(size=(n, B.MLP_IN))
    Y = np.stack([np.tanh(X[:, 0] + 0.5 * X[:, 3]), 0.5 * X[:, 9] * X[:, 10], 0.1 * X[:, 1]], 1)
    Y += rng.normal(scale=0.7, size=Y.shape)
    mu = np.array([0.0, 0.0, 2.0, 3.5, 5.0, 5.5, 5.5, 8.0, 3.0, 0.7, 0.0, 3.0])
    return (X * 0.8 + mu).astype(np.float32), (Y * 5e-3).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, Y = _rows(case, seed)
        return dict(case=case, X=X, Y=Y)
    if kind == "sort":
        n = case["n"]
        keys = torch.randint(0, 1 << KEY_BITS - 1, (n,), generator=_gen(seed), device=DEV, dtype=torch.int64)
        keys = (keys >> 6) << 7      # nearby bodies share their upper bits; the lowest come out equal
        return dict(case=case, keys=keys, out=torch.empty_like(keys),
                    perm=torch.empty(n, dtype=torch.int32, device=DEV))
    g = _gen(seed)
    bz = B.Bonsai(B.Config(ncrit=case["ncrit"], group_pack=case["pack"]))
    s = dict(case=case, bz=bz)
    if kind == "ensemble":
        sizes = _sizes(case)
        systems = [_bodies(g, k, False) for k in sizes]
        pos, mass, vel = (torch.cat([b[j] for b in systems]).contiguous() for j in range(3))
        bz.set_bodies(pos, mass, vel).set_systems(np.cumsum([0] + sizes))
        n = int(mass.numel())
    else:
        n = case["n"]
        pos, mass, vel = _bodies(g, n, case.get("merger", False))
    if kind == "eval":
        where = dict(device="cpu", pin_memory=True) if case["host"] else dict(device=DEV)
        if case["host"]:
            pos, mass, vel = (t.cpu().pin_memory() for t in (pos, mass, vel))
        s.update(pos=pos, mass=mass, vel=vel, acc=torch.empty(n, 3, **where), pot=torch.empty(n, **where))
        if case["learned"]:
            s["net"] = B.MLP(0)
            s["net"].set_params(*_network(seed))
            B.bonsai_set_learned(bz.ctx, s["net"], case["theta"], 0.5, 1.0)
        return s
    if kind == "sph":
        bz.set_bodies(pos, mass, vel).build()
        s.update(h=_smoothing(pos, n, case["neighbours"]), rho=torch.empty(n, device=DEV),
                 count=torch.empty(n, dtype=torch.int32, device=DEV))
        return s
    if kind != "ensemble":
        bz.set_bodies(pos, mass, vel)
    B.bonsai_set_params(bz.ctx, case["theta"], case["eps"])
    s.update(pos=torch.empty(n, 3, device=DEV), vel=torch.empty(n, 3, device=DEV))
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

DT = 1.0 / 256.0        # shared step
DT_MAX = 1.0 / 16.0     # cycle of block time steps


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "train":
        net, losses = L.train(s["X"], s["Y"], epochs=case["epochs"], batch=case["batch"], lr=2e-3, wd=1e-4, seed=0)
        params, norm = net.get_params()
        return dict(params=params, norm=norm, losses=losses)
    if kind == "sort":
        B.bonsai_sort_keys_static(s["keys"], s["out"], s["perm"])
        return dict(keys=s["out"], perm=s["perm"])
    bz = s["bz"]
    if kind == "eval":
        bz.set_bodies(s["pos"], s["mass"], s["vel"]).build().multipoles()
        if case["learned"]:
            B.bonsai_forces_learned(bz.ctx, case["eps"], s["acc"], s["pot"])
        else:
            bz.forces(case["theta"], case["eps"], s["acc"], s["pot"])
        return dict(acc=s["acc"], pot=s["pot"])
    if kind == "sph":
        B.bonsai_sph_density(bz.ctx, s["h"], s["rho"], s["count"])
        return dict(rho=s["rho"], count=s["count"])
    if kind == "block":
        bz.block_cycle(DT_MAX, case["max_level"], case["eta"], case["rebuild"])
    else:
        bz.step(DT)
    B.bonsai_get_bodies(bz.ctx, s["pos"], s["vel"])
    return dict(pos=s["pos"], vel=s["vel"])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _walk_flops(n, theta):
    """65 flops per body-cell and 23 per body-body interaction; the counts per
    body as measured on Plummer spheres (theta 0.5, 0.75, 1.0)."""
    pc, pp = {0.5: (2.4, 2.3), 0.75: (1.0, 1.0), 1.0: (0.63, 0.8)}[case_theta(theta)]
    return n * (65.0 * pc * max(300.0, 727.0 + 37.0 * (math.log2(n) - 15.0)) + 23.0 * pp * 415.0)


def case_theta(theta):
    return min((0.5, 0.75, 1.0), key=lambda t: abs(t - theta))


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "eval":
        flops = _walk_flops(n, case["theta"])
        if case["learned"]:          # the network and the judge's direct sum
            flops += n * 2.0 * (B.MLP_IN * B.MLP_H + B.MLP_H * B.MLP_H + B.MLP_H * B.MLP_OUT) + 23.0 * min(n, 4096) * n
        return dict(bytes=n * 44.0, flops=flops)
    if kind == "step":               # state in (position, mass, velocity, acceleration), state out, caller-order copy
        return dict(bytes=n * (44.0 + 44.0 + 24.0), flops=_walk_flops(n, case["theta"]))
    if kind == "ensemble":
        return dict(bytes=sum(_sizes(case)) * 112.0, flops=sum(_walk_flops(k, case["theta"]) for k in _sizes(case)))
    if kind == "block":              # about two walks of every body per cycle (eta 0.4), half the steps at most
        steps = 1 << case["max_level"]
        share = 0.37 if case["eta"] > 0.3 else 0.73
        return dict(bytes=n * 112.0, flops=max(1.0, share * steps) * _walk_flops(n, case["theta"]))
    if kind == "sph":                # 20 flops per neighbour
        return dict(bytes=n * (16.0 + 4.0 + 8.0), flops=n * 20.0 * case["neighbours"])
    if kind == "train":
        rows = float(n) * case["epochs"]
        return dict(bytes=rows * 4.0 * (B.MLP_IN + B.MLP_OUT) + 8.0 * B.MLP_NPARAM, flops=rows * 6.0 * B.MLP_NPARAM)
    return dict(bytes=n * (8.0 + 8.0 + 4.0), flops=0.0)


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _direct(pos, mass, eps, targets):
    x, m = pos.double(), mass.double()
    acc = torch.empty(targets.shape[0], 3, device=DEV, dtype=torch.float64)
    pot = torch.empty(targets.shape[0], device=DEV, dtype=torch.float64)
    rows = max(1, (1 << 27) // x.shape[0])
    for a in range(0, targets.shape[0], rows):
        t = targets[a:a + rows]
        y = x[t]
        d = [x[None, :, k] - y[:, None, k] for k in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps
        w = m[None, :] * torch.rsqrt(r2)
        w[torch.arange(t.shape[0], device=DEV), t] = 0.0
        pot[a:a + rows] = -w.sum(1)
        w /= r2
        for k in range(3):
            acc[a:a + rows, k] = (w * d[k]).sum(1)
    return acc, pot


def _density(pos, mass, h):
    x, m = pos.double(), mass.double()
    n = x.shape[0]
    rho = torch.empty(n, device=DEV, dtype=torch.float64)
    rows = max(1, (1 << 27) // n)
    for a in range(0, n, rows):
        y, hh = x[a:a + rows], h[a:a + rows].double()
        q = torch.zeros(y.shape[0], n, device=DEV, dtype=torch.float64)
        for k in range(3):
            q += (x[None, :, k] - y[:, None, k]).square()
        q = torch.sqrt(q) / hh[:, None]
        w = torch.where(q <= 0.5, 1.0 - 6.0 * q * q + 6.0 * q * q * q, 2.0 * (1.0 - q).clamp_min(0.0) ** 3)
        rho[a:a + rows] = (m[None, :] * w).sum(1) * 8.0 / math.pi / hh ** 3
    return rho


class _Xorshift:
    """xorshift64*, as the network's documented initialisation and shuffles use it."""

    MASK = (1 << 64) - 1

    def __init__(self, seed):
        self.s = (seed * 0x9E3779B97F4A7C15 + 0x2545F4914F6CDD1D) & self.MASK or 1

    def next(self):
        s = self.s
        s ^= s >> 12
        s = (s ^ (s << 25)) & self.MASK
        s ^= s >> 27
        self.s = s
        return (s * 0x2545F4914F6CDD1D) & self.MASK

    def uniform(self):
        return (self.next() >> 11) / 9007199254740992.0

    def normal(self):
        u1, u2 = self.uniform(), self.uniform()
        return math.sqrt(-2.0 * math.log(max(u1, 1e-300))) * math.cos(2.0 * math.pi * u2)


def _bf16(x):
    return x.float().bfloat16().double()


def _train_exact(case, X, Y):
    """Forward and backward in float64 on the bfloat16-rounded inputs, weights and activations, AdamW in float64."""
    X, Y = torch.from_numpy(X).to(DEV).double(), torch.from_numpy(Y).to(DEV).double()
    n, batch = case["n"], case["batch"]
    mu = X.mean(0)
    sigma = (X.square().mean(0) - mu * mu).clamp_min(0.0).sqrt().clamp_min(1e-6)
    ysig = Y.square().mean().sqrt().clamp_min(1e-12)
    h, i, o = B.MLP_H, B.MLP_IN, B.MLP_OUT
    rng = _Xorshift(0)
    shapes = [(h, i), (h,), (h, h), (h,), (o, h), (o,)]
    P = []
    for s in shapes:
        if len(s) == 2:
            sd = math.sqrt(2.0 / s[1])
            # the stored initial weights are float32
            w = np.array([sd * rng.normal() for _ in range(s[0] * s[1])]).astype(np.float32).reshape(s)
            P.append(torch.from_numpy(w).to(DEV).double())
        else:
            P.append(torch.zeros(s, device=DEV, dtype=torch.float64))
    M, V = [torch.zeros_like(p) for p in P], [torch.zeros_like(p) for p in P]
    rng = _Xorshift(0)
    perm = list(range(n))
    Xn, Yn = _bf16((X - mu) / sigma), Y / ysig
    step, losses = 0, []
    for _ in range(case["epochs"]):
        for k in range(n - 1, 0, -1):
            j = rng.next() % (k + 1)
            perm[k], perm[j] = perm[j], perm[k]
        order = torch.tensor(perm, device=DEV)
        total, count = 0.0, 0
        for a in range(0, n, batch):
            t = order[a:a + batch]
            x, y = Xn[t], Yn[t]
            W1, W2, W3 = _bf16(P[0]), _bf16(P[2]), _bf16(P[4])
            h1 = _bf16((x @ W1.T + P[1]).clamp_min(0.0))
            h2 = _bf16((h1 @ W2.T + P[3]).clamp_min(0.0))
            r = h2 @ W3.T + P[5] - y
            total += float(r.square().mean())
            count += 1
            dy = r * (2.0 / r.numel())
            dh2 = (dy @ W3) * (h2 > 0)
            dh1 = (dh2 @ W2) * (h1 > 0)
            G = [dh1.T @ x, dh1.sum(0), dh2.T @ h1, dh2.sum(0), dy.T @ h2, dy.sum(0)]
            step += 1
            for p, g, m, v in zip(P, G, M, V):
                m.mul_(0.9).add_(g, alpha=0.1)
                v.mul_(0.999).add_(g * g, alpha=0.001)
                u = (m / (1.0 - 0.9 ** step)) / ((v / (1.0 - 0.999 ** step)).sqrt() + 1e-8)
                p.sub_(2e-3 * (u + (1e-4 * p if p.dim() == 2 else 0.0)))
        losses.append(total / count)
    return dict(params=torch.cat([p.reshape(-1) for p in P]), norm=torch.cat([mu, sigma, ysig.reshape(1)]),
                losses=torch.tensor(losses, dtype=torch.float64))


def exact(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "train":
        return _train_exact(case, *_rows(case, seed))
    if n > 1 << 18 or kind not in ("eval", "sph") or case.get("learned"):
        return None          # O(n^2) over about 20 s, whole numbers, or an outcome of many evaluations
    pos, mass, _ = _bodies(_gen(seed), n, case.get("merger", False))
    if kind == "sph":
        return dict(rho=_density(pos, mass, _smoothing(pos, n, case["neighbours"])), count=None)
    acc, pot = _direct(pos, mass, case["eps"], torch.arange(n, device=DEV))
    return dict(acc=acc, pot=pot)
