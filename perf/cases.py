"""The work a user of this framework has it do, as measurable cases.

Every case goes through the public binding (`ptadd.Context`) as the drivers
of the package do: load a network, a batch or a surrogate once, then per pass
put the start state in, run the call, and take its results out.  The bursts
use the well-conditioned step dt = 5e-13 s, at which two runs that round
differently stay together.

`exact` restates the mathematics in plain torch in 64 bits.
"""

import math

import numpy as np
import torch

from paper_2005_02498_gb300 import ptadd
from paper_2005_02498_gb300 import workloads as W

MAT = W.Material()
DT = 5e-13
FLOP_PER_PAIR = 679.0  # 4 field points of one source on one target segment, with the force
PREC = {"fp64": ptadd.PTADD_FP64, "mixed": ptadd.PTADD_MIXED}
DIMS = ((30, 256), (256, 256), (256, 256), (256, 6))
MLP_FLOP = 2.0 * sum(i * o for i, o in DIMS)
MLP_PARAMS = sum(i * o + o for i, o in DIMS)
CAPTURE = dict(capture_radius=10e-9, max_break_time=1e-3, stuck_disp=1e-2 * W.BURGERS)
LOOPS_PER_UM3 = 16.0


# ------------------------------------------------------------------- cases
def listed():
    return [
        # one loop pair, the smallest box that moves: every DD step is launches and latency
        dict(name="burst_42_fp64", kind="burst", loops=2, nodes=21, ragged=0, pinned=0.0, precision="fp64", steps=20,
             consistent=False),
        # the PTA driver's default box (16 loops of 32 segments in 1 um^3), one chunk of its running average
        dict(name="burst_512_fp64", kind="burst", loops=16, nodes=32, ragged=0, pinned=0.0, precision="fp64",
             steps=20, consistent=False),
        # the junction-controlled microstructure of the single-box loop: most loops sessile, few mobile
        dict(name="junctions_1280_fp64", kind="junctions", loops=40, precision="fp64", steps=20),
        # loops of uneven node counts, some sessile, with the consistent mass matrix of the Galerkin mobility
        dict(name="burst_ragged_consistent", kind="burst", loops=53, nodes=27, ragged=18, pinned=0.3,
             precision="fp64", steps=10, consistent=True),
        # an ordinary mixed-precision burst
        dict(name="burst_8192_mixed", kind="burst", loops=256, nodes=32, ragged=0, pinned=0.0, precision="mixed",
             steps=10, consistent=False),
        # the large realisation of the headline benchmark, in mixed precision
        dict(name="burst_32768_mixed", kind="burst", loops=1024, nodes=32, ragged=0, pinned=0.0, precision="mixed",
             steps=2, consistent=False),
        # its plain FP64 force evaluation, left on the device
        dict(name="forces_32768_fp64", kind="forces", loops=1024, nodes=32, precision="fp64"),
        # realisations of 1k to 16k segments advanced together: surrogate labels, closure fallbacks
        dict(name="batch_32_mixed", kind="batch", R=32, n_min=1024, n_max=16384, precision="mixed", steps=2),
        # the block driver's boxes: a few small FP64 realisations in lock step
        dict(name="batch_9x512_fp64", kind="batch", R=9, n_min=512, n_max=512, precision="fp64", steps=10),
        # the surrogate over a million material points held on the device
        dict(name="predict_1m", kind="predict", n=1000000, host=False),
        # one load step of a 16^3 mesoscale grid, from and to host arrays
        dict(name="predict_4096_host", kind="predict", n=4096, host=True),
        # two epochs of surrogate training at the default minibatch
        dict(name="train_8192", kind="train", n=8192, batch=512, epochs=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["burst", "burst", "burst", "junctions", "forces", "batch", "batch", "predict", "predict", "train"])
    if kind == "burst":
        precision = rng.choice(["fp64", "mixed"])
        nodes = rng.randint(12, 48)
        # mixed precision is for boxes whose far field dominates
        segments = _log_int(rng, 40, 6000) if precision == "fp64" else _log_int(rng, 4000, 24000)
        steps = rng.randint(2, 20)
        return dict(kind=kind, loops=max(2, segments // nodes), nodes=nodes, ragged=rng.choice([0, nodes // 2]),
                    pinned=rng.choice([0.0, round(rng.uniform(0.1, 0.6), 2)]), precision=precision,
                    steps=steps if segments < 3000 else 2 + steps // 8,
                    consistent=rng.random() < 0.3)
    if kind == "junctions":
        return dict(kind=kind, loops=rng.randint(16, 64), precision="fp64", steps=rng.randint(4, 20))
    if kind == "forces":
        nodes = rng.randint(12, 48)
        return dict(kind=kind, loops=max(2, _log_int(rng, 600, 24000) // nodes), nodes=nodes, precision="fp64")
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind=kind, R=rng.randint(2, 32), n_min=1024, n_max=_log_int(rng, 4000, 16384),
                        precision="mixed", steps=rng.randint(1, 3))
        n = rng.randint(200, 3000)
        return dict(kind=kind, R=rng.randint(2, 16), n_min=n, n_max=n + rng.randint(0, n), precision="fp64",
                    steps=rng.randint(1, 5))
    if kind == "predict":
        host = rng.random() < 0.4
        return dict(kind=kind, n=_log_int(rng, 100, 60000) if host else _log_int(rng, 1000, 1000000), host=host)
    return dict(kind=kind, n=rng.randint(1200, 8192), batch=16 * rng.randint(8, 64), epochs=rng.randint(1, 2))


# ------------------------------------------------------------------ inputs
def _ring(rng, m, edge):
    """One circular glide loop of m nodes (radius, centre, phase, sense and slip system drawn)."""
    bh, nh = W.fcc_slip_systems()
    s = int(rng.integers(12))
    r = rng.uniform(0.05, 0.2) * W.MICRON
    c = rng.uniform(0.0, edge, size=3)
    phi = rng.uniform(0.0, 2.0 * math.pi) + rng.choice([-1.0, 1.0]) * 2.0 * math.pi / m * np.arange(m)
    e1, e2 = bh[s], np.cross(nh[s], bh[s])
    return c + r * (np.cos(phi)[:, None] * e1 + np.sin(phi)[:, None] * e2), W.BURGERS * e1, nh[s]


def _sizes(case):
    """Numbers drawn for a case's sizes: they belong to the case, so inputs of another seed have the same shapes."""
    return np.random.default_rng([int(case[k]) for k in sorted(case) if isinstance(case[k], int)])


def _network(case, seed):
    rng = np.random.default_rng([seed, 2005])
    if case["kind"] == "junctions":
        return W.junction_microstructure(seed, W.uniaxial_stress(100e6), 1e13, 2e14, n_loops=case["loops"])
    loops, nodes, ragged = case["loops"], case["nodes"], case.get("ragged", 0)
    edge = (loops / LOOPS_PER_UM3) ** (1.0 / 3.0) * W.MICRON
    if loops == 1024:
        edge = W.LARGE_LOOPS["box_edge"]
    counts = nodes + (_sizes(case).integers(-ragged, ragged + 1, size=loops) if ragged else np.zeros(loops, np.int64))
    counts = np.maximum(counts, 5)
    rings = [_ring(rng, int(m), edge) for m in counts]
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    pin = np.zeros(int(off[-1]), np.uint8)
    for k in range(loops):
        if rng.random() < case.get("pinned", 0.0):
            pin[off[k]:off[k + 1]] = 1
    if case.get("pinned"):
        pin[off[0]:off[1]] = 0  # something moves
        pin[off[0]] = 1         # and one loop is held at a node
    sig = rng.uniform(-100e6, 100e6, size=6) if case["kind"] == "burst" and loops < 1024 else W.uniaxial_stress(50e6)
    return W.Network(np.ascontiguousarray(np.concatenate([r[0] for r in rings])), off,
                     np.ascontiguousarray([r[1] for r in rings]), np.ascontiguousarray([r[2] for r in rings]), pin,
                     edge ** 3, sig)


def _batch(case, seed):
    """The batched ensemble's recipe: uneven realisations at 16 loops per um^3, a stress of +-200 MPa and a
    sessile share of 0.1 to 0.9 (whole loops) for each."""
    rng, nets = np.random.default_rng([seed, 1003]), []
    for n in _sizes(case).integers(case["n_min"], case["n_max"] + 1, size=case["R"]):
        loops = max(2, int(round(n / 32)))
        edge = (loops / LOOPS_PER_UM3) ** (1.0 / 3.0) * W.MICRON
        xyz, off, bv, nv = W.circular_loops(rng, loops, edge)
        held = np.arange(loops) < min(loops - 1, int(round(loops * rng.uniform(0.1, 0.9))))
        nets.append(W.Network(xyz, off, bv, nv, np.repeat(rng.permutation(held), 32).astype(np.uint8), edge ** 3,
                              rng.uniform(-200e6, 200e6, size=6)))
    return W.batch_from_networks(nets)


def _closure_inputs(gen, n):
    """Raw closure features [n, 30] on the GPU: stresses of +-200 MPa, densities of 1e11 .. 2e13 per class."""
    u = torch.rand((n, 30), generator=gen, device="cuda", dtype=torch.float64)
    f = torch.empty_like(u)
    f[:, :6] = (2.0 * u[:, :6] - 1.0) * 200e6
    f[:, 6:] = 10.0 ** (11.0 + 2.3 * u[:, 6:])
    return f


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _weights(seed):
    rng = np.random.default_rng([seed, 256])
    parts = []
    for i, o in DIMS:
        parts.append(rng.uniform(-1.0, 1.0, size=i * o) * math.sqrt(6.0 / (i + o)))
        parts.append(rng.normal(0.0, 0.05, size=o))
    return np.concatenate(parts).astype(np.float32)


def _closures(gen, n):
    """Closure features and smooth rate labels of the size that DD gives (1e4 .. 1e6 per second)."""
    f = _closure_inputs(gen, n)
    s = f[:, :6] / 200e6
    m = f[:, 6:18].sum(1, keepdim=True) / 1e13
    return f, 1e5 * torch.tanh(2.0 * s) * m + 2e4 * s.roll(1, 1) * s


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("burst", "junctions", "forces"):
        net = _network(case, seed)
        ctx = ptadd.Context(MAT.as_tuple(), PREC[case["precision"]], 0)
        ctx.set_network(net)
        state = dict(kind=kind, case=case, ctx=ctx, x0=net.xyz)
        if kind == "burst":
            ctx.set_mobility(case["consistent"])
        elif kind == "junctions":
            ctx.set_junctions(seed=seed, **CAPTURE)
            state["blob"] = ctx.get_state()
        else:
            state["F"] = torch.empty((net.n_nodes, 3), dtype=torch.float64, device="cuda")
        return state
    if kind == "batch":
        batch = _batch(case, seed)
        ctx = ptadd.Context(MAT.as_tuple(), PREC[case["precision"]], 0)
        ctx.batch_set(batch)
        return dict(kind=kind, case=case, ctx=ctx, x0=batch.xyz)
    ctx = ptadd.Context(MAT.as_tuple(), ptadd.PTADD_MIXED, 0)
    if kind == "predict":
        f, y = _closures(_gen(seed), 4096)
        ctx.surrogate_fit(f.cpu().numpy(), y.cpu().numpy(), epochs=0, seed=seed)  # the maps and the trust region
        ctx.mlp_set_params(_weights(seed))
        q = _closure_inputs(_gen(seed + 1), case["n"])
        state = dict(kind=kind, case=case, ctx=ctx)
        if case["host"]:
            state["feat"] = q.cpu().numpy()
        else:
            state.update(feat=q, lp6=torch.empty((case["n"], 6), dtype=torch.float64, device="cuda"),
                         inside=torch.empty(case["n"], dtype=torch.uint8, device="cuda"))
            torch.cuda.synchronize()
        return state
    x, y, p = _training(case, seed)
    return dict(kind=kind, case=case, ctx=ctx, x=x, y=y, p=p, seed=seed)


def _training(case, seed):
    f, y = _closures(_gen(seed), case["n"])
    x = torch.cat([f[:, :6] / 200e6, torch.log10(f[:, 6:] + 1e10)], 1)
    x = (x - x.mean(0)) / x.std(0)
    y = (y - y.mean(0)) / y.std(0)
    return x.float().cpu().numpy(), y.float().cpu().numpy(), _weights(seed)


# -------------------------------------------------------------------- pass
def run(state):
    kind, case, ctx = state["kind"], state["case"], state["ctx"]
    if kind == "burst":
        ctx.set_nodes(state["x0"])
        Lp, rho = ctx.advance(case["steps"], DT)
        return dict(Lp=Lp, rho=rho, nodes=ctx.get_nodes())
    if kind == "junctions":
        ctx.set_state(state["blob"])
        Lp, rho = ctx.advance(case["steps"], DT)
        j = ctx.junctions()
        return dict(Lp=Lp, rho=rho, nodes=ctx.get_nodes(), held=j["seg"], count=j["count"], break_time=j["break_time"],
                    clock=j["clock"])
    if kind == "forces":
        ctx.set_nodes(state["x0"])
        ctx.get_forces_dev(state["F"].data_ptr())
        return state["F"]
    if kind == "batch":
        ctx.batch_set_nodes(state["x0"])
        Lp, rho = ctx.batch_advance(case["steps"], DT)
        return dict(Lp=Lp, rho=rho, nodes=ctx.batch_get_nodes())
    if kind == "predict":
        if case["host"]:
            lp6, inside = ctx.surrogate_predict(state["feat"])
            return dict(lp6=lp6, inside=inside)
        ctx.surrogate_predict_dev(case["n"], state["feat"].data_ptr(), state["lp6"].data_ptr(),
                                  state["inside"].data_ptr())
        return dict(lp6=state["lp6"], inside=state["inside"])
    ctx.mlp_set_params(state["p"])
    losses = ctx.mlp_train(state["x"], state["y"], epochs=case["epochs"], batch=case["batch"], seed=state["seed"])
    return dict(losses=losses, params=ctx.mlp_get_params())


# -------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind in ("burst", "forces", "junctions"):
        n = case["loops"] * case.get("nodes", 32)
        free = 1.0 - case.get("pinned", 0.0)
        if kind == "junctions":
            free = 0.05  # the mobile share of the recipe's densities
        return dict(bytes=48.0 * n, flops=FLOP_PER_PAIR * free * n * n * case.get("steps", 1))
    if kind == "batch":
        a, b = float(case["n_min"]), float(case["n_max"])
        mean, square = 0.5 * (a + b), (a * a + a * b + b * b) / 3.0
        return dict(bytes=48.0 * case["R"] * mean, flops=FLOP_PER_PAIR * 0.5 * case["R"] * square * case["steps"])
    if kind == "predict":
        return dict(bytes=289.0 * case["n"], flops=MLP_FLOP * case["n"])
    samples = float(case["n"] // case["batch"] * case["batch"] * case["epochs"])
    return dict(bytes=144.0 * case["n"] + 8.0 * MLP_PARAMS, flops=3.0 * MLP_FLOP * samples)


# ------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    if kind in ("burst", "forces"):
        net = _network(case, seed)
        if kind == "forces":
            return _Box(net).forces()[0]
        return _exact_burst(net, case["steps"], case["consistent"])
    if kind == "junctions":
        return None  # the captures are decisions, not numbers
    if kind == "batch":
        b = _batch(case, seed)
        one = [_exact_burst(b.realisation(r), case["steps"], False) for r in range(b.R)]
        return dict(Lp=np.stack([o["Lp"] for o in one]), rho=np.array([o["rho"] for o in one]),
                    nodes=np.concatenate([o["nodes"] for o in one]))
    if kind == "predict":
        f, y = _closures(_gen(seed), 4096)
        x = _features(f)
        xm, xs, ym, ys = x.mean(0), x.std(0, unbiased=False), y.mean(0), y.std(0, unbiased=False)
        z = (_features(_closure_inputs(_gen(seed + 1), case["n"])) - xm) / xs
        return dict(lp6=_mlp(_layers(_weights(seed)), z)[-1] * ys + ym, inside=None)
    return _exact_training(case, seed)


def _features(f):
    return torch.cat([f[:, :6] / 200e6, torch.log10(f[:, 6:] + 1e10)], 1)


def _layers(p):
    p, out, at = torch.from_numpy(p).double().cuda(), [], 0
    for i, o in DIMS:
        out.append((p[at:at + i * o].reshape(o, i).clone(), p[at + i * o:at + i * o + o].clone()))
        at += i * o + o
    return out


def _mlp(layers, x):
    h = [x]
    for k, (w, b) in enumerate(layers):
        z = h[-1] @ w.T + b
        h.append(torch.nn.functional.gelu(z) if k < 3 else z)
    return h


def _splitmix64(s):
    s = (s + 0x9E3779B97F4A7C15) & 0xFFFFFFFFFFFFFFFF
    z = ((s ^ (s >> 30)) * 0xBF58476D1CE4E5B9) & 0xFFFFFFFFFFFFFFFF
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & 0xFFFFFFFFFFFFFFFF
    return s, z ^ (z >> 31)


def _exact_training(case, seed):
    x, y, p = _training(case, seed)
    x, y = torch.from_numpy(x).double().cuda(), torch.from_numpy(y).double().cuda()
    n, batch = case["n"], case["batch"]
    params = [t.requires_grad_() for layer in _layers(p) for t in layer]
    opt = torch.optim.Adam(params, lr=1e-3, betas=(0.9, 0.999), eps=1e-8)
    perm, s, losses = list(range(n)), int(seed), []
    for _ in range(case["epochs"]):
        for i in range(n - 1, 0, -1):
            s, r = _splitmix64(s)
            j = r % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        order, total = torch.tensor(perm, device="cuda"), 0.0
        for b in range(n // batch):
            at = order[b * batch:(b + 1) * batch]
            loss = ((_mlp(list(zip(params[::2], params[1::2])), x[at])[-1] - y[at]) ** 2).mean()
            opt.zero_grad()
            loss.backward()
            opt.step()
            total += float(loss)
        losses.append(total / (n // batch))
    return dict(losses=np.array(losses), params=torch.cat([t.detach().reshape(-1) for t in params]))


def _cross(a, b):
    return (a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0])


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


class _Box:
    """Forces and glide velocities of one network in plain torch, 64 bits; lengths in units of a power of two
    near |b|, stresses in mu, so that the scaling is exact."""

    def __init__(self, net):
        d = dict(dtype=torch.float64, device="cuda")
        self.unit = 2.0 ** round(math.log2(MAT.b))
        self.x = torch.tensor(net.xyz, **d) / self.unit
        counts = np.diff(net.loop_off)
        ids = np.arange(net.n_nodes)
        self.nxt = torch.tensor(np.concatenate([np.roll(ids[a:b], -1) for a, b in zip(net.loop_off, net.loop_off[1:])]),
                                device="cuda")
        self.prv = torch.tensor(np.concatenate([np.roll(ids[a:b], 1) for a, b in zip(net.loop_off, net.loop_off[1:])]),
                                device="cuda")
        self.b = torch.tensor(np.repeat(net.burgers, counts, 0), **d) / self.unit
        self.n = torch.tensor(np.repeat(net.normal, counts, 0), **d)
        self.pin = torch.tensor(net.pinned.astype(bool), device="cuda")
        s = net.sig_app / MAT.mu
        self.sig = torch.tensor([[s[0], s[5], s[4]], [s[5], s[1], s[3]], [s[4], s[3], s[2]]], **d)
        self.off, self.volume = net.loop_off, net.volume
        z = np.array([0.8611363115940526, 0.3399810435848563])
        w = np.array([0.3478548451374538, 0.6521451548625461])
        self.xi = [0.5 * (1 - z[0]), 0.5 * (1 - z[1]), 0.5 * (1 + z[1]), 0.5 * (1 + z[0])]
        self.w = [0.5 * w[0], 0.5 * w[1], 0.5 * w[1], 0.5 * w[0]]

    def stress_on(self, xq, bq):
        """(sigma b') at points xq [P, 3] with target Burgers vectors bq [P, 3], from every segment: the
        nonsingular isotropic field of a straight segment, its line integrals in closed form."""
        a2, r = (MAT.a / self.unit) ** 2, -(1.0 - MAT.nu) / 2.0
        D = self.x[self.nxt] - self.x
        L = D.norm(dim=1)
        t = tuple((D / L[:, None]).T)
        b = tuple(self.b.T)
        q = _cross(b, t)
        p = tuple(c[:, None] for c in bq.T)
        R = tuple(xq[:, k, None] - self.x[None, :, k] for k in range(3))
        y = _dot(R, t)
        Rp = tuple(R[k] - y * t[k] for k in range(3))
        del R
        d2 = _dot(Rp, Rp) + a2
        u2 = L - y
        i1, i2 = (y * y + d2).rsqrt(), (u2 * u2 + d2).rsqrt()
        m, c = -y * i1, u2 * i2
        one = (y <= 0) | (y >= L)  # both ends on one side of the foot of the perpendicular
        i12, ss, S = (i1 * i2) ** 2, i1 * i1 + i2 * i2, c * c + c * m + m * m
        Li = L * (u2 - y) * i12
        J1 = Li / (i1 + i2)
        J0 = torch.where(one, Li / (c + m), (c - m) / d2)
        K2 = J0 * torch.where(one, (y * y + u2 * u2 + d2) * i12 / (1 + c * m) + ss, (3 - S) / d2)
        K3, K4 = J1 * (i1 * i2 + ss), J0 * S
        del i12, ss, S, Li, m, c, one, d2, u2, y
        B0 = a2 * K2 + J0
        A0, C1 = B0 + J0, r * (a2 * K3 + 2 * J1) + J1
        tb, qb = _dot(t, p), _dot(q, p)
        X = _cross(Rp, b)
        Rb, qR = _dot(Rp, p), _dot(Rp, q)
        cX, cq = r * tb * A0, C1 * tb - J0 * Rb
        cR = qR * (K2 * Rb - K3 * tb) - J0 * qb
        ct = r * A0 * _dot(X, p) + C1 * qb + qR * (K4 * tb - K3 * Rb)
        sb = (qR * B0).sum(1)
        del A0, C1, K3, K4, J0, J1, K2, Rb, qR, B0, tb, qb
        c2 = 1.0 / (4.0 * math.pi * (1.0 - MAT.nu))
        return torch.stack([c2 * ((cX * X[k] + cq * q[k] + cR * Rp[k] + ct * t[k]).sum(1) + sb * bq[:, k])
                            for k in range(3)], 1)

    def forces(self, targets=None):
        """Nodal forces in N and in internal units."""
        n = self.x.shape[0]
        D = self.x[self.nxt] - self.x
        fs, fe = torch.zeros_like(self.x), torch.zeros_like(self.x)
        step = max(1, (1 << 22) // n)
        seg = torch.arange(n, device="cuda") if targets is None else targets
        for at in range(0, seg.numel(), step):
            k = seg[at:at + step]
            for xi, w in zip(self.xi, self.w):
                s = self.stress_on(self.x[k] + xi * D[k], self.b[k]) + self.b[k] @ self.sig
                f = torch.linalg.cross(s, D[k])
                fs[k] += w * (1 - xi) * f
                fe[k] += w * xi * f
        F = fs + fe[self.prv]
        return F * MAT.mu * self.unit ** 2, F

    def velocities(self, F, consistent):
        P = F - self.n * (self.n * F).sum(1, keepdim=True)
        L = (self.x[self.nxt] - self.x).norm(dim=1)
        if not consistent:
            v = P / (0.5 * (L + L[self.prv]))[:, None]
            v[self.pin] = 0.0
            return v
        v = torch.zeros_like(F)
        for a, b in zip(self.off, self.off[1:]):
            free = (~self.pin[a:b]).nonzero()[:, 0]
            if not free.numel():
                continue
            m = int(b - a)
            M = torch.zeros((m, m), dtype=torch.float64, device="cuda")
            k = torch.arange(m, device="cuda")
            j = (k + 1) % m
            l = L[a:b]
            M.index_put_((k, k), l / 3, accumulate=True)
            M.index_put_((j, j), l / 3, accumulate=True)
            M.index_put_((k, j), l / 6, accumulate=True)
            M.index_put_((j, k), l / 6, accumulate=True)
            v[a + free] = torch.linalg.solve(M[free][:, free], P[a:b][free])
        return v


def _exact_burst(net, steps, consistent):
    box = _Box(net)
    dt = DT * MAT.mu / MAT.B
    targets = (~(box.pin & box.pin[box.nxt])).nonzero()[:, 0]
    Lp, rho = torch.zeros((3, 3), dtype=torch.float64, device="cuda"), 0.0
    for _ in range(steps):
        v = box.velocities(box.forces(targets)[1], consistent)
        D = box.x[box.nxt] - box.x
        Lp = Lp + box.b.T @ torch.linalg.cross(D, 0.5 * (v + v[box.nxt]))
        rho = rho + D.norm(dim=1).sum()
        box.x = box.x + dt * v
    u = box.unit
    return dict(Lp=(Lp * u ** 3 * MAT.mu / (MAT.B * box.volume * steps)).cpu().numpy(),
                rho=float(rho) * u / (box.volume * steps), nodes=(box.x * u).cpu().numpy())
