"""Performance cases of the fractional-ADE lattice Boltzmann framework.

Each case is one unit of work of a program that uses the package: a run of a lattice from its
initial concentration (reset, time steps, concentration read into device memory), an ensemble
of uneven problems advanced together, a loss and its gradient of a parameter fit, or a
Monte-Carlo walk with its histogram.  The handle, with the launch configuration that the
library picks by itself, is what such a program keeps; the parameters, initial fields and
observations come from the seed.

Problems are posed in physical units, as the paper's validations are: the longest axis spans
[0, 1] (dx = 1 / (nodes - 1)), and dt puts the relaxation time of the largest D at 1.  The
concentration of a form that works in FP32 is returned as FP32: the ABI's FP64 arrays hold
those values widened.

``exact`` restates the scheme (arXiv:1706.09161) in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_1706_09161_gb300 import lbm
from paper_1706_09161_gb300.workloads import Problem

# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # the smallest problem: pure fractional diffusion in FP64, where a step is two short launches
        run_case("bgk_64_fp64", (64, 64), "fp64", "bgk", 200),
        # FP64 in 3-D, at the paper's own 3-D validation size: the reference runs of a study
        run_case("bgk_80x80x80_fp64", (80, 80, 80), "fp64", "bgk", 8),
        # the benchmark lattice in the tensor-core form that carries FP32's precision
        run_case("mrt_512_bf16x6", (512, 512), "bf16x6split", "mrt", 256),
        # the same lattice in plain FP32 arithmetic
        run_case("mrt_512_fp32", (512, 512), "fp32", "mrt", 128),
        # a lattice whose sides are no multiple of any tile or of 16 bytes
        run_case("mrt_301x203_bf16x6", (301, 203), "bf16x6split", "mrt", 128),
        # the large 3-D lattice, streamed from HBM, in both tensor-core forms offered for it
        run_case("mrt_256x256x256_tf32", (256, 256, 256), "tf32split", "mrt", 16),
        run_case("mrt_256x256x256_bf16x6", (256, 256, 256), "bf16x6split", "mrt", 16),
        # a 3-D box with ragged sides
        run_case("mrt_130x101x75_bf16x6", (130, 101, 75), "bf16x6split", "mrt", 32),
        # D(x), g(x) and u(x) varying from node to node
        run_case("varying_512_bf16x6", (512, 512), "bf16x6split", "mrt", 128, fields=True),
        # an ensemble of uneven sides advanced by grouped launches
        dict(name="batch_16_bf16x6", kind="batch", precision="bf16x6split", steps=64,
             sides="128,256,384,512,768,1024,256,512,128,1024,384,768,512,256,384,128"),
        # one evaluation of a parameter fit: forward, recomputation from checkpoints, adjoint
        dict(name="fit_256_fp32", kind="fit", n0=256, n1=256, steps=300, snaps=10, ckpt=100, precision="fp32"),
        # the Monte-Carlo counterpart: killed stable-Levy paths and their histogram
        dict(name="walk_2d_fp32", kind="walk", d=2, paths=4000000, steps=50, precision="fp32"),
    ]


def run_case(name, grid, precision, collision, steps, fields=False):
    c = dict(kind="run", d=len(grid), n0=grid[0], n1=grid[1], n2=grid[2] if len(grid) == 3 else 1,
             precision=precision, collision=collision, steps=steps, fields=fields)
    return dict(name=name, **c) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    """A side length over [lo, hi], every second one a multiple of 16."""
    n = _log_int(rng, lo, hi)
    return n if rng.random() < 0.5 else max(lo, n // 16 * 16)


def draw(rng):
    kind = rng.choice(["run2", "run2", "run2", "run3", "run3", "fields", "batch", "fit", "walk"])
    tc = ["bf16x6split", "bf16split", "tf32split"]
    if kind in ("run2", "fields"):
        prec = rng.choice(["fp64", "fp32"] + tc)
        hi = 256 if prec == "fp64" else 1024
        grid = (_side(rng, 48, hi), _side(rng, 48, hi))
        return run_case(None, grid, prec, rng.choice(["bgk", "mrt"]), _log_int(rng, 16, 160), fields=kind == "fields")
    if kind == "run3":
        prec = rng.choice(["fp64", "fp32"] + tc)
        hi = 72 if prec == "fp64" else 200
        return run_case(None, tuple(_side(rng, 24, hi) for _ in range(3)), prec, rng.choice(["bgk", "mrt"]),
                        _log_int(rng, 4, 12))
    if kind == "batch":
        sides = [_side(rng, 64, 768) for _ in range(rng.randint(3, 12))]
        return dict(kind="batch", precision=rng.choice(["bf16x6split", "bf16split", "fp32"]), steps=_log_int(rng, 8, 48),
                    sides=",".join(str(s) for s in sides))
    if kind == "fit":
        snaps = rng.randint(2, 8)
        return dict(kind="fit", n0=_side(rng, 48, 256), n1=_side(rng, 48, 256), steps=snaps * _log_int(rng, 4, 24),
                    snaps=snaps, ckpt=rng.choice([20, 50, 100]), precision=rng.choice(["fp32", "fp32", "bf16x6split"]))
    return dict(kind="walk", d=rng.choice([2, 3]), paths=_log_int(rng, 1 << 14, 1 << 20), steps=_log_int(rng, 16, 64),
                precision=rng.choice(["fp32", "fp64"]))


# --------------------------------------------------------------------------- inputs


def _hill(grid, centre, sigma, dx):
    """Gaussian hill, zero on the walls, of unit peak (numpy, axis 0 of the problem fastest)."""
    out = np.ones(())
    for n, c in zip(grid, centre):
        x = np.arange(n) * dx
        line = np.exp(-0.5 * ((x - c * (n - 1) * dx) / sigma) ** 2)
        line[0] = line[-1] = 0.0
        out = line.reshape((n,) + (1,) * out.ndim) * out
    return np.ascontiguousarray(out)


def _problem(rng, grid, collision):
    d = len(grid)
    e2 = 1.0 / 3.0 if d == 2 else 0.25
    dx = 1.0 / (max(grid) - 1)
    Dd = [float(v) for v in rng.uniform(0.01, 0.03, size=d)]
    if collision == "bgk":
        Dd = Dd[:1] * d
    nfree = {2: 2, 3: 3}[d] if collision == "mrt" else 0
    pb = Problem(d=d, collision=collision, grid=tuple(grid),
                 alpha=tuple(float(v) for v in rng.uniform(1.4, 1.95, size=d)),
                 p=tuple(float(v) for v in rng.uniform(0.1, 0.9, size=d)), g=(1.0,) * d,
                 D=tuple(tuple(Dd[i] if i == j else 0.0 for j in range(d)) for i in range(d)),
                 u=tuple(float(v) for v in rng.uniform(-0.1, 0.1, size=d)),
                 s_free=tuple(float(v) for v in rng.uniform(0.8, 1.6, size=nfree)),
                 dx=dx, dt=0.5 * e2 * dx * dx / max(Dd))
    C0 = _hill(grid, rng.uniform(0.35, 0.65, size=d), float(rng.uniform(0.06, 0.12)), dx)
    return pb, C0


def _wave(rng, grid, amp):
    axes = np.meshgrid(*[np.linspace(0.0, 1.0, n) for n in reversed(grid)], indexing="ij")
    k = rng.uniform(0.5, 2.0, size=len(grid))
    return amp * np.sin(2 * np.pi * (rng.uniform() + sum(a * x for a, x in zip(k, axes))))


def _fields(rng, pb):
    """Smooth D(x) (with off-diagonal entries under MRT, spherical under BGK), g(x) and u(x)."""
    d, D0 = pb.d, pb.D[0][0]
    D = np.zeros((d, d) + pb.shape)
    for i in range(d):
        D[i, i] = D0 * (1.0 + _wave(rng, pb.grid, 0.4)) if pb.collision == "mrt" or i == 0 else D[0, 0]
    if pb.collision == "mrt":
        D[0, 1] = D[1, 0] = D0 * _wave(rng, pb.grid, 0.1)
    g = np.stack([1.0 + _wave(rng, pb.grid, 0.2) for _ in range(d)])
    u = np.stack([pb.u[i] + _wave(rng, pb.grid, 0.05) for i in range(d)])
    return {"D": D, "g": g, "u": u}


def _grid(case):
    return (case["n0"], case["n1"], case["n2"])[:case["d"]]


def _run_inputs(case, seed):
    rng = np.random.default_rng(seed)
    pb, C0 = _problem(rng, _grid(case), case["collision"])
    return pb, C0, _fields(rng, pb) if case["fields"] else None


def _batch_inputs(case, seed):
    rng = np.random.default_rng(seed)
    return [_problem(rng, (int(s), int(s)), "mrt") for s in case["sides"].split(",")]


def _fit_inputs(case, seed):
    """Problem, initial field, snapshot steps, observed plumes (hills with noise) and the guess theta."""
    rng = np.random.default_rng(seed)
    pb, C0 = _problem(rng, (case["n0"], case["n1"]), "mrt")
    snaps = [case["steps"] * (k + 1) // case["snaps"] for k in range(case["snaps"])]
    centre = rng.uniform(0.4, 0.6, size=2)
    obs = np.stack([_hill(pb.grid, centre, 0.09 + 0.01 * k / len(snaps), pb.dx) for k in range(len(snaps))])
    obs += rng.normal(0.0, 1e-3, size=obs.shape)
    theta = np.array(pb.alpha + pb.p + (pb.D[0][0], pb.D[1][1]) + pb.u, dtype=np.float32)
    return pb, C0, snaps, obs, theta


WALK = dict(alpha=(1.5, 1.7, 1.8), p=(0.3, 0.8, 0.5), D=(0.1, 0.1, 0.08), u=(0.2, -0.1, 0.0), dt=1.0 / 2400)
WALK_CELLS = 64


def _walk_start(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = 0.5 + 0.1 * torch.randn(case["d"], case["paths"], dtype=torch.float64, device="cuda", generator=g)
    return x.clamp_(0.05, 0.95)


# --------------------------------------------------------------------------- a user's program


def prepare(case, seed):
    kind = case["kind"]
    if kind == "walk":
        d = case["d"]
        prm = lbm.walk_params(d, WALK["alpha"], WALK["p"], WALK["D"], (1.0,) * d, WALK["u"], (0.0,) * d, (1.0,) * d,
                              WALK["dt"], seed, case["precision"])
        return dict(case=case, prm=prm, X=_walk_start(case, seed))
    stream = torch.cuda.Stream()
    s = dict(case=case, stream=stream)
    if kind == "run":
        pb, C0, fields = _run_inputs(case, seed)
        s["lat"] = lbm.Lattice(pb, C0, case["precision"], stream=stream.cuda_stream)
        if fields:
            s["lat"].set_fields(**fields)
    elif kind == "batch":
        probs = _batch_inputs(case, seed)
        s["lat"] = lbm.Batch([p for p, _ in probs], [c for _, c in probs], case["precision"], stream=stream.cuda_stream)
    else:
        pb, C0, snaps, obs, theta = _fit_inputs(case, seed)
        s.update(pb=pb, C0=C0, snaps=snaps, obs=obs, theta=torch.tensor(theta, device="cuda"))
        s["lat"] = lbm.Lattice(pb, C0, case["precision"], stream=stream.cuda_stream)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "run":
        lat = s["lat"]
        with torch.cuda.stream(s["stream"]):
            C = torch.empty(lat.shape, dtype=torch.float64, device="cuda")
            lat.reset()
            lat.step(case["steps"])
            lat.C_into(C)
            return C if case["precision"] == "fp64" else C.float()
    if case["kind"] == "batch":
        b = s["lat"]
        with torch.cuda.stream(s["stream"]):
            out = [torch.empty(shape, dtype=torch.float64, device="cuda") for shape in b.shapes]
            b.reset()
            b.step(case["steps"])
            for k, C in enumerate(out):
                b.C_into(k, C)
            return [C.float() for C in out]
    if case["kind"] == "fit":
        theta = s["theta"].clone().requires_grad_(True)
        loss = lbm.snapshot_loss(s["pb"], s["C0"], s["snaps"], s["obs"], theta, precision=case["precision"],
                                 ckpt_every=case["ckpt"], lattice=s["lat"])
        loss.backward()
        return dict(loss=loss.detach(), grad=theta.grad)
    d, n = case["d"], case["paths"]
    st = torch.cuda.current_stream().cuda_stream
    X = s["X"].clone()
    alive = torch.ones(n, dtype=torch.uint8, device="cuda")
    counts = torch.zeros((WALK_CELLS + 1,) * d, dtype=torch.int32, device="cuda")
    lbm.lbm_walk(s["prm"], n, X.data_ptr(), alive.data_ptr(), 0, case["steps"], st)
    lbm.lbm_walk_density(s["prm"], n, X.data_ptr(), alive.data_ptr(), (WALK_CELLS + 1,) * d, 1.0 / WALK_CELLS,
                         counts.data_ptr(), st)
    return dict(X=X if case["precision"] == "fp64" else X.float(), alive=alive, counts=counts)


# --------------------------------------------------------------------------- work that a pass cannot do without


def _step_work(grid, elem):
    """Bytes and flops of one time step: populations in and out and C out; 2 side flops per node
    and axis in the operator, about 2 Q^2 in the collision."""
    d, nodes = len(grid), math.prod(grid)
    Q = 2 * d + 1
    return nodes * (2 * Q + 1) * elem, nodes * (2 * sum(grid) + 2 * Q * Q)


def work(case):
    kind, steps = case["kind"], case["steps"]
    if kind == "walk":  # positions in and out, flags out; about 300 operations per increment of an axis
        return dict(bytes=case["paths"] * (16 * case["d"] + 1), flops=300 * case["d"] * case["paths"] * steps)
    if kind == "batch":
        per = [_step_work((int(s), int(s)), 4) for s in case["sides"].split(",")]
    else:
        per = [_step_work(_grid(dict(d=2, n2=1, **case) if kind == "fit" else case), 8 if case["precision"] == "fp64" else 4)]
    b, f = (steps * sum(v) for v in zip(*per))
    # a fit's evaluation: the forward step, its adjoint, and the weights' gradient, each as much again
    return dict(bytes=2 * b, flops=3 * f) if kind == "fit" else dict(bytes=b, flops=f)


# --------------------------------------------------------------------------- the scheme in 64 bits

DT = torch.float64


def _matrix(alpha, p, n, dx):
    """p I+^(2-alpha) + (1-p) I-^(2-alpha) on a line of n nodes by product integration on linear
    elements (Eqs. 1Dminus_discret, c+, c-); the line's own end entries are 0 for alpha < 2."""
    gam = 2.0 - alpha
    s = gam + 1.0
    k = torch.arange(1, n + 1, dtype=DT, device="cuda")
    pw = torch.cat([torch.zeros(1, dtype=DT, device="cuda"), k ** s])                   # 0^s .. n^s
    a = pw[2:] - 2.0 * pw[1:-1] + pw[:-2]                                               # a[k-1], k = 1..n-1
    m = k[:-1]
    b = s * m ** gam - pw[1:-1] + pw[:-2]                                               # b[m-1], m = 1..n-1
    row = torch.arange(n, device="cuda")
    diff = row[:, None] - row[None, :]
    W = torch.where(diff > 0, a[(diff - 1).clamp(min=0)], torch.zeros((), dtype=DT, device="cuda"))
    W = W + torch.diag((row > 0).to(DT))
    W = torch.cat([torch.cat([torch.zeros(1, dtype=DT, device="cuda"), b])[:, None], W[:, 1:]], dim=1)
    return dx ** gam / torch.exp(torch.lgamma(2.0 + gam)) * (p * W + (1.0 - p) * W.flip(0, 1))


class _Scheme:
    """The lattice Boltzmann step in FP64; theta = (alpha, p, D, u) may carry gradients."""

    def __init__(self, pb, theta=None, fields=None):
        d = self.d = pb.d
        dev = dict(dtype=DT, device="cuda")
        if theta is None:
            theta = torch.tensor(pb.alpha + pb.p + tuple(pb.D[i][i] for i in range(d)) + pb.u, **dev)
        alpha, p, D, u = theta[:d], theta[d:2 * d], theta[2 * d:3 * d], theta[3 * d:]
        shape = pb.shape
        f = {k: torch.tensor(v, **dev) for k, v in (fields or {}).items()}
        self.g = f.get("g")
        Dm = f["D"].movedim((0, 1), (-2, -1)) if "D" in f else torch.diag(D)             # (..., d, d)
        e2 = 1.0 / 3.0 if d == 2 else 0.25
        self.w0 = e2
        self.wi = (1.0 - e2) / (2 * d)
        self.adv = (f["u"] if "u" in f else u.reshape((d,) + (1,) * d)) * (pb.dt / pb.dx / e2 * self.wi)
        self.K = [_matrix(alpha[i], p[i], pb.grid[i], pb.dx) for i in range(d)]
        Q = 2 * d + 1
        lamb = Dm * (pb.dt / pb.dx ** 2 / e2) + 0.5 * torch.eye(d, **dev)                # relaxation times
        if pb.collision == "bgk":
            Om = torch.eye(Q, **dev) / lamb[..., :1, :1]
        else:
            rows = [[1] * Q] + [[(q == 2 * i + 1) - (q == 2 * i + 2) for q in range(Q)] for i in range(d)]
            rows += [[2 * d] + [-1] * (2 * d)]
            rows += [[0, 1, 1, -1, -1]] if d == 2 else [[0, 2, 2, -1, -1, -1, -1], [0, 0, 0, 1, 1, -1, -1]]
            M = torch.tensor(rows, **dev)
            L = torch.diag_embed(torch.tensor([1.0] * (1 + d) + list(pb.s_free), **dev)).expand(lamb.shape[:-2] + (Q, Q)).clone()
            L[..., 1:1 + d, 1:1 + d] = torch.linalg.inv(lamb)
            Om = torch.linalg.inv(M) @ L @ M
        self.Om = Om.movedim((-2, -1), (0, 1)) if Om.dim() > 2 else Om.reshape((Q, Q) + (1,) * d)
        self.unknown = torch.zeros((Q,) + shape, dtype=torch.bool, device="cuda")
        for q in range(1, Q):
            self.unknown[q].select(d - 1 - (q - 1) // 2, 0 if q % 2 else -1)[:] = True
        self.k = self.unknown.sum(0)
        self.Cw = pb.C_wall

    def F(self, C):
        out = []
        for mu, K in enumerate(self.K):
            x = C if self.g is None else self.g[mu] * C
            dim = self.d - 1 - mu
            out.append(torch.movedim(torch.tensordot(K, x, dims=([1], [dim])), 0, dim))
        return out

    def feq(self, C, F):
        out = [C - self.w0 * sum(F)]
        for mu in range(self.d):
            out += [self.wi * F[mu] + self.adv[mu] * C, self.wi * F[mu] - self.adv[mu] * C]
        return torch.stack(out)

    def start(self, C0):
        return self.feq(C0, self.F(C0))

    def step(self, f):
        C = f.sum(0)
        dl = f - self.feq(C, self.F(C))
        fs = f - (self.Om * dl[None]).sum(1)
        new = [fs[0]]
        for q in range(1, 2 * self.d + 1):
            new.append(torch.roll(fs[q], 1 if q % 2 else -1, self.d - 1 - (q - 1) // 2))
        new = torch.stack(new).masked_fill(self.unknown, 0.0)
        fill = (self.Cw - new.sum(0)) / self.k.clamp(min=1)
        return torch.where(self.unknown, fill, new)


def _exact_run(pb, C0, steps, fields=None):
    with torch.no_grad():
        S = _Scheme(pb, fields=fields)
        f = S.start(torch.tensor(C0, device="cuda"))
        for _ in range(steps):
            f = S.step(f)
        return f.sum(0)


def _exact_fit(case, seed):
    pb, C0, snaps, obs, theta = _fit_inputs(case, seed)
    th = torch.tensor(theta, dtype=DT, device="cuda").requires_grad_(True)
    S = _Scheme(pb, th)
    obs = torch.tensor(obs, device="cuda")
    f = S.start(torch.tensor(C0, device="cuda"))
    loss = torch.zeros((), dtype=DT, device="cuda")
    t = 0
    for k, at in enumerate(snaps):
        while t < at:
            f = S.step(f)
            t += 1
        loss = loss + (f.sum(0) - obs[k]).square().sum()
    loss.backward()
    return dict(loss=loss.detach(), grad=th.grad)


def _philox(i, step, call, seed):
    """Philox4x32-10 (Salmon et al., SC 2011) of counter (i, 0, step, call); 32-bit words in int64."""
    mask = 0xFFFFFFFF

    def mul(m, x):
        t = x * (m & 0xFFFF)
        return ((x * (m >> 16) + (t >> 16)) >> 16) & mask, (x * m) & mask
    c = [i, torch.zeros_like(i), torch.full_like(i, step), torch.full_like(i, call)]
    k0, k1 = seed & mask, seed >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _exact_walk(case, seed):
    """The walk with stable increments by the formula of Chambers, Mallows and Stuck (Weron 1996)."""
    d, n, dt = case["d"], case["paths"], WALK["dt"]
    X = _walk_start(case, seed)
    live = torch.ones(n, dtype=torch.bool, device="cuda")
    i = torch.arange(n, device="cuda")

    def uniform(o):
        return (o.to(DT) + 0.5) / 2.0 ** 32 if case["precision"] == "fp64" else ((o >> 9).to(DT) + 0.5) / 2.0 ** 23
    for step in range(case["steps"]):
        o = _philox(i, step, 0, seed)
        if d == 3:
            o = o + _philox(i, step, 1, seed)[:2]
        move = []
        for mu in range(d):
            a, D, u, beta = WALK["alpha"][mu], WALK["D"][mu], WALK["u"][mu], 2.0 * WALK["p"][mu] - 1.0
            V = math.pi * (uniform(o[2 * mu]) - 0.5)
            W = -torch.log(uniform(o[2 * mu + 1]))
            t = beta * math.tan(math.pi * a / 2.0)
            B = math.atan(t) / a
            S = (1.0 + t * t) ** (0.5 / a) * torch.sin(a * (V + B)) / torch.cos(V) ** (1.0 / a) \
                * (torch.cos(V - a * (V + B)).clamp(min=0.0) / W) ** ((1.0 - a) / a)
            move.append(u * dt + (D * -math.cos(math.pi * a / 2.0) * dt) ** (1.0 / a) * S)
        X = torch.where(live, X + torch.stack(move), X)
        live = live & ((X > 0.0) & (X < 1.0)).all(0)
    return dict(X=X, alive=None, counts=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "run":
        pb, C0, fields = _run_inputs(case, seed)
        return _exact_run(pb, C0, case["steps"], fields)
    if kind == "batch":
        return [_exact_run(pb, C0, case["steps"]) for pb, C0 in _batch_inputs(case, seed)]
    return _exact_fit(case, seed) if kind == "fit" else _exact_walk(case, seed)
