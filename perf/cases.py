"""Timed cases of the fractional-Laplacian solver: what its users run.

A case is a dict of plain values with a "kind":

  apply    y = M u, one operator apply (``Plan.apply``), FP32 or FP64
  precond  z = (shift I + scale C h^d L)^{-1} r (``Plan.precond``)
  solve    M u = f (``Plan.solve``), plain FP64 CG or FP32 CG inside FP64
           refinement, on a box or on an L-shaped domain
  steps    consecutive theta steps of the diffusion problem
           (``Plan.time_step``), each from the one before
  batch    many elliptic problems of uneven size at once (``solve_batched``)
  net      loss and gradients of the preconditioner network over a batch
           (``Net.loss_grad``, what one training step computes)

Solves run to 1e-10 and below, the accuracy at which the repository's tests
compare solutions; at 1e-8 two correct solutions may differ by 1e-9.
``exact`` evaluates the same discrete problems in 64 bits with torch alone:
the operator from its definition (singularity-subtracted trapezoidal rule,
polynomial window of radius 20 h) by torch.fft on the doubled grid, the
Laplacian solve by dense sine matrices, solves by conjugate gradients.
"""

import math

import numpy as np
import torch

from paper_1802_03770_gb300 import _lib
from paper_1802_03770_gb300.api import Net, Plan, solve_batched

DEVICE = "cuda"
PRECONDS = {"fd": _lib.FL_PRECOND_FD, "none": _lib.FL_PRECOND_NONE, "auto": _lib.FL_PRECOND_AUTO,
            "shifted": _lib.FL_PRECOND_SHIFTED}
MODES = {"f64": _lib.FL_MODE_F64, "mixed": _lib.FL_MODE_MIXED}
DTYPES = {"f32": torch.float32, "f64": torch.float64}
RHO = 20.0   # window radius / h of a plan with default options


def listed():
    return [
        # the smallest call: the 64 x 64 grid of the dense-LU check, bound by launches and latency
        dict(name="apply2d_f32_64", kind="apply", d=2, n="64x64", alpha=1.0, dtype="f32"),
        # the operator inside every FP32 CG iteration of the 1024 x 1024 benchmark
        dict(name="apply2d_f32_1024", kind="apply", d=2, n="1024x1024", alpha=1.5, dtype="f32"),
        # FP64 residuals on the paper's 1023 x 1023 grid
        dict(name="apply2d_f64_1023", kind="apply", d=2, n="1023x1023", alpha=0.75, dtype="f64"),
        # the operator on the 256^3 grid of the diffusion run, streamed from HBM
        dict(name="apply3d_f32_256", kind="apply", d=3, n="256x256x256", alpha=1.5, dtype="f32"),
        # an FP64 apply on a ragged 3D box (padded lengths 256, 512, 256)
        dict(name="apply3d_f64_ragged", kind="apply", d=3, n="96x135x75", alpha=1.25, dtype="f64"),
        # the fast Poisson solve of a time step on a ragged grid, the preconditioner alone
        dict(name="precond2d_f32_ragged", kind="precond", d=2, n="700x1001", alpha=1.5, dtype="f32",
             shift=1.0, scale=1e-3),
        # the benchmark's solve: 1024 x 1024, FP32 CG inside FP64 refinement, the paper's preconditioner
        dict(name="solve2d_mixed_1024", kind="solve", d=2, n="1024x1024", alpha=1.5, mode="mixed",
             precond="fd", tol=1e-10, domain="box"),
        # plain FP64 CG on the paper's 511 x 511 grid
        dict(name="solve2d_f64_511", kind="solve", d=2, n="511x511", alpha=1.25, mode="f64",
             precond="fd", tol=1e-10, domain="box"),
        # an L-shaped domain (occluded grid), f = 1 up to noise, the paper's preconditioner on the domain
        dict(name="solve2d_lshape_255", kind="solve", d=2, n="255x255", alpha=1.75, mode="mixed",
             precond="fd", tol=1e-10, domain="lshape"),
        # two backward Euler steps of the 256^3 diffusion run (dt = 1e-3)
        dict(name="steps3d_mixed_256", kind="steps", d=3, n="256x256x256", alpha=1.5, theta=1.0, dt=1e-3,
             count=2, mode="mixed", tol=1e-10),
        # many uneven 2D problems at once, sides 96 .. 768
        dict(name="batch2d_mixed_48", kind="batch", count=48, lo=96, hi=768, tol=1e-10, pick=7),
        # one training step's loss and gradients, 512 x 512, two samples
        dict(name="net_grad_512", kind="net", H=512, W=512, batch=2),
    ]


def _log(rng, lo, hi):
    """An integer between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _box(rng, d, lo, hi, most):
    """Extents of a box of at most `most` points."""
    while True:
        n = [_log(rng, lo, hi) for _ in range(d)]
        if rng.random() < 0.4:
            n = [n[0]] * d
        if math.prod(n) <= most:
            return "x".join(str(v) for v in n)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "precond", "solve", "solve", "steps", "batch", "net"])
    alpha = round(rng.uniform(0.5, 1.8), 3)
    if kind == "apply":
        d = rng.choice([1, 2, 2, 3, 3])
        box = _box(rng, d, {1: 31, 2: 31, 3: 15}[d], {1: 4096, 2: 1536, 3: 256}[d], 1 << 24)
        return dict(kind=kind, d=d, n=box, alpha=alpha, dtype=rng.choice(["f32", "f64"]))
    if kind == "precond":
        d = rng.choice([2, 2, 3])
        box = _box(rng, d, {2: 31, 3: 15}[d], {2: 1024, 3: 200}[d], 1 << 22)
        shift = rng.choice([0.0, 1.0])
        return dict(kind=kind, d=d, n=box, alpha=alpha, dtype=rng.choice(["f32", "f64"]), shift=shift,
                    scale=1.0 if shift == 0.0 else 1e-3)
    if kind == "solve":
        d = rng.choice([1, 2, 2, 2, 3])
        box = _box(rng, d, {1: 63, 2: 47, 3: 15}[d], {1: 2047, 2: 1024, 3: 96}[d], 1 << 20)
        domain = "lshape" if d == 2 and rng.random() < 0.25 else "box"
        if domain == "lshape":
            box = "x".join([str(_log(rng, 47, 300))] * 2)
        precond = rng.choice(["fd", "shifted"]) if alpha >= 1.0 and domain == "box" else "fd"
        return dict(kind=kind, d=d, n=box, alpha=alpha, mode=rng.choice(["f64", "mixed", "mixed"]),
                    precond=precond if alpha >= 1.0 else "auto", tol=1e-10, domain=domain)
    if kind == "steps":
        d = rng.choice([2, 3])
        box = _box(rng, d, {2: 63, 3: 31}[d], {2: 1023, 3: 160}[d], 1 << 22)
        return dict(kind=kind, d=d, n=box, alpha=alpha, theta=rng.choice([0.5, 1.0]), dt=1e-3,
                    count=rng.randint(1, 3), mode=rng.choice(["mixed", "mixed", "f64"]), tol=1e-10)
    if kind == "batch":
        hi = rng.choice([256, 384, 512, 640])
        return dict(kind=kind, count=_log(rng, 4, 40), lo=rng.choice([33, 64, 96]), hi=hi, tol=1e-10,
                    pick=rng.randrange(1 << 20))
    return dict(kind=kind, H=64 * rng.randint(1, 8), W=64 * rng.randint(1, 8), batch=rng.randint(1, 2))


def _extents(case):
    return tuple(int(v) for v in case["n"].split("x"))


def _spacing(n):
    return 1.0 / (max(n) + 1)


def _mask(case, n):
    """The unit square without its upper right quarter, as the paper's occluded grid."""
    if case.get("domain", "box") == "box":
        return None
    m = np.ones(n, dtype=np.uint8)
    m[n[0] // 2:, n[1] // 2:] = 0
    return m


def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _bumps(n, count, seed, w_lo=0.05, w_hi=0.2):
    """Sum of Gaussians with random centres, widths and amplitudes on the interior grid (FP64, shape n)."""
    rng = np.random.default_rng(seed)
    axes = [torch.arange(1, v + 1, dtype=torch.float64, device=DEVICE) / (v + 1) for v in n]
    factors = []
    for _ in range(count):
        c, w, a = rng.random(len(n)), rng.uniform(w_lo, w_hi), rng.standard_normal()
        fs = [torch.exp(-((x - float(c[i])) ** 2) / (2.0 * w * w)) for i, x in enumerate(axes)]
        fs[0] = fs[0] * float(a)
        factors.append(fs)
    per = [torch.stack([f[i] for f in factors]) for i in range(len(n))]
    spec = ",".join("b" + "xyz"[i] for i in range(len(n))) + "->" + "xyz"[:len(n)]
    return torch.einsum(spec, *per).contiguous()


def _noise(n, seed):
    return torch.randn(n, dtype=torch.float64, device=DEVICE, generator=_gen(seed))


def _field(case, n, seed):
    """The input field of an apply, a preconditioner solve, a solve or a time step (FP64)."""
    kind = case["kind"]
    if kind == "precond":
        return _noise(n, seed)                       # a CG residual
    if kind == "steps":
        return _bumps(n, 16, seed, 0.05, 0.15)
    if kind == "solve" and case["domain"] == "lshape":
        return 1.0 + 0.01 * _bumps(n, 4, seed)
    f = _bumps(n, 32, seed)
    return f + 1e-3 * _noise(n, seed) if kind == "apply" else f   # CG directions are not smooth


def _batch_problems(case):
    """(side, alpha) of a batch: sides uniform between lo and hi, alpha ~ U(0.5, 1.8)."""
    rng = np.random.default_rng(case["pick"])
    return [(int(rng.integers(case["lo"], case["hi"] + 1)), float(rng.uniform(0.5, 1.8)))
            for _ in range(case["count"])]


# layers of the network: (name, cin, cout, kernel), in the order of the parameter vector
_LAYERS = [("e0a", 3, 16, 3), ("e0b", 16, 16, 3), ("e1a", 16, 32, 3), ("e1b", 32, 32, 3), ("ba", 32, 64, 3),
           ("bb", 64, 64, 3), ("d1a", 96, 32, 3), ("d1b", 32, 32, 3), ("d0a", 48, 16, 3), ("d0b", 16, 16, 3),
           ("head", 16, 1, 1)]


def _net_inputs(case, seed):
    """Parameters (He-normal), features [r / s_r, z0 / s_z, alpha] and targets of a training batch."""
    rng = np.random.default_rng(seed)
    params = []
    for _, cin, cout, k in _LAYERS:
        params.append(rng.standard_normal(cout * cin * k * k) * math.sqrt(2.0 / (cin * k * k)))
        params.append(0.01 * rng.standard_normal(cout))
    params = np.concatenate(params).astype(np.float32)
    b, H, W = case["batch"], case["H"], case["W"]
    xs = torch.empty((b, 3, H, W), dtype=torch.float32, device=DEVICE)
    ts = torch.empty((b, H, W), dtype=torch.float32, device=DEVICE)
    for i in range(b):
        r = _noise((H, W), seed + 17 * i) + _bumps((H, W), 8, seed + i)
        z = _bumps((H, W), 16, seed + 1000 + i)
        t = _bumps((H, W), 8, seed + 2000 + i) + 0.1 * _noise((H, W), seed + 29 * i + 3)
        xs[i, 0] = r / r.square().mean().sqrt()
        xs[i, 1] = z / z.square().mean().sqrt()
        xs[i, 2] = float(rng.uniform(0.3, 1.8))
        ts[i] = t / z.square().mean().sqrt()
    return params, xs, ts


def prepare(case, seed):
    if case["kind"] == "net":
        params, xs, ts = _net_inputs(case, seed)
        net = Net(case["H"], case["W"])
        net.set_params(params)
        return dict(case=case, net=net, xs=xs, ts=ts)
    if case["kind"] == "batch":
        probs = _batch_problems(case)
        plans = [Plan(2, (n, n), 1.0 / (n + 1), a) for n, a in probs]
        fs = [_bumps((n, n), 16, seed + 31 * i).view(-1) for i, (n, _) in enumerate(probs)]
        return dict(case=case, plans=plans, fs=fs)
    n = _extents(case)
    plan = Plan(case["d"], n, _spacing(n), case["alpha"], mask=_mask(case, n))
    x = _field(case, n, seed).to(DTYPES[case.get("dtype", "f64")])
    return dict(case=case, plan=plan, x=x)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        return state["plan"].apply(state["x"])
    if kind == "precond":
        return state["plan"].precond(state["x"], shift=case["shift"], scale=case["scale"])
    if kind == "solve":
        u, _ = state["plan"].solve(state["x"], tol=case["tol"], maxit=4000,
                                   mode=MODES[case["mode"]] | PRECONDS[case["precond"]])
        return u
    if kind == "steps":
        u, seq = state["x"], []
        for _ in range(case["count"]):
            u, _ = state["plan"].time_step(u, case["dt"], theta=case["theta"], tol=case["tol"],
                                           mode=MODES[case["mode"]])
            seq.append(u)
        return seq
    if kind == "batch":
        us, _ = solve_batched(state["plans"], state["fs"], tol=case["tol"], maxit=4000)
        return us
    loss = state["net"].loss_grad(state["xs"], state["ts"])
    _, grads = state["net"].get_params(grads=True)
    return dict(loss=loss, grads=grads)


def _apply_work(n, size):
    """One apply: field in and out and the kernel's distinct values; a real FFT of the doubled box and back."""
    N, P = math.prod(n), math.prod(2 * v for v in n)
    return 3 * N * size, 5.0 * P * math.log2(P)


def work(case):
    kind = case["kind"]
    if kind == "net":
        # 3 x 3 convolutions forward, to the inputs and to the weights: 3 x 2 x macs
        lev = {"e0a": 0, "e0b": 0, "e1a": 1, "e1b": 1, "ba": 2, "bb": 2, "d1a": 1, "d1b": 1, "d0a": 0, "d0b": 0,
               "head": 0}
        px = case["H"] * case["W"]
        macs = sum(ci * co * k * k * px / 4 ** lev[name] for name, ci, co, k in _LAYERS)
        count = sum(ci * co * k * k + co for _, ci, co, k in _LAYERS)
        return {"bytes": case["batch"] * 4 * px * 4 + 8 * count, "flops": 6.0 * macs * case["batch"]}
    if kind == "batch":
        b = f = 0.0
        for n, _ in _batch_problems(case):
            bb, ff = _apply_work((n, n), 8)
            b, f = b + bb, f + 30 * ff
        return {"bytes": b, "flops": f}
    n = _extents(case)
    size = 4 if case.get("dtype") == "f32" else 8
    b, f = _apply_work(n, size)
    if kind == "precond":
        # sine transforms along all axes but one (a real FFT of 2(n+1) points each way), a tridiagonal solve
        N = math.prod(n)
        return {"bytes": 2 * N * size, "flops": sum(5.0 * N * math.log2(2 * v + 2) for v in n[1:]) + 8.0 * N}
    if kind == "solve":
        return {"bytes": b, "flops": 30 * f}         # tens of applies: 30 are counted
    if kind == "steps":
        return {"bytes": (case["count"] + 2) * math.prod(n) * 8, "flops": case["count"] * 10 * f}
    return {"bytes": b, "flops": f}


# --- the same results in 64 bits, with torch alone ------------------------------


def _lattice_sum(d, s):
    """sum over m in Z^d, m != 0, of |m|^{-s} (s > d), by the theta-function integral: pi^{-s/2} Gamma(s/2) Z
    = int_1^inf (theta(t)^d - 1)(t^{s/2} + t^{(d-s)/2}) dt/t - 2/s - 2/(d-s)."""
    x, w = np.polynomial.legendre.leggauss(200)
    t, w = 1.0 + 7.0 * (x + 1.0), 7.0 * w
    q = 2.0 * sum(np.exp(-math.pi * k * k * t) for k in range(1, 12))
    power = {1: q, 2: q * (2.0 + q), 3: q * (3.0 + q * (3.0 + q))}[d]
    total = np.sum(w * power * (t ** (s / 2) + t ** ((d - s) / 2)) / t) - 2.0 / s - 2.0 / (d - s)
    return float(total) * math.pi ** (s / 2) / math.gamma(s / 2)


def _stencil_weight(d, alpha):
    """Window sum minus window integral of the singular part, in units of h (window radius RHO)."""
    k = int(RHO) + 1
    ax = np.arange(-k, k + 1, dtype=np.float64)
    m = np.stack(np.meshgrid(*([ax] * d), indexing="ij"), axis=-1).reshape(-1, d)
    r = np.sqrt((m * m).sum(1))
    m, r = m[(r > 0) & (r < RHO)], r[(r > 0) & (r < RHO)]
    t = r / RHO
    win = 1 - 35 * t ** 4 + 84 * t ** 5 - 70 * t ** 6 + 20 * t ** 7
    lattice = 0.5 * np.sum(win * m[:, 0] ** 2 / r ** (d + alpha))
    moment = sum(c / (k - alpha) for c, k in ((1, 2), (-35, 6), (84, 7), (-70, 8), (20, 9)))
    area = 2.0 * math.pi ** (d / 2) / math.gamma(d / 2)
    return float(lattice - 0.5 * area / d * RHO ** (2.0 - alpha) * moment)


class _Operator:
    """M on a box (or the part of it that `mask` selects), by torch.fft in FP64."""

    def __init__(self, n, alpha, mask=None):
        self.n, self.d, self.alpha = tuple(n), len(n), alpha
        d, h = self.d, _spacing(n)
        self.a = _stencil_weight(d, alpha)
        self.c = (2.0 ** alpha * math.gamma((d + alpha) / 2) / (math.pi ** (d / 2) * abs(math.gamma(-alpha / 2)))
                  * h ** -alpha)
        self.mask = None if mask is None else torch.tensor(mask, dtype=torch.float64, device=DEVICE)
        self.shape = tuple(2 * v for v in n)
        sq = torch.zeros((1,) * d, dtype=torch.float64, device=DEVICE)
        inside = torch.ones((1,) * d, dtype=torch.float64, device=DEVICE)
        for i, v in enumerate(n):
            m = torch.arange(2 * v, dtype=torch.float64, device=DEVICE)
            m = torch.minimum(m, 2 * v - m).view([-1 if j == i else 1 for j in range(d)])
            sq, inside = sq + m * m, inside * (m < v)
        k = -torch.where(sq > 0, sq, torch.ones_like(sq)) ** (-(d + alpha) / 2) * inside
        k[(0,) * d] = _lattice_sum(d, d + alpha) - 2 * d * self.a
        for i, v in enumerate(n):
            for j in (1, 2 * v - 1):
                if v > 1:
                    k[tuple(j if q == i else 0 for q in range(d))] += self.a
        self.khat = torch.fft.rfftn(self.c * k).real.contiguous()

    def __call__(self, u):
        u = u if self.mask is None else u * self.mask
        y = torch.fft.irfftn(torch.fft.rfftn(u, s=self.shape) * self.khat, s=self.shape)
        y = y[tuple(slice(0, v) for v in self.n)].contiguous()
        return y if self.mask is None else y * self.mask

    def laplace_solve(self, r, shift, scale):
        """(shift I + scale C h^d L)^{-1} r by sine matrices along every axis."""
        lam = torch.zeros((1,) * self.d, dtype=torch.float64, device=DEVICE)
        mats = []
        for i, v in enumerate(self.n):
            j = torch.arange(1, v + 1, dtype=torch.int64, device=DEVICE)
            jk = (j[:, None] * j[None, :]) % (2 * (v + 1))
            mats.append(torch.sin(math.pi / (v + 1) * jk.double()) * math.sqrt(2.0 / (v + 1)))
            e = 4.0 * torch.sin(math.pi / (2 * (v + 1)) * j.double()) ** 2
            lam = lam + (-self.a * self.c) * e.view([-1 if q == i else 1 for q in range(self.d)])

        def sines(x):
            for i, s in enumerate(mats):
                x = torch.movedim(torch.tensordot(s, x, dims=([1], [i])), 0, i)
            return x

        return sines(sines(r) / (shift + scale * lam))

    def solve(self, f, shift=0.0, scale=1.0, x0=None):
        """(shift I + scale M)^{-1} f by conjugate gradients, restarted from the true residual."""
        f = f if self.mask is None else f * self.mask
        x = torch.zeros_like(f) if x0 is None else x0.clone()
        goal = 1e-14 * float(f.norm())
        for target in (1e-9, 1e-6, 1e-3):
            r = f - (shift * x + scale * self(x))
            p, rr, e = r.clone(), float(r.square().sum()), torch.zeros_like(f)
            stop = max(goal, target * math.sqrt(rr)) ** 2
            for _ in range(5000):
                if rr <= stop:
                    break
                q = shift * p + scale * self(p)
                al = rr / float((p * q).sum())
                e += al * p
                r -= al * q
                new = float(r.square().sum())
                p = r + (new / rr) * p
                rr = new
            x = x + e
        return x


def _exact_net(case, seed):
    """Loss and gradients with BF16 weights and everything else in FP64."""
    F = torch.nn.functional
    params, xs, ts = _net_inputs(case, seed)
    p = torch.tensor(params, device=DEVICE)
    leaves, at = {}, 0
    for name, cin, cout, k in _LAYERS:
        w = p[at:at + cout * cin * k * k].view(cout, cin, k, k)
        at += w.numel()
        b = p[at:at + cout]
        at += cout
        leaves[name] = (w.bfloat16().double().requires_grad_(), b.double().requires_grad_())

    def conv(name, x, act=True):
        w, b = leaves[name]
        y = F.conv2d(x, w, b, padding=w.shape[-1] // 2)
        return torch.relu(y) if act else y

    def up(x):
        return x.repeat_interleave(2, dim=2).repeat_interleave(2, dim=3)

    x = xs.double()
    e0 = conv("e0b", conv("e0a", x))
    e1 = conv("e1b", conv("e1a", F.avg_pool2d(e0, 2)))
    bt = conv("bb", conv("ba", F.avg_pool2d(e1, 2)))
    d1 = conv("d1b", conv("d1a", torch.cat([up(bt), e1], 1)))
    d0 = conv("d0b", conv("d0a", torch.cat([up(d1), e0], 1)))
    loss = (conv("head", d0, act=False)[:, 0] - ts.double()).square().mean()
    loss.backward()
    grads = torch.cat([t.grad.reshape(-1) for name, *_ in _LAYERS for t in leaves[name]])
    return dict(loss=loss.detach(), grads=grads)


def exact(case, seed):
    kind = case["kind"]
    if kind == "net":
        return _exact_net(case, seed)
    if kind == "batch":
        # the larger problems would take minutes
        out = []
        for i, (n, a) in enumerate(_batch_problems(case)):
            out.append(_Operator((n, n), a).solve(_bumps((n, n), 16, seed + 31 * i)).view(-1) if n <= 256 else None)
        return out
    n = _extents(case)
    op = _Operator(n, case["alpha"], _mask(case, n))
    x = _field(case, n, seed).to(DTYPES[case.get("dtype", "f64")]).double()
    if kind == "apply":
        return op(x)
    if kind == "precond":
        return op.laplace_solve(x, case["shift"], case["scale"])
    if kind == "solve":
        return op.solve(x)
    seq, u, th, dt = [], x, case["theta"], case["dt"]
    for _ in range(case["count"]):
        b = u - (1.0 - th) * dt * op(u) if th < 1.0 else u
        u = op.solve(b, 1.0, th * dt, x0=u)
        seq.append(u)
    return seq
