"""The calls that a program built on this package makes, with inputs of the
sizes and distributions that it meets, for timing and for comparing results.

A case is a plain dict:

  kind    what is called:
            hessvec    one Gauss-Newton Hessian-vector product at a linearisation
                       point (the body of a PCG iteration)
            gradient   one reduced gradient with its energies (a Gauss-Newton or
                       gradient-descent iteration's first call)
            train      a batch of differentiable shoots: forward and backward
            metric     the metric operator K = L^-1 on vector fields, through a handle
            noalloc    the same operator through the entry point without allocation
            register   one whole registration
  n0, n1, n2           the grid
  form    f32, f64 (compute and stored states), or bf16 (FP32 compute, states
          stored as bfloat16)
  nt      time steps; ckpt: states kept every so many steps (1: all)
  metric_space         V or L2; interp: cubic or linear
  mode    jacobi or discrete (the gradient's mode)
  batch   members of a train case, or fields of a metric case

The images are nested ellipsoids with noise, the target is the same phantom
seen through a smooth displacement, the velocity at the linearisation point
is a random smooth field of n_min / 20 voxels peak displacement, half of the
one that made the target, as in the middle of a registration.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_1807_04638_gb300 as pkg
from paper_1807_04638_gb300.autograd import Shooter, shoot

ALPHA = 0.005
WEIGHT = 1e-3
TWO_PI = 2.0 * math.pi
# registration of a case of kind register: iterations and the caps of each
GN, PCG, RTOL = 2, 5, 0.1


def _case(kind, n, form="f32", nt=10, **kw):
    c = {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2], "form": form, "nt": nt, "ckpt": 1, "metric_space": "V",
         "interp": "cubic", "mode": "jacobi", "batch": 3 if kind in ("metric", "noalloc") else 1}
    c.update(kw)
    return c


def listed():
    cases = [
        # the benchmark's headline: a PCG iteration of the 128^3 registration
        _case("hessvec", (128, 128, 128), name="hv_128"),
        # the smallest grid of the serving trace: launches and latency count
        _case("hessvec", (64, 64, 64), name="hv_64"),
        # the largest grid of the serving trace, mixed radices 3 and 5
        _case("hessvec", (160, 192, 160), name="hv_160x192x160"),
        # a volume cropped to its content: no axis is a round number, odd last axis
        _case("hessvec", (75, 90, 81), nt=6, metric_space="L2", name="hv_75x90x81"),
        # the brain-shaped volume in its memory-saving form (bfloat16 states, checkpoints)
        _case("hessvec", (256, 300, 256), "bf16", ckpt=2, name="hv_256x300x256_bf16"),
        # the plain FP64 method, which the FP32 form is judged against
        _case("hessvec", (64, 64, 64), "f64", name="hv_64_f64"),
        # first call of every Gauss-Newton iteration at the headline size
        _case("gradient", (128, 128, 128), name="grad_128"),
        # gradient descent with the exact gradient of the discrete energy
        _case("gradient", (96, 96, 96), mode="discrete", name="grad_96_discrete"),
        # the differentiable layer inside a training step: a batch of eight 96^3 pairs
        _case("train", (96, 96, 96), batch=8, name="train_8x96"),
        # smoothing a velocity field with K at the headline size
        _case("metric", (128, 128, 128), name="metric_128"),
        # the smallest call: K on a small field inside another program's loop
        _case("noalloc", (32, 32, 32), name="noalloc_32"),
        # a whole small registration, with its host decisions
        _case("register", (64, 64, 64), name="register_64"),
    ]
    return cases


def _smooth(m):
    for r in (2, 3, 5):
        while m % r == 0:
            m //= r
    return m == 1


def draw(rng):
    kind = rng.choice(["hessvec"] * 6 + ["gradient"] * 3 + ["train", "metric", "noalloc", "register"])
    form = "f32"
    if kind in ("hessvec", "gradient", "train", "register"):
        form = rng.choice(["f32"] * 5 + ["f64"] + (["bf16"] if kind in ("hessvec", "gradient") else []))
    elif rng.random() < 0.3:
        form = "f64"
    # points of the grid: log-uniform up to what the kind is used for
    most = {"hessvec": 5e6, "gradient": 5e6, "train": 1e6, "metric": 8e6, "noalloc": 1.2e6, "register": 3e5}[kind]
    if form == "f64":
        most = min(most, 6e5)
    regular = rng.random() < 0.5  # volumes resampled to a multiple of 16, or cropped to any size that is taken
    while True:
        side = math.exp(rng.uniform(math.log(16.0 ** 3), math.log(most))) ** (1.0 / 3.0)
        n = []
        for _ in range(3):
            want = side * math.exp(rng.uniform(-0.3, 0.3))
            ok = [m for m in range(12, 321) if _smooth(m) and (m % 16 == 0 or not regular)]
            n.append(min(ok, key=lambda m: abs(math.log(m / want))))
        if n[0] * n[1] * n[2] <= most:
            break
    c = _case(kind, n, form, nt=rng.choice([5, 8, 10]))
    if kind in ("hessvec", "gradient"):
        c["metric_space"] = rng.choice(["V", "V", "L2"])
        if rng.random() < 0.2:
            c["ckpt"] = rng.choice([2, 3])
    if kind == "gradient" and form != "bf16" and c["ckpt"] == 1 and rng.random() < 0.3:
        c["mode"] = "discrete"
    if kind in ("gradient", "train") and rng.random() < 0.2:
        c["interp"] = "linear"
    if kind == "train":
        c["batch"] = rng.choice([2, 4, 8])
    if kind in ("metric", "noalloc"):
        c["batch"] = rng.choice([1, 3])
    if kind == "noalloc" and form == "f64":
        c["n2"] = min(c["n2"], 64)
    return c


# ------------------------------------------------------------------ inputs
def _grid(case):
    return case["n0"], case["n1"], case["n2"]


def _dtype(case):
    return torch.float64 if case["form"] == "f64" else torch.float32


def _wave(n):
    """Integer wave numbers of a half spectrum, broadcastable, in FP64."""
    k = (np.rint(np.fft.fftfreq(n[0]) * n[0]), np.rint(np.fft.fftfreq(n[1]) * n[1]), np.rint(np.fft.rfftfreq(n[2]) * n[2]))
    shape = ((-1, 1, 1), (1, -1, 1), (1, 1, -1))
    return [torch.tensor(k[a], dtype=torch.float64, device="cuda").reshape(shape[a]) for a in range(3)]


def _band_field(n, gen, kmax, comps=3):
    """Random smooth periodic fields of wave numbers |k| <= kmax."""
    k = _wave(n)
    keep = (k[0] ** 2 + k[1] ** 2 + k[2] ** 2 <= kmax ** 2).double()
    x = torch.randn((comps,) + n, generator=gen, dtype=torch.float64, device="cuda")
    return torch.fft.irfftn(torch.fft.rfftn(x, dim=(-3, -2, -1)) * keep, s=n, dim=(-3, -2, -1))


def _velocity(n, gen, kmax, voxels):
    """Random smooth velocity whose largest displacement in unit time is `voxels`."""
    v = _band_field(n, gen, kmax)
    h = min(TWO_PI / m for m in n)
    return v * (voxels * h / v.square().sum(0).sqrt().max())


def _pair(n, gen, v):
    """Nested ellipsoids and the same seen through the displacement v, with noise."""
    nn = torch.tensor(n, dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1)
    x = torch.stack(torch.meshgrid(*[torch.arange(m, dtype=torch.float64, device="cuda") for m in n], indexing="ij"))
    r = torch.rand(9, generator=gen, dtype=torch.float64, device="cuda")
    semi = (0.30 + 0.12 * r[:3]).reshape(3, 1, 1, 1) * nn
    centre = nn / 2 + (4 * r[3:6] - 2).reshape(3, 1, 1, 1) * nn / 64
    k = _wave(n)
    blur = torch.exp(-0.5 * TWO_PI ** 2 * ((k[0] / n[0]) ** 2 + (k[1] / n[1]) ** 2 + (k[2] / n[2]) ** 2))

    def phantom(p):
        d = p - centre
        d = d - nn * torch.round(d / nn)
        img = torch.zeros(n, dtype=torch.float64, device="cuda")
        for scale, level in ((1.0, 0.2), (0.6 + 0.15 * float(r[6]), 0.5), (0.35 + 0.15 * float(r[7]), 0.9)):
            img = torch.where(((d / (semi * scale)) ** 2).sum(0) < 1.0, torch.full_like(img, level), img)
        return torch.fft.irfftn(torch.fft.rfftn(img) * blur, s=n)

    h = torch.tensor([TWO_PI / m for m in n], dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1)
    noise = [0.02 * torch.randn(n, generator=gen, dtype=torch.float64, device="cuda") for _ in range(2)]
    return phantom(x) + noise[0], phantom(x - v / h) + noise[1]


def _inputs(case, seed):
    """The case's arrays, in the type that the call takes."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, t = _grid(case), _dtype(case)
    if case["kind"] in ("metric", "noalloc"):
        x = _band_field(n, gen, min(n) / 6.0, case["batch"])
        x = x + 0.05 * torch.randn((case["batch"],) + n, generator=gen, dtype=torch.float64, device="cuda")
        return {"x": x.to(t).contiguous()}
    kmax = max(1.0, min(6.0, (min(n) - 1) // 3))
    got = []
    for _ in range(case["batch"] if case["kind"] == "train" else 1):
        v = _velocity(n, gen, kmax, min(n) / 20.0)
        I0, I1 = _pair(n, gen, v)
        d = _band_field(n, gen, kmax)
        d = d * (TWO_PI / max(n)) / d.square().mean().sqrt()
        got.append({"v": 0.5 * v, "I0": I0, "I1": I1, "d": d})
    if case["kind"] == "train":
        return {k: torch.stack([g[k] for g in got]).to(t).contiguous() for k in ("v", "I0", "I1")}
    return {k: a.to(t).contiguous() for k, a in got[0].items()}


_STREAM = []


def _stream():
    """The program's own stream, on which its handles run."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def _params(case):
    kind = {"f32": pkg.LDDMM_F32, "f64": pkg.LDDMM_F64, "bf16": pkg.LDDMM_F32}[case["form"]]
    return pkg.default_params(
        alpha=ALPHA, weight=WEIGHT, nt=case["nt"], compute_dtype=kind,
        state_dtype=pkg.LDDMM_BF16 if case["form"] == "bf16" else kind, checkpoint_every=case["ckpt"],
        space=pkg.LDDMM_SPACE_L2 if case["metric_space"] == "L2" else pkg.LDDMM_SPACE_V,
        interp=pkg.LDDMM_INTERP_LINEAR if case["interp"] == "linear" else pkg.LDDMM_INTERP_CUBIC,
        gradient_mode=pkg.LDDMM_GRAD_DISCRETE if case["mode"] == "discrete" else pkg.LDDMM_GRAD_JACOBI,
        gn_maxit=GN, pcg_maxit=PCG, pcg_rtol=RTOL)


def prepare(case, seed):
    a = _inputs(case, seed)
    s = {"case": case, **a}
    kind = case["kind"]
    if kind == "noalloc":
        s["out"] = torch.empty_like(a["x"])
        s["stream"] = _stream()
    elif kind == "train":
        s["shooter"] = Shooter(_grid(case), case["batch"], _params(case))
    else:
        s["handle"] = h = pkg.Handle(_grid(case), _params(case), stream=_stream())
        if kind == "metric":
            s["out"] = torch.empty_like(a["x"])
        else:
            s["grad"], s["out"] = h.new_vec(), h.new_vec()
    torch.cuda.synchronize()
    if kind == "hessvec":
        s["handle"].lddmm_gradient(a["v"], a["I0"], a["I1"], s["grad"], energy=False)
    return s


def run(s):
    case = s["case"]
    kind, h = case["kind"], s.get("handle")
    if kind == "hessvec":
        h.lddmm_hessvec(s["d"], s["out"])
        return s["out"]
    if kind == "gradient":
        e = h.lddmm_gradient(s["v"], s["I0"], s["I1"], s["grad"])
        return {"energy": list(e), "grad": s["grad"]}
    if kind == "train":
        v = s["v"].clone().requires_grad_(True)
        m1 = shoot(v, s["I0"], s["shooter"])
        (m1 - s["I1"]).square().sum().backward()
        return {"m1": m1.detach(), "grad": v.grad}
    if kind == "metric":
        h.lddmm_apply_metric(s["x"], s["out"], -1)
        return s["out"]
    if kind == "noalloc":
        pkg.apply_metric_noalloc(s["x"], s["out"], -1, ALPHA, stream=s["stream"])
        return s["out"]
    with torch.cuda.stream(h.stream):
        v = torch.zeros_like(s["v"])
    r = h.lddmm_register(s["I0"], s["I1"], v)
    return {"v0": v, "energy": r["energy"], "mse_rel": r["mse_rel"],
            "pcg_iters": r["pcg_iters"]}


def work(case):
    """Inputs read once, outputs written once and, in a sweep, the velocity of
    every stored stage read once; the transforms of a stage at 2.5 N log2 N
    flops each (14 + 10 real transforms in a Jacobi stage, 10 + 4 in a
    shooting stage, the fewest that the equations are known to need)."""
    n = _grid(case)
    N = n[0] * n[1] * n[2]
    t = 8 if case["form"] == "f64" else 4
    st = 2 if case["form"] == "bf16" else t
    fft = 2.5 * N * math.log2(N)
    stages = 2 * case["nt"]
    shoot_f, sweep_f = 14 * fft * stages, 24 * fft * stages
    states = 3 * N * st * stages
    kind = case["kind"]
    if kind in ("metric", "noalloc"):
        return {"bytes": 2 * case["batch"] * N * t, "flops": case["batch"] * 2 * fft}
    reshoot = shoot_f if case["ckpt"] > 1 else 0.0
    if kind == "hessvec":
        return {"bytes": 6 * N * t + 2 * states, "flops": 2 * (sweep_f + reshoot)}
    grad = {"bytes": 8 * N * t + 2 * states, "flops": shoot_f + sweep_f + reshoot}
    if kind == "gradient":
        return grad
    if kind == "train":
        return {k: case["batch"] * x for k, x in grad.items()}
    # GN iterations of a gradient, PCG Hessian products and a line search, then the last gradient
    return {"bytes": (GN + 1) * grad["bytes"] + GN * PCG * (6 * N * t + 2 * states) + GN * states,
            "flops": (GN + 1) * grad["flops"] + GN * (2 * PCG * sweep_f + shoot_f)}


# ------------------------------------------------------------------ the same in 64 bits
class _Exact:
    """The method in FP64 on torch's transforms."""

    def __init__(self, case):
        self.case, self.n = case, _grid(case)
        k = _wave(self.n)
        cut = [(m - 1) // 3 for m in self.n]
        self.ksq = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
        self.L = (1.0 + ALPHA * self.ksq) ** 2
        self.P = ((k[0].abs() <= cut[0]) & (k[1].abs() <= cut[1]) & (k[2].abs() <= cut[2])).double()
        self.ik = [1j * torch.where(2 * k[a].abs() == self.n[a], torch.zeros_like(k[a]), k[a]) for a in range(3)]
        self.h = [TWO_PI / m for m in self.n]
        self.cell = self.h[0] * self.h[1] * self.h[2]
        self.dt = 1.0 / case["nt"]

    def f(self, x):
        return torch.fft.rfftn(x, dim=(-3, -2, -1))

    def i(self, X):
        return torch.fft.irfftn(X, s=self.n, dim=(-3, -2, -1))

    def jac(self, V):
        return torch.stack([torch.stack([self.i(self.ik[j] * V[c]) for j in range(3)]) for c in range(3)])

    def state(self, V):
        M = self.L * V
        return self.i(V), self.jac(V), self.i(M), self.jac(M)

    def adstar(self, v, Dv, m, Dm):
        tr = Dv[0, 0] + Dv[1, 1] + Dv[2, 2]
        return torch.stack([m[i] * tr + sum(Dv[j, i] * m[j] + Dm[i, j] * v[j] for j in range(3)) for i in range(3)])

    def rhs(self, V):
        return -self.P / self.L * self.f(self.adstar(*self.state(V)))

    def steps(self, v0):
        """Spectral velocities at the steps and at the Heun predictors."""
        V, at, pred = self.P * self.f(v0), [], []
        for _ in range(self.case["nt"]):
            R = self.rhs(V)
            at.append(V)
            pred.append(V + self.dt * R)
            V = V + 0.5 * self.dt * (R + self.rhs(pred[-1]))
        return at + [V], pred

    def interp(self, f, d):
        """Samples of f [C, n] at the grid points displaced by d voxels [3, n]."""
        cubic = self.case["interp"] == "cubic"
        base = torch.floor(d.detach())
        t = d - base
        if cubic:
            w = [[0.5 * (-x ** 3 + 2 * x ** 2 - x), 0.5 * (3 * x ** 3 - 5 * x ** 2 + 2),
                  0.5 * (-3 * x ** 3 + 4 * x ** 2 + x), 0.5 * (x ** 3 - x ** 2)] for x in t]
        else:
            w = [[1 - x, x] for x in t]
        lo = -1 if cubic else 0
        at = []
        for a in range(3):
            shape = [1, 1, 1]
            shape[a] = -1
            at.append(base[a].long() + torch.arange(self.n[a], device="cuda").reshape(shape))
        flat, out = f.reshape(f.shape[0], -1), 0.0
        for a in range(len(w[0])):
            i0 = torch.remainder(at[0] + lo + a, self.n[0]) * self.n[1]
            for b in range(len(w[0])):
                i1 = (i0 + torch.remainder(at[1] + lo + b, self.n[1])) * self.n[2]
                wab = w[0][a] * w[1][b]
                for c in range(len(w[0])):
                    ix = i1 + torch.remainder(at[2] + lo + c, self.n[2])
                    out = out + wab * w[2][c] * flat[:, ix.reshape(-1)].reshape((-1,) + self.n)
        return out

    def map_step(self, u, a, b, h):
        disp = -0.5 * self.dt * (b + self.interp(a, -self.dt * b / h))
        return disp + self.interp(u, disp / h)

    def transport(self, at):
        h = torch.tensor(self.h, dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1)
        v = [self.i(V) for V in at]
        u = torch.zeros_like(v[0])
        for a, b in zip(v[:-1], v[1:]):
            u = checkpoint(self.map_step, u, a, b, h, use_reentrant=False)
        return u, h

    def image(self, at, I0):
        u, h = self.transport(at)
        return self.interp(I0[None], u / h)[0]

    def grad(self, f):
        F = self.f(f)
        return torch.stack([self.i(self.ik[j] * F) for j in range(3)])

    def tangent(self, V, E, X):
        v, Dv, m, Dm = self.state(V)
        M = self.L * E
        p = self.adstar(self.i(E), self.jac(E), m, Dm) + self.adstar(v, Dv, self.i(M), self.jac(M))
        xi, Dx = self.i(X), self.jac(X)
        q = torch.stack([sum(Dv[i, j] * xi[j] - Dx[i, j] * v[j] for j in range(3)) for i in range(3)])
        return -self.P / self.L * self.f(p), E + self.P * self.f(q)

    def adjoint(self, V, Ye, Yx):
        v, Dv, m, Dm = self.state(V)
        y, yx = self.i(self.P / self.L * Ye), self.i(self.P * Yx)
        my, tr = (m * y).sum(0), Dv[0, 0] + Dv[1, 1] + Dv[2, 2]
        E, X = [], []
        for c in range(3):
            a = self.f(-sum(Dm[i, c] * y[i] for i in range(3)))
            b = self.f(tr * y[c] + sum(Dv[c, i] * y[i] for i in range(3)))
            x = self.f(sum(Dv[i, c] * yx[i] for i in range(3)))
            for j in range(3):
                a = a + self.ik[j] * self.f(m[c] * y[j] + (my if j == c else 0.0))
                b = b - self.ik[j] * self.f(v[j] * y[c])
                x = x + self.ik[j] * self.f(v[j] * yx[c])
            E.append(a - self.L * b)
            X.append(x)
        return torch.stack(E) + Yx, torch.stack(X)

    def sweep_back(self, at, pred, c):
        dt, Yx = self.dt, self.f(c)
        Ye = torch.zeros_like(Yx)
        for k in reversed(range(self.case["nt"])):
            ae, ax = self.adjoint(pred[k], Ye, Yx)
            te, tx = self.adjoint(at[k], 0.5 * dt * Ye + 0.5 * dt * dt * ae, 0.5 * dt * Yx + 0.5 * dt * dt * ax)
            Ye, Yx = Ye + 0.5 * dt * ae + te, Yx + 0.5 * dt * ax + tx
        return self.P * Ye

    def out(self, v, B):
        """2 w L v + B in the metric that is asked for."""
        G = 2 * WEIGHT * self.L * self.f(v) + B
        return self.i(G / self.L if self.case["metric_space"] == "V" else G)

    def hessvec(self, a):
        at, pred = self.steps(a["v"])
        gm = self.grad(self.image(at, a["I0"]))
        E = self.P * self.f(a["d"])
        X = torch.zeros_like(E)
        for k in range(self.case["nt"]):
            be, bx = self.tangent(at[k], E, X)
            ce, cx = self.tangent(pred[k], E + self.dt * be, X + self.dt * bx)
            E, X = E + 0.5 * self.dt * (be + ce), X + 0.5 * self.dt * (bx + cx)
        c = 2 * (gm * self.i(X)).sum(0) * gm
        return self.out(a["d"], self.sweep_back(at, pred, c))

    def energy(self, v, m1, I1):
        data = self.cell * (m1 - I1).square().sum()
        reg = WEIGHT * self.cell * (self.i(self.L * self.f(v)) * v).sum()
        return torch.stack([data + reg, data, reg])

    def gradient(self, a):
        if self.case["mode"] == "discrete":
            v = a["v"].clone().requires_grad_(True)
            e = self.energy(v, self.image(self.steps(v)[0], a["I0"]), a["I1"])
            g = torch.autograd.grad(e[0], v)[0] / self.cell
            if self.case["metric_space"] == "V":
                g = self.i(self.f(g) / self.L)
            return {"energy": e.tolist(), "grad": g.detach()}
        at, pred = self.steps(a["v"])
        m1 = self.image(at, a["I0"])
        b = self.sweep_back(at, pred, -2 * (m1 - a["I1"]) * self.grad(m1))
        return {"energy": self.energy(a["v"], m1, a["I1"]).tolist(), "grad": self.out(a["v"], b)}

    def train(self, a):
        m, g = [], []
        for v, I0, I1 in zip(a["v"], a["I0"], a["I1"]):
            at, pred = self.steps(v)
            m.append(self.image(at, I0))
            g.append(self.i(self.sweep_back(at, pred, -2 * (m[-1] - I1) * self.grad(m[-1]))))
        return {"m1": torch.stack(m), "grad": torch.stack(g)}


def exact(case, seed):
    """What run() returns, in 64 bits; None where it would take too long (the
    discrete gradient of a large grid by automatic differentiation) or where
    rounding decides what is done (a whole registration)."""
    N = case["n0"] * case["n1"] * case["n2"]
    if case["kind"] == "register" or (case["mode"] == "discrete" and N > 1.2e6):
        return None
    a = {k: x.double() for k, x in _inputs(case, seed).items()}
    ex = _Exact(case)
    if case["kind"] in ("metric", "noalloc"):
        return ex.i(ex.f(a["x"]) / ex.L)
    with torch.set_grad_enabled(case["mode"] == "discrete"):
        return getattr(ex, case["kind"])(a)
