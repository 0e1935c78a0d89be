"""The calls whose time this repository is measured by.

Each case is one call of the public binding (paper_1408_6299_gb300.lib / .autograd) as a registration
program makes it. The sizes are those of the repository's own workloads (bench.py, synth.py, the tests) and
grids between and beyond them: powers of two per axis, square, cubic and ragged. Images, velocities and
directions are band-limited random fields and Gaussian blobs as in synth.py, drawn on the GPU from the seed.

The matvec of a mixed context and the iterates of a mixed solve come out of single-precision sweeps: they
carry single precision's accuracy whatever the type of the array that holds them (the library states 1e-5
per matvec), so those results are handed on as float32. All others are float64.
"""
import math

import torch

from paper_1408_6299_gb300 import autograd, lib

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # the smallest call of the double-precision method: one Hessian matvec of the 32^2 sinusoid workload
        _case("hess-32x32-fp64", "hessvec", (32, 32), 16, beta=1e-2),
        # one PCG matvec of the 128^2 blob workload as a mixed-precision solve makes it
        _case("hess-128x128-mixed", "hessvec", (128, 128), 32, reg=2, mixed=True),
        # the reduced gradient of the same workload, once per outer iteration
        _case("grad-128x128-fp64", "gradient", (128, 128), 32, reg=2),
        # the state solve of one large 2D image pair (every objective evaluation of a line search is one)
        _case("transport-512x512-fp64", "transport", (512, 512), 128),
        # one PCG matvec of the 64^3 Stokes workload: three Chebyshev coefficients, Leray projection
        _case("hess-64c-stokes-mixed", "hessvec", (64, 64, 64), 32, n_c=3, stokes=True, beta=1e-2, mixed=True),
        # the reduced gradient of that workload
        _case("grad-64c-stokes-fp64", "gradient", (64, 64, 64), 32, n_c=3, stokes=True, beta=1e-2),
        # differentiable transport, forward and backward (discrete adjoint), on that workload
        _case("autograd-64c-fp64", "autograd", (64, 64, 64), 32, n_c=3, stokes=True),
        # full Newton matvec on a ragged grid with checkpoints every 4 steps
        _case("newton-32x64x128-mixed", "hessvec", (32, 64, 128), 32, mixed=True, ckpt=4, newton=True),
        # the reduced gradient of a mid-size 3D problem with checkpoints every 8 steps
        _case("grad-128c-ckpt8-fp64", "gradient", (128, 128, 128), 64, reg=2, ckpt=8),
        # the headline matvec: 256^3, 128 steps, checkpoints every 8
        _case("hess-256c-ckpt8-mixed", "hessvec", (256, 256, 256), 128, reg=2, mixed=True, ckpt=8),
        # the preconditioner of that problem, applied once per PCG iteration
        _case("precond-256c", "precond", (256, 256, 256), 128, reg=2),
        # a batch of image pairs registered together: 64^2, 128^2 and 256^2 at 4:2:1, three outer iterations
        # each (the budget of a serving program; single-precision rounding grows through every further
        # Krylov solve, and the iterates of longer runs agree to fewer digits than float32 holds)
        _case("lockstep-4-2-1-mixed", "lockstep", (64, 64), 16, beta=1e-2, mixed=True, count=4),
    ]


def _case(name, op, n, n_t, n_c=1, reg=1, stokes=False, beta=1e-3, mixed=False, ckpt=0, newton=False, count=0):
    c = dict(op=op, n0=n[0], n1=n[1], n2=n[2] if len(n) == 3 else 0, n_t=n_t, n_c=n_c, reg=reg, stokes=stokes,
             beta=beta, mixed=mixed, ckpt=ckpt, newton=newton, count=count)
    return dict(c, name=name) if name else c


def draw(rng):
    op = rng.choice(["hessvec"] * 4 + ["gradient"] * 3 + ["transport", "autograd", "precond"])
    d = rng.choice([2, 3])
    lo, hi = (5, 9) if d == 2 else (3, 8)
    while True:
        n = tuple(1 << rng.randint(lo, hi) for _ in range(d))
        if 2 ** 10 <= math.prod(n) <= 2 ** 21:
            break
    n_c = rng.choice([1, 1, 1, 2, 3])
    stokes = rng.random() < 0.3
    mixed = op == "hessvec" and rng.random() < 0.7
    ckpt = rng.choice([0, 0, 4, 8]) if op in ("hessvec", "gradient") else 0
    newton = op == "hessvec" and rng.random() < 0.2
    reg = rng.choice([1, 2]) if max(n) <= 256 else 1  # H2 is used up to 256 points per axis
    # time steps: the CFL number of speed 0.3 at most 0.2, as the workloads keep it
    n_t = 8
    while 0.3 * max(n) / TWO_PI / n_t > 0.2:
        n_t *= 2
    n_t *= rng.choice([1, 1, 2])
    return _case("", op, n, n_t, n_c, reg, stokes, rng.choice([1e-2, 1e-3]), mixed, ckpt, newton)


def _grid(case):
    return tuple(case[k] for k in ("n0", "n1", "n2") if case[k])


# ----------------------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------------------
def _k(n, half=True):
    """Integer wavenumbers per axis, broadcast to the (half) spectrum."""
    ks = []
    for a, m in enumerate(n):
        last = half and a == len(n) - 1
        k = torch.arange(m // 2 + 1, device="cuda") if last else (torch.fft.fftfreq(m, 1.0 / m, device="cuda"))
        ks.append(k.double().reshape([-1 if b == a else 1 for b in range(len(n))]))
    return ks


def _spec(u, n):
    return torch.fft.rfftn(u, dim=tuple(range(-len(n), 0)))


def _real(U, n):
    return torch.fft.irfftn(U, s=n, dim=tuple(range(-len(n), 0)))


def _band(n, gen, kmax, slope=0.0, fields=1):
    """Random real fields with amplitudes |k|^-slope on 0 < |k| <= kmax and no Nyquist modes."""
    k = _k(n)
    kk = sum(x * x for x in k).sqrt()
    amp = torch.where((kk > 0) & (kk <= kmax), kk.clamp(min=1.0) ** -slope, torch.zeros_like(kk))
    for a, x in enumerate(k):
        amp = torch.where(x.abs() == n[a] // 2, torch.zeros_like(amp), amp)
    return _real(_spec(torch.randn((fields,) + n, dtype=torch.float64, device="cuda", generator=gen), n) * amp, n)


def _leray(w, n):
    """The divergence-free part of d fields (leading axis)."""
    k = [torch.where(x.abs() == n[a] // 2, torch.zeros_like(x), x) for a, x in enumerate(_k(n))]
    kk = sum(x * x for x in k)
    W = _spec(w, n)
    q = sum(k[i] * W[i] for i in range(len(n))) / torch.where(kk > 0, kk, torch.ones_like(kk))
    return _real(torch.stack([W[i] - k[i] * q for i in range(len(n))]), n)


def _velocity(n, gen, n_c, speed, stokes, kmax):
    """n_c coefficient fields whose speeds add up to at most `speed`."""
    out = []
    for w in ([1.0], [0.7, 0.3], [0.6, 0.25, 0.15])[n_c - 1]:
        v = _band(n, gen, kmax, 1.5, len(n))
        if stokes:
            v = _leray(v, n)
        out.append(v * (w * speed / v.square().sum(0).sqrt().max()))
    return torch.stack(out).contiguous()


def _blobs(n, gen, count=8):
    img = torch.zeros(n, dtype=torch.float64, device="cuda")
    x = [(torch.arange(m, device="cuda").double() * (TWO_PI / m)).reshape([-1 if b == a else 1 for b in range(len(n))])
         for a, m in enumerate(n)]
    p = torch.rand((count, len(n) + 2), dtype=torch.float64, device="cuda", generator=gen)
    for q in p:
        r2 = 0.0
        for a in range(len(n)):
            dx = (x[a] - TWO_PI * q[a]).abs()
            r2 = r2 + torch.minimum(dx, TWO_PI - dx) ** 2
        img = img + (0.2 + 0.8 * q[-1]) * torch.exp(-r2 / (2.0 * (0.2 + 0.3 * q[-2]) ** 2))
    k = _k(n)
    kk = sum(a * a for a in k).sqrt()
    keep = kk <= min(32, min(n) // 2 - 1)
    return _real(_spec(img, n) * keep, n).contiguous()


def _inputs(case, seed):
    """Template, velocities (true, linearisation point, direction) and an adjoint seed."""
    n, d, n_c = _grid(case), len(_grid(case)), case["n_c"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    small = min(n) // 2 - 1
    if d == 2:
        m = _blobs(n, gen)
    else:
        m = _band(n, gen, min(small, 48))[0]
        m = (m / m.std()).contiguous()
    kv = min(small, 8)
    v = _velocity(n, gen, n_c, 0.3, case["stokes"], kv)
    vt = _velocity(n, gen, n_c, 1.0, case["stokes"], kv)
    return dict(m=m, v_true=v, v=(0.6 * v).contiguous(), vt=vt,
                G=torch.randn(n, dtype=torch.float64, device="cuda", generator=gen))


def _pairs(case):
    """Shapes of a batch: 64^2, 128^2 and 256^2 at 4:2:1, their time steps, alternating weights."""
    out = []
    for size, n_t, share in ((64, 16, 4), (128, 32, 2), (256, 64, 1)):
        out += [((size, size), n_t, 1e-2 if i % 2 else 1e-3) for i in range(share * case["count"])]
    return out


def prepare(case, seed):
    op, n = case["op"], _grid(case)
    if op == "lockstep":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        makers, problems = {}, []
        for shape, n_t, beta in _pairs(case):
            if shape not in makers:
                makers[shape] = lib.Registration(shape, n_t)
            mT, v = _blobs(shape, gen), _velocity(shape, gen, 1, 0.3, False, 16)
            mR = torch.empty_like(mT)
            makers[shape].transport(v, mT, mR)
            problems.append(dict(n=shape, n_t=n_t, beta=beta, reg=1, mT=mT, mR=mR, v=torch.zeros_like(v)))
        for r in makers.values():
            r.close()
        return dict(op=op, problems=problems, precision=lib.REG_MIXED if case["mixed"] else lib.REG_FP64)
    s = _inputs(case, seed)
    if op == "autograd":
        R = autograd.make_transport(n, case["n_t"], case["n_c"])
        return dict(op=op, R=R, m=s["m"].requires_grad_(), v=s["v"].requires_grad_(), G=s["G"])
    R = lib.Registration(n, case["n_t"], case["n_c"], case["beta"], case["reg"], case["stokes"],
                         lib.REG_MIXED if case["mixed"] else lib.REG_FP64, case["ckpt"],
                         hessian=lib.REG_HESS_NEWTON if case["newton"] else lib.REG_HESS_GN)
    if op == "transport":
        return dict(op=op, R=R, v=s["v"], m=s["m"], out=torch.empty_like(s["m"]))
    if op == "precond":
        return dict(op=op, R=R, r=s["vt"], out=torch.empty_like(s["vt"]))
    mR = torch.empty_like(s["m"])
    R.transport(s["v_true"], s["m"], mR)
    R.set_images(s["m"], mR)
    out = torch.empty_like(s["vt"])
    if op == "gradient":
        return dict(op=op, R=R, v=s["v"], out=out)
    R.linearize(s["v"])
    return dict(op=op, R=R, vt=s["vt"], out=out, mixed=case["mixed"])


def run(state):
    op = state["op"]
    if op == "hessvec":
        state["R"].hessvec(state["vt"], state["out"])
        return state["out"].float() if state["mixed"] else state["out"]
    if op == "gradient":
        J = state["R"].gradient(state["v"], state["out"])
        return dict(g=state["out"], J=J)
    if op == "transport":
        state["R"].transport(state["v"], state["m"], state["out"])
        return state["out"]
    if op == "precond":
        state["R"].precond(state["r"], state["out"])
        return state["out"]
    if op == "autograd":
        m1 = autograd.transport(state["m"], state["v"], state["R"])
        gm, gv = torch.autograd.grad(m1, (state["m"], state["v"]), state["G"])
        return dict(m1=m1.detach(), gm=gm, gv=gv)
    for p in state["problems"]:
        p["v"].zero_()
    lib.solve_lockstep(state["problems"], state["precision"], max_outer=3)
    # one output per shape: the solutions of its pairs
    by = {}
    for p in state["problems"]:
        by.setdefault("v%d" % p["n"][0], []).append(p["v"])
    return {k: torch.stack(v).float() if state["precision"] == lib.REG_MIXED else torch.stack(v) for k, v in by.items()}


# ----------------------------------------------------------------------------------------------------------
# what one pass cannot do without
# ----------------------------------------------------------------------------------------------------------
def _stage(n):
    """Operations of one Heun stage: a forward and an inverse transform per axis, and the update."""
    N = math.prod(n)
    return N * (sum(5.0 * math.log2(m) for m in n) + 4.0 * len(n) + 4.0)


def work(case):
    n, n_c, op, n_t = _grid(case), case["n_c"], case["op"], case["n_t"]
    N, d = math.prod(n), len(_grid(case))
    vec = 8.0 * n_c * d * N
    ffts = n_c * d * N * 5.0 * math.log2(N)  # one coefficient vector to Fourier space and back
    if op == "lockstep":
        # per pair four gradients and objectives and about nine matvecs, four stages per step and sweep pair
        flops = sum((4 * 6.0 + 9 * 4.0) * nt * _stage(s) for s, nt, _ in _pairs(case))
        return dict(bytes=sum(32.0 * math.prod(s) for s, _, _ in _pairs(case)), flops=flops)
    if op == "precond":
        return dict(bytes=2 * vec, flops=ffts)
    if op == "transport":
        return dict(bytes=vec + 16.0 * N, flops=2.0 * n_t * _stage(n))
    if op == "autograd":  # state, then state and adjoint; inputs v, m, G; outputs m_1 and both gradients
        return dict(bytes=2 * vec + 32.0 * N, flops=6.0 * n_t * _stage(n))
    if op == "gradient":  # state and adjoint, again the state between checkpoints
        return dict(bytes=2 * vec + 16.0 * N, flops=(6.0 if case["ckpt"] else 4.0) * n_t * _stage(n) + ffts)
    # matvec: incremental state and adjoint; the state twice more between checkpoints; Newton: the adjoint and
    # the source of the incremental adjoint too. Reads the direction, the velocity and the stored states.
    stages = 4.0 + (4.0 if case["ckpt"] else 0.0) + (3.0 if case["newton"] else 0.0)
    w = 4.0 if case["mixed"] else 8.0
    stored = w * N * (n_t // case["ckpt"] + 1 if case["ckpt"] else (n_t + 1) * d)
    return dict(bytes=2 * vec + w * n_c * d * N + stored, flops=stages * n_t * _stage(n) + ffts)


# ----------------------------------------------------------------------------------------------------------
# the same in 64 bits with torch
# ----------------------------------------------------------------------------------------------------------
class _Exact:
    def __init__(self, case):
        self.case, self.n, self.n_t, self.n_c = case, _grid(case), case["n_t"], case["n_c"]
        self.d, self.h = len(self.n), 1.0 / case["n_t"]
        self.k = _k(self.n)
        self.km = [torch.where(x.abs() == self.n[a] // 2, torch.zeros_like(x), x) for a, x in enumerate(self.k)]
        kk = sum(x * x for x in self.k)
        self.a = kk if case["reg"] == 1 else kk * kk
        one = lambda m: 0.0 if m % 2 else 2.0 / (1.0 - m * m)  # noqa: E731
        self.C = torch.tensor([[0.25 * (one(a + b) + one(abs(a - b))) for b in range(self.n_c)]
                               for a in range(self.n_c)], dtype=torch.float64, device="cuda")
        self.T = [[math.cos(l * math.acos(max(-1.0, min(1.0, 2.0 * j / self.n_t - 1.0)))) for l in range(self.n_c)]
                  for j in range(self.n_t + 1)]

    def grad(self, u):
        U = _spec(u, self.n)
        return torch.stack([_real(1j * k * U, self.n) for k in self.km])

    def div(self, w):
        return _real(sum(1j * self.km[i] * _spec(w[i], self.n) for i in range(self.d)), self.n)

    def at(self, v, j):
        return sum(self.T[j][l] * v[l] for l in range(self.n_c))

    def state(self, v, m):
        """m at every node."""
        out = [m]
        for j in range(self.n_t):
            k1 = -(self.at(v, j) * self.grad(m)).sum(0)
            k2 = -(self.at(v, j + 1) * self.grad(m + self.h * k1)).sum(0)
            m = m + 0.5 * self.h * (k1 + k2)
            out.append(m)
        return out

    def adjoint(self, v, lam, source=None):
        """lam at every node, backward from t = 1; source: the extra right-hand side at node j."""
        out = [lam]
        s = (lambda j: 0.0) if source is None else source
        for j in range(self.n_t - 1, -1, -1):
            k1 = self.div(self.at(v, j + 1) * lam) + s(j + 1)
            k2 = self.div(self.at(v, j) * (lam + self.h * k1)) + s(j)
            lam = lam + 0.5 * self.h * (k1 + k2)
            out.append(lam)
        return out[::-1]

    def force(self, terms):
        """sum_j w_j T_l(t_j) terms(j), trapezoid weights."""
        f = 0.0
        for j in range(self.n_t + 1):
            w = self.h * (0.5 if j in (0, self.n_t) else 1.0)
            t = terms(j)
            f = f + torch.stack([w * self.T[j][l] * t for l in range(self.n_c)])
        return f

    def regularised(self, v):
        """beta (C x A) v."""
        return self.case["beta"] * torch.einsum("ab,b...->a...", self.C, _real(self.a * _spec(v, self.n), self.n))

    def tail(self, v, f):
        if self.case["stokes"]:
            f = torch.stack([_leray(x, self.n) for x in f])
        return self.regularised(v) + f


def exact(case, seed):
    if case["op"] == "lockstep":
        return None
    s, E = _inputs(case, seed), _Exact(case)
    v, m, op = s["v"], s["m"], case["op"]
    if op == "precond":
        a = E.a.clone()
        zero = (0,) * E.d
        a[zero] = 1.0
        R = _spec(s["vt"], E.n) / (case["beta"] * a)
        R[(slice(None), slice(None)) + zero] *= case["beta"]
        return torch.einsum("ab,b...->a...", torch.linalg.inv(E.C), _real(R, E.n))
    if op == "transport":
        return E.state(v, m)[-1]
    if op == "autograd":
        m, v = m.requires_grad_(), v.requires_grad_()
        m1 = E.state(v, m)[-1]
        gm, gv = torch.autograd.grad(m1, (m, v), s["G"])
        return dict(m1=m1.detach(), gm=gm, gv=gv)
    mR = E.state(s["v_true"], m)[-1]
    ms = E.state(v, m)
    if op == "gradient":
        lam = E.adjoint(v, mR - ms[-1])
        g = E.tail(v, E.force(lambda j: lam[j] * E.grad(ms[j])))
        hd = math.prod(TWO_PI / x for x in E.n)
        J = 0.5 * hd * (mR - ms[-1]).square().sum() + 0.5 * hd * (v * E.regularised(v)).sum()
        return dict(g=g, J=float(J))
    vt = s["vt"]
    mt = [torch.zeros_like(m)]
    for j in range(E.n_t):
        x = mt[-1]
        k1 = -(E.at(v, j) * E.grad(x)).sum(0) - (E.at(vt, j) * E.grad(ms[j])).sum(0)
        k2 = (-(E.at(v, j + 1) * E.grad(x + E.h * k1)).sum(0) - (E.at(vt, j + 1) * E.grad(ms[j + 1])).sum(0))
        mt.append(x + 0.5 * E.h * (k1 + k2))
    if not case["newton"]:
        lt = E.adjoint(v, -mt[-1])
        return E.tail(vt, E.force(lambda j: lt[j] * E.grad(ms[j])))
    lam = E.adjoint(v, mR - ms[-1])
    lt = E.adjoint(v, -mt[-1], lambda j: E.div(E.at(vt, j) * lam[j]))
    return E.tail(vt, E.force(lambda j: lt[j] * E.grad(ms[j]) + lam[j] * E.grad(mt[j])))
