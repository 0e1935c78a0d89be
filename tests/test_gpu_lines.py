"""The line transforms behind the transport stages, at the sizes where their
plans change: every axis length on rows and columns, few lines (one or two per
block), full narrow blocks, wide plans and paired columns, one and two axis
lengths per stage; and what fixed-point lines could get wrong: magnitudes far
from one, zero lines, infinities and NaN.

FP64 results are compared with Heun steps on torch's double-precision FFT. A
step adds h v . grad u with |h v k| <= 0.4, and a derivative's rounding error
is below 1e-15 log2(L) of its largest mode, so 1e-12 has two digits to spare.
Mixed results are compared with FP64 ones to the 1e-5 of the mixed path.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1408_6299_gb300 import lib, synth
from gpu_util import cuda, empty, host, pair, rel

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12
MIXED_TOL = 1e-5

GRIDS = [
    (8, 8), (16, 8), (512, 64), (32, 512), (8, 16, 32), (64, 8, 512), (8, 512, 256),  # few lines
    (64, 64, 8), (128, 64, 16), (64, 128, 32), (64, 64, 64), (64, 64, 128), (32, 128, 256), (16, 256, 512),  # narrow
    (512, 512, 16), (512, 256, 32), (512, 512, 64), (64, 512, 256), (256, 128, 512), (256, 256, 128),  # wide
]
IDS = ["x".join(map(str, n)) for n in GRIDS]


def white(n, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, generator=gen, dtype=torch.float64, device="cuda")


def smooth(n, k, seed):
    """A unit-size field of low modes."""
    import torch
    axes = [torch.arange(m, device="cuda", dtype=torch.float64) * (2 * np.pi / m) for m in n]
    x = torch.meshgrid(*axes, indexing="ij")
    r = np.random.default_rng(seed)
    return sum(torch.sin(r.integers(1, k + 1) * xi + r.uniform(0, 6)) * torch.cos(x[0] + r.uniform(0, 6)) for xi in x) / len(n)


def velocity(n, size):
    import torch
    return torch.stack([smooth(n, 2, 40 + i) for i in range(len(n))])[None].mul_(size).contiguous()


def torch_cat(*t):
    import torch
    return torch.cat(t).contiguous()


def derivative(u, axis):
    import torch
    n = u.shape[axis]
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    k[n // 2] = 0
    shape = [1] * u.dim()
    shape[axis] = n
    return torch.fft.ifft(torch.fft.fft(u, dim=axis) * (1j * k.reshape(shape)), dim=axis).real


def heun(u, rhs, n_t):
    h = 1.0 / n_t
    for _ in range(n_t):
        k1 = rhs(u)
        u = u + 0.5 * h * (k1 + rhs(u + h * k1))
    return u


@pytest.mark.parametrize("n", GRIDS, ids=IDS)
def test_fp64_stages_match_fft(n):
    import torch
    d, n_t = len(n), 2
    v = velocity(n, 0.4 * n_t / (d * max(n) / 2))
    u = white(n, 1)
    R = lib.Registration(n, n_t, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    m1, gm = empty(n), empty(n)
    R.transport(v, u, m1)
    ref = heun(u, lambda y: -sum(v[0, i] * derivative(y, i) for i in range(d)), n_t)
    assert float((m1 - ref).norm() / ref.norm()) < FP64_TOL
    R.transport_adjoint(v, u, u, None, gm)
    ref = heun(u, lambda y: sum(derivative(y * v[0, i], i) for i in range(d)), n_t)
    assert float((gm - ref).norm() / ref.norm()) < FP64_TOL
    R.close()
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", GRIDS, ids=IDS)
def test_mixed_stages_match_fp64(n):
    import torch
    n_t = 2
    v = velocity(n, 0.4 * n_t / (len(n) * max(n) / 2))
    mT, mR, vt = smooth(n, 3, 7), smooth(n, 3, 8), velocity(n, 1.0)
    out = []
    for precision in (lib.REG_FP64, lib.REG_MIXED):
        R = lib.Registration(n, n_t, 1, 1e-2, lib.REG_H1, False, precision, 2 if min(n) >= 64 else 0)
        R.set_images(mT, mR)
        R.linearize(v)
        out.append(empty(R.coef_shape()))
        R.hessvec(vt, out[-1])
        R.close()
        torch.cuda.empty_cache()
    assert float((out[1] - out[0]).norm() / out[0].norm()) < MIXED_TOL


@pytest.mark.parametrize("n", [(16, 64), (64, 64, 64), (256, 256, 128)], ids=["16x64", "64c", "256x256x128"])
@pytest.mark.parametrize("e", [1000, 600, -600, -1000, -1040])
def test_magnitudes(n, e):
    # transport is linear in the image; at 2^-1040 values are subnormal, a spacing of 2^-34 of them
    import torch
    v = velocity(n, 0.4 / (len(n) * max(n) / 4))
    u = white(n, 2)
    u[1] = 0  # zero rows beside others
    R = lib.Registration(n, 2, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    a, b = empty(n), empty(n)
    R.transport(v, u, a)
    lo, hi = 2.0 ** (e // 2), 2.0 ** (e - e // 2)
    R.transport(v, u * lo * hi, b)
    back = b / lo / hi
    assert float((back - a).norm() / a.norm()) < (1e-8 if e == -1040 else FP64_TOL)
    R.transport(v, torch.zeros_like(u), b)
    assert not b.any()
    R.close()


@pytest.mark.parametrize("n", [(8, 16), (64, 256), (512, 512)], ids=["8x16", "64x256", "512x512"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_values_spread(n, bad):
    # one step: stage 1 spoils the row and the column of the point, stage 2 every line that meets them
    import torch
    u = white(n, 3)
    u[n[0] // 3, n[1] // 3] = bad
    R = lib.Registration(n, 1, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    m1 = empty(n)
    R.transport(velocity(n, 0.1), u, m1)
    assert not torch.isfinite(m1).any()
    R.close()


@pytest.mark.parametrize("n_t,ckpt", [(7, 0), (8, 0), (9, 3), (15, 5)])
def test_force_groups(n_t, ckpt):
    # the body force is summed over groups of time nodes: whole, partial and single-node groups
    n = (16, 32)
    r = np.random.default_rng(n_t)
    c = dict(n=n, n_t=n_t, n_c=3, beta=1e-2, reg=lib.REG_H2, stokes=True)
    mT, mR = synth.random_spectral_field(n, r, 4.0), synth.random_spectral_field(n, r, 4.0)
    v = np.stack([synth.velocity_field(n, r, 3, 0.2 / (l + 1)) for l in range(3)])
    vt = np.stack([synth.velocity_field(n, r, 3, 1.0) for _ in range(3)])
    for precision, tol in ((lib.REG_FP64, 1e-10), (lib.REG_MIXED, MIXED_TOL)):
        R, P = pair(c, precision=precision, ckpt=ckpt)
        R.set_images(cuda(mT), cuda(mR))
        g, Hv = empty(R.coef_shape()), empty(R.coef_shape())
        R.gradient(cuda(v), g)
        assert rel(host(g), P.gradient(v, mT, mR)[0]) < 1e-10
        for _ in range(3):  # launched, captured and replayed
            R.hessvec(cuda(vt), Hv)
            assert rel(host(Hv), P.hessvec(v, mT, vt)) < tol


@pytest.mark.parametrize("n,n_t", [((64, 32), 7), ((32, 32, 32), 6), ((256, 256, 128), 3)],
                         ids=["64x32", "32c", "256x256x128"])
def test_time_dependent_velocity(n, n_t):
    # nodes formed in groups of four (the last one partial), and one by one in the largest fields
    d = len(n)
    size = 0.2 * n_t / (d * max(n) / 2)
    v = torch_cat(velocity(n, size), velocity(n, 0.5 * size).flip(1))
    u = white(n, 5)
    R = lib.Registration(n, n_t, 2, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    m1 = empty(n)
    R.transport(v, u, m1)
    h = 1.0 / n_t

    def rhs(y, j):
        a = v[0] + (2.0 * j / n_t - 1.0) * v[1]
        return -sum(a[i] * derivative(y, i) for i in range(d))

    for j in range(n_t):
        k1 = rhs(u, j)
        u = u + 0.5 * h * (k1 + rhs(u + h * k1, j + 1))
    assert float((m1 - u).norm() / u.norm()) < FP64_TOL
    R.close()


@pytest.mark.parametrize("ckpt", [0, 3])
def test_replayed_sweeps_follow_their_inputs(ckpt):
    # inputs formed on the NULL stream just before each call, in changing buffers
    import torch
    n, n_t = (32, 32, 32), 6
    R = lib.Registration(n, n_t, 2, 1e-2, lib.REG_H1, False, lib.REG_MIXED, ckpt)
    R.set_images(smooth(n, 3, 7), smooth(n, 3, 8))
    v = torch.cat([velocity(n, 0.05), velocity(n, 0.02)])
    R.linearize(v)
    vt = torch.cat([velocity(n, 1.0), velocity(n, 0.5)])
    first, keep = empty(R.coef_shape()), []
    R.hessvec(vt, first)
    for k in range(1, 7):
        x, y = vt.clone(), empty(R.coef_shape())
        x.mul_(2.0 ** k)  # exact
        R.hessvec(x, y)
        keep.append((x, y))
        assert torch.equal(y, first * 2.0 ** k), k
    R.linearize(torch.flip(v, (0,)).contiguous())  # another point: the same sweeps, other states
    other = empty(R.coef_shape())
    R.hessvec(vt, other)
    fresh = lib.Registration(n, n_t, 2, 1e-2, lib.REG_H1, False, lib.REG_MIXED, ckpt)
    fresh.set_images(smooth(n, 3, 7), smooth(n, 3, 8))
    fresh.linearize(torch.flip(v, (0,)).contiguous())
    ref = empty(R.coef_shape())
    fresh.hessvec(vt, ref)
    assert torch.equal(other, ref) and not torch.equal(other, first)


@pytest.mark.parametrize("n", [(16, 16), (8, 16, 32)], ids=["16x16", "8x16x32"])
@pytest.mark.parametrize("n_c", [1, 3])
def test_views_at_odd_offsets(n, n_c):
    # arrays that start 8 bytes behind a 16-byte boundary give the same results
    import torch

    def odd(t):
        buf = torch.zeros(t.numel() + 1, dtype=torch.float64, device="cuda")[1:].view(t.shape)
        buf.copy_(t)
        assert buf.data_ptr() % 16 == 8
        return buf

    res = []
    for f in (lambda t: t, odd):
        R = lib.Registration(n, 4, n_c, 1e-2, lib.REG_H1, n_c > 1, lib.REG_FP64, 0)
        v = f(torch.cat([velocity(n, 0.1 / (l + 1)) for l in range(n_c)]))
        u = f(smooth(n, 3, 7))
        shape = R.coef_shape()
        out = [f(empty(s)) for s in (n, shape, shape, shape, shape, shape, n, (len(n),) + n, n, n, shape)]
        R.transport(v, u, out[0])
        R.set_images(u, f(smooth(n, 3, 8)))
        R.gradient(v, out[1])
        R.hessvec(v, out[2])
        R.precond(v, out[3])
        R.regularization(v, out[4])
        R.transport_adjoint(v, u, u, out[5], out[6])
        R.displacement(v, out[7])
        R.smooth(0.3, u, out[8])
        R.detF(v, 2, out[9])
        out[10].copy_(v)
        R.solve(out[10], max_outer=1)
        res.append([t.clone() for t in out] + [torch.tensor(R.cfl(v))])
    for a, b in zip(*res):
        assert torch.equal(a, b)
