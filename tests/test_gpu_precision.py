"""Rounding of single steps, where a norm over the whole result does not show it."""
import numpy as np
import pytest

from paper_1408_6299_gb300 import lib
from gpu_util import empty

pytestmark = pytest.mark.gpu


def pattern(n, k):
    """cos(k x) for k = n/4 (1, 0, -1, 0) and k = n/2 (1, -1): exact values."""
    import torch
    return torch.tensor([1.0, 0.0, -1.0, 0.0] if 4 * k == n else [1.0, -1.0], dtype=torch.float64,
                        device="cuda").repeat(4 * k if 4 * k != n else k)[:n]


@pytest.mark.parametrize("n_c", [1, 2])
@pytest.mark.parametrize("reg", [lib.REG_H1, lib.REG_H2])
@pytest.mark.parametrize("n", [(8, 32), (16, 128), (8, 32, 64)], ids=["8x32", "16x128", "8x32x64"])
def test_preconditioner_factor_rounded_as_one_division(n, reg, n_c):
    # One mode at a time, its part of the result taken out exactly: 1 / (beta a), rounded as a product and a division,
    # with one unit for the way through the transforms (fixed point, some 2^-60 of the mode).
    import itertools
    import math

    import torch
    R = lib.Registration(n, 4, n_c, 1.0, reg, False, lib.REG_FP64, 0)
    z = empty(R.coef_shape())
    for beta in (1e-3, 7e-5, 0.3, 1.1e-2, 3e-6):
        R.set_beta(beta)
        # (a Nyquist mode of the last axis shares its slot with k = 0 there and takes their difference)
        for quarter in itertools.product(*[(True, False)] * (len(n) - 1), (True,)):
            k = [m // 4 if q else m // 2 for m, q in zip(n, quarter)]
            u = torch.ones(n, dtype=torch.float64, device="cuda")
            for a, (m, q) in enumerate(zip(n, k)):
                u = u * pattern(m, q).reshape([-1 if b == a else 1 for b in range(len(n))])
            r = u.expand(R.coef_shape()).contiguous()
            R.precond(r, z)
            kk = float(sum(q * q for q in k)) ** reg
            factor = 1.0 / (beta * kk)
            for i in range(len(n)):  # the inverse Gram matrix has a row (1, 0)
                got = math.fsum((z[0, i] * u).flatten().tolist()) / float(u.abs().sum())  # the mode alone
                assert abs(got - factor) <= np.spacing(factor), (beta, k, (got - factor) / np.spacing(factor))
    R.close()


ROW_GRIDS = [(8, 8), (16, 16), (64, 64), (16, 128), (32, 256), (8, 512), (8, 16, 32), (64, 64, 64), (256, 128, 128),
             (512, 512, 16), (128, 512, 64), (128, 256, 256), (64, 256, 512)]
ROW_IDS = ["x".join(map(str, n)) for n in ROW_GRIDS]


def uneven_rows(n, ratio, seed):
    """White noise whose rows differ in size by `ratio` (either one of a pair the larger), some of them zero."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randn(n, generator=gen, dtype=torch.float64, device="cuda").reshape(-1, n[-1])
    size = torch.ones(u.shape[0], dtype=torch.float64, device="cuda")
    size[1::4] = ratio
    size[2::4] = ratio
    if u.shape[0] >= 16:
        size[5::16] = 0
        size[10::16] = 0
    return (u * size[:, None]).reshape(n).contiguous()


def last_axis_velocity(n, size, seed):
    """A velocity along the last axis alone: rows do not meet."""
    import torch
    r = np.random.default_rng(seed)
    x = torch.arange(n[-1], device="cuda", dtype=torch.float64) * (2 * np.pi / n[-1])
    v = torch.zeros((1, len(n)) + n, dtype=torch.float64, device="cuda")
    v[0, -1] = size * (torch.sin(x + r.uniform(0, 6)) + 0.5 * torch.cos(2 * x + r.uniform(0, 6)))
    return v


def row_error(a, b):
    """The largest error of a row, relative to that row; zero rows have to be zero."""
    import torch
    a, b = a.reshape(-1, a.shape[-1]), b.reshape(-1, b.shape[-1])
    size = b.norm(dim=1)
    assert not bool(a[size == 0].any())
    return float(((a - b).norm(dim=1)[size > 0] / size[size > 0]).max())


@pytest.mark.parametrize("n", ROW_GRIDS, ids=ROW_IDS)
def test_rows_keep_their_own_accuracy(n):
    # two Heun steps against torch's FFT along the rows; the tolerance of the line tests, here for every row
    import torch
    k = torch.fft.fftfreq(n[-1], 1.0 / n[-1], device="cuda", dtype=torch.float64)
    k[n[-1] // 2] = 0
    d = lambda y: torch.fft.ifft(torch.fft.fft(y) * (1j * k)).real  # noqa: E731
    n_t = 2
    v, u = last_axis_velocity(n, 0.4 * n_t / (n[-1] / 2), 3), uneven_rows(n, 2.0 ** -27, 1)
    R = lib.Registration(n, n_t, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    m1, gm = empty(n), empty(n)
    R.transport(v, u, m1)
    R.transport_adjoint(v, u, u, None, gm)
    R.close()
    for got, rhs in ((m1, lambda y: -v[0, -1] * d(y)), (gm, lambda y: d(y * v[0, -1]))):
        y, h = u, 1.0 / n_t
        for _ in range(n_t):
            k1 = rhs(y)
            y = y + 0.5 * h * (k1 + rhs(y + h * k1))
        assert row_error(got, y) < 1e-12


@pytest.mark.parametrize("ckpt", [0, 2])
@pytest.mark.parametrize("n", ROW_GRIDS, ids=ROW_IDS)
def test_rows_keep_their_own_accuracy_mixed(n, ckpt):
    # the force along the rows, lambda~ dm/dz, of a matvec whose velocities follow the rows: the mixed path's
    # tolerance against double precision, here for every row (beta: no regularisation beside it)
    import torch
    n_t, out = 4, []
    v, vt = last_axis_velocity(n, 0.4 * n_t / (n[-1] / 2), 3), last_axis_velocity(n, 1.0, 4)
    mT = uneven_rows(n, 2.0 ** -20, 1)
    for precision in (lib.REG_FP64, lib.REG_MIXED):
        R = lib.Registration(n, n_t, 1, 1e-60, lib.REG_H1, False, precision, ckpt)
        R.set_images(mT, mT)
        R.linearize(v)
        H = empty(R.coef_shape())
        R.hessvec(vt, H)
        out.append(H[0, -1].clone())
        R.close()
        torch.cuda.empty_cache()
    zero = mT.reshape(-1, n[-1]).norm(dim=1) == 0  # the tail leaves 1e-60 of the other rows in them
    for o in out:
        o.reshape(-1, n[-1])[zero] *= (o.reshape(-1, n[-1])[zero].abs() > 1e-50)
    assert row_error(out[1], out[0]) < 1e-5
