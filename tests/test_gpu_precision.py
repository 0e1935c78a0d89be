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
