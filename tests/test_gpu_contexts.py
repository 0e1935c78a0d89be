"""Contexts beside other work: fresh ones used at once, and what surrounds the
streams they work on."""
import numpy as np
import pytest

from paper_1408_6299_gb300 import lib
from gpu_util import empty

pytestmark = pytest.mark.gpu


def field(n, seed):
    """Low modes of unit size."""
    import torch
    axes = [torch.arange(m, device="cuda", dtype=torch.float64) * (2 * np.pi / m) for m in n]
    x = torch.meshgrid(*axes, indexing="ij")
    r = np.random.default_rng(seed)
    return sum(torch.sin(r.integers(1, 4) * xi + r.uniform(0, 6)) * torch.cos(x[0] + r.uniform(0, 6)) for xi in x) / len(n)


def coefs(n, n_c, size, seed=0):
    import torch
    return torch.stack([torch.stack([field(n, seed + 10 * l + i) for i in range(len(n))]) for l in range(n_c)]) * size


def test_fresh_context_reads_complete_tables():
    # A context on a non-blocking stream, used as soon as it exists: its tables must have arrived. The refined
    # det F makes such a context in the middle of a call.
    import torch
    n, n_c = (64, 32), 3
    v, u = coefs(n, n_c, 0.1), field(n, 7)
    ref = None
    for k in range(20):
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        R = lib.Registration(n, 4, n_c, 1e-2, lib.REG_H2, True, lib.REG_FP64, 0, stream=s.cuda_stream)
        det, z, m1 = empty((128, 64)), empty(R.coef_shape()), empty(n)
        R.detF_refined(v, 1, 2, det)
        R.precond(v, z)
        R.transport(v, u, m1)
        out = [t.clone() for t in (det, z, m1)]
        ref = ref or out
        assert all(torch.equal(a, b) for a, b in zip(out, ref)), k
        R.close()
