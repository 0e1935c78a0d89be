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


LEGACY, PER_THREAD = 1, 2  # cudaStreamLegacy, cudaStreamPerThread


@pytest.mark.parametrize("handle", [LEGACY, PER_THREAD], ids=["legacy", "per-thread"])
def test_special_stream_handles(handle):
    # launched, captured and replayed; the inputs are written on the NULL stream just before
    import torch
    n = (32, 32)
    v, u = coefs(n, 1, 0.1), field(n, 7)
    R = lib.Registration(n, 6, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0, stream=handle)
    one, g1, H1 = empty(n), empty(R.coef_shape()), empty(R.coef_shape())
    R.set_images(u, field(n, 8))
    R.transport(v, u, one)
    R.gradient(v, g1)
    R.hessvec(v, H1)
    for k in range(1, 5):
        x, m1, g, H = u.clone(), empty(n), empty(R.coef_shape()), empty(R.coef_shape())
        x.mul_(2.0 ** k)  # exact, and transport is linear in the image
        if handle == PER_THREAD:
            torch.cuda.synchronize()
        R.transport(v, x, m1)
        R.gradient(v, g)
        R.hessvec(v, H)
        assert torch.equal(m1, one * 2.0 ** k) and torch.equal(g, g1) and torch.equal(H, H1), k
    R.close()


def test_stream_shared_with_other_threads():
    # Two contexts and a counter, each in its own thread, on one stream. The contexts are made to capture again
    # and again; what the others enqueue meanwhile has to run once, and their synchronisations to succeed.
    import threading

    import torch
    n = (32, 32)
    s = torch.cuda.Stream()
    v, u = coefs(n, 1, 0.1), field(n, 7)
    torch.cuda.synchronize()
    refs, outs, errors, stop = {}, {0: [], 1: []}, [], threading.Event()
    for n_t in (4, 6):
        R = lib.Registration(n, n_t, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
        refs[n_t] = empty(n)
        R.transport(v, u, refs[n_t])
        R.close()
    counter = torch.zeros(1024, dtype=torch.float64, device="cuda")
    bufs = {w: [torch.empty_like(u) for _ in range(120)] for w in outs}
    torch.cuda.synchronize()

    def guard(f):
        def go():
            try:
                f()
            except BaseException as e:
                errors.append(repr(e))
        return threading.Thread(target=go)

    def context(w):
        def go():
            R = lib.Registration(n, 4, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0, stream=s.cuda_stream)
            for i, m1 in enumerate(bufs[w]):
                if i % 4 == 0:  # each setting twice launched, captured and replayed
                    R.set_time_steps(6 if R.n_t == 4 else 4)
                R.transport(v, u, m1)
                outs[w].append(R.n_t)
            R.close()
        return go

    added = [0]

    def count():
        with torch.cuda.stream(s):
            while not stop.is_set():
                counter.add_(1.0)
                added[0] += 1
                if added[0] % 64 == 0:
                    s.synchronize()

    workers, other = [guard(context(w)) for w in outs], guard(count)
    other.start()
    for t in workers:
        t.start()
    for t in workers:
        t.join()
    stop.set()
    other.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert added[0] and bool((counter == float(added[0])).all())
    for w in outs:
        for m1, n_t in zip(bufs[w], outs[w]):
            assert torch.equal(m1, refs[n_t]), (w, n_t)


def test_last_problem_of_a_stack_keeps_its_beta():
    # seven of eight stacked problems start at their minimum, so the eighth goes on in a stack of its own: the
    # iterates of that problem solved as a stack of one, bit for bit
    import torch
    n = (32, 32)
    u, mR = field(n, 7), empty(n)
    M = lib.Registration(n, 8, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    M.transport(coefs(n, 1, 0.2), u, mR)
    M.close()

    def problem(ref, beta):
        return dict(n=n, n_t=8, beta=beta, mT=u, mR=ref, v=torch.zeros((1, 2) + n, dtype=torch.float64, device="cuda"))

    probs = [problem(u, 1e-1 if i else 1e-3) for i in range(8)]
    probs[5] = problem(mR, 1e-2)
    one = problem(mR, 1e-2)
    rep = lib.solve_lockstep(probs, lib.REG_FP64, grad_rtol=1e-3)[5]
    alone = lib.solve_lockstep([one], lib.REG_FP64, grad_rtol=1e-3)[0]
    for k in ("outer", "pcg_iters", "ls_trials", "status", "J"):
        assert rep[k] == alone[k], (k, rep[k], alone[k])
    assert torch.equal(probs[5]["v"], one["v"])


def test_call_refused_under_capture_leaves_nothing_half_done():
    # a call synchronises, so a capture of the caller's refuses it; what it set up meanwhile was only recorded
    import ctypes

    import torch
    drv = ctypes.CDLL("libcuda.so.1")
    n = (32, 64)
    r = coefs(n, 1, 1.0)
    ref, z = empty((1, 2) + n), empty((1, 2) + n)
    R = lib.Registration(n, 4, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    R.precond(r, ref)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    S = lib.Registration(n, 4, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0, stream=s.cuda_stream)
    graph = ctypes.c_void_p()
    assert drv.cuStreamBeginCapture_v2(ctypes.c_void_p(s.cuda_stream), 2) == 0  # relaxed
    try:
        with pytest.raises(lib.RegError):
            S.precond(r, z)
    finally:
        assert drv.cuStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) != 0
    torch.cuda.synchronize()
    S.precond(r, z)
    assert torch.equal(z, ref)
    S.close()
    R.close()


def test_launches_counted_alike_by_one_and_by_many_workers():
    # eight problems of one shape and eight weights: one context each, whoever solves it
    import torch
    n = (32, 32)
    u, mR = field(n, 7), empty(n)
    M = lib.Registration(n, 8, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
    M.transport(coefs(n, 1, 0.2), u, mR)
    M.close()

    def launches(workers):
        probs = [dict(n=n, n_t=8, beta=1e-2 * (1 + i), mT=u, mR=mR, v=torch.zeros((1, 2) + n, dtype=torch.float64,
                                                                                 device="cuda")) for i in range(8)]
        before = lib.launch_count()
        lib.solve_batched(probs, lib.REG_FP64, workers=workers, grad_rtol=1e-3)
        return lib.launch_count() - before

    launches(1)  # settles the autotuner
    one = launches(1)
    assert one > 0
    for _ in range(3):
        assert launches(8) == one


@pytest.mark.parametrize("n_t,ckpt", [(20, 0), (20, 4), (20, 10), (9, 9)])
def test_newton_over_more_nodes_than_a_force_group(n_t, ckpt):
    # the rings of the backward sweep wrap; tolerances of the Newton parity tests
    from oracle import oracle as O
    from paper_1408_6299_gb300 import synth
    from gpu_util import cuda, host, pair, rel
    c = synth.stokes_3d(16, n_t=n_t, n_c=3)
    P = O.Problem(c["n"], n_t, c["n_c"], c["beta"], c["reg"], c["stokes"])
    mR = P.state(c["v_true"], c["mT"])[-1]
    v = 0.5 * c["v_true"]
    ref = P.hessvec_newton(v, c["mT"], mR, c["vt"])
    for precision, tol in ((lib.REG_FP64, 1e-10), (lib.REG_MIXED, 1e-5)):
        R, _ = pair(c, precision=precision, ckpt=ckpt)
        R.set_hessian(lib.REG_HESS_NEWTON)
        R.set_images(cuda(c["mT"]), cuda(mR))
        R.linearize(cuda(v))
        Hv = empty(R.coef_shape())
        for _ in range(3):  # launched, captured and replayed
            R.hessvec(cuda(c["vt"]), Hv)
            assert rel(host(Hv), ref) < tol
        R.close()


# grids whose rings hold fewer than eight nodes: full Newton 3 and 1, discrete adjoint 4, trapezoid 3
@pytest.mark.parametrize("what,n,n_t,ckpt", [
    ("newton", (256, 256, 256), 7, 0), ("newton", (512, 256, 256), 5, 0), ("newton", (256, 256, 256), 8, 4),
    ("adjoint", (512, 256, 256), 9, 0), ("gradient", (512, 512, 512), 5, 0)])
def test_rings_bounded_by_memory(what, n, n_t, ckpt):
    # fields that do not vary along the first axis: the same on 8 points there, where the rings hold eight nodes
    import torch
    small = (8,) + n[1:]
    d, size = 3, 0.4 * n_t / (3 * max(n) / 2)
    out = []
    for m in (small, n):
        def make(seed, count=None):
            f = torch.stack([field(small[1:], seed + i) for i in range(count or 1)])
            f = f[:, None].expand((count or 1,) + m).contiguous()
            return f[None] if count else f[0]
        R = lib.Registration(m, n_t, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, ckpt,
                             quadrature=lib.REG_QUAD_DISCRETE if what == "adjoint" else lib.REG_QUAD_TRAPEZOID,
                             hessian=lib.REG_HESS_NEWTON if what == "newton" else lib.REG_HESS_GN)
        u, v, res = make(7), make(20, d) * size, empty((1, d) + m)
        if what == "adjoint":
            gm = empty(m)
            R.transport_adjoint(v, u, make(8), res, gm)
            out.append([res[0, :, :8].clone(), gm[:8].clone()])
        else:
            R.set_images(u, make(8))
            if what == "gradient":
                R.gradient(v, res)
            else:
                R.linearize(v)
                R.hessvec(make(30, d), res)
            out.append([res[0, :, :8].clone()])
        R.close()
        del R, u, v, res
        torch.cuda.empty_cache()
    for a, b in zip(*out):
        assert float((a - b).norm() / b.norm()) < 1e-10


def test_newton_matvec_memory():
    # 59 fields of a store-all context with two steps where the rings are bounded; the matvec held 58 before its
    # body force was summed in groups, and five more fields than that are allowed here
    import torch
    n = (256, 256, 256)
    u, v = field(n, 7), coefs(n, 1, 0.001)
    Hv = torch.empty_like(v)
    R = lib.Registration(n, 2, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0, hessian=lib.REG_HESS_NEWTON)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    R.set_images(u, u)
    R.linearize(v)
    R.hessvec(v, Hv)
    assert (free - torch.cuda.mem_get_info()[0]) / (8.0 * u.numel()) < 63
    R.close()


def stack(n, count, n_t=2):
    """count problems of one shape, the first two the same in every stack."""
    import torch
    out = []
    for i in range(count):
        u = field(n, 7 + i)
        out.append(dict(n=n, n_t=n_t, beta=1e-2, mT=u, mR=torch.roll(u, 1, 0).contiguous(),
                        v=torch.zeros((1, 2) + n, dtype=torch.float64, device="cuda")))
    return out


TUNED_STACKS = r"""
import sys
sys.path[:0] = [%r, %r]
from test_gpu_contexts import stack
from paper_1408_6299_gb300 import lib
for count in (37, 39):  # on either side of the line between the plans, one rounded size
    lib.solve_lockstep(stack((256, 256), count), lib.REG_MIXED, max_outer=1)
"""


def test_tuner_keeps_the_plans_apart(tmp_path):
    import json
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    cache = tmp_path / "tune_cache.json"
    subprocess.run([sys.executable, "-c", TUNED_STACKS % (os.path.dirname(here), here)], check=True, timeout=600,
                   env=dict(os.environ, REG_TUNE_CACHE=str(cache)))
    keys = [k for k in json.loads(cache.read_text()) if "cols|plain" in k and k.endswith("|f32|L256|n4194304")]
    assert len(keys) == 2, keys


def test_double_precision_bits_do_not_depend_on_the_stack():
    # the larger stack alone would run wide plans
    import torch
    n, vs = (256, 256), []
    for count in (2, 80):
        probs = stack(n, count)
        lib.solve_lockstep(probs, lib.REG_FP64, max_outer=1)
        vs.append([p["v"] for p in probs[:2]])
    for a, b in zip(*vs):
        assert bool(a.any()) and torch.equal(a, b)


TUNED_TRANSPORT = r"""
import sys
sys.path[:0] = [%r, %r]
from test_gpu_contexts import coefs, empty, field
from paper_1408_6299_gb300 import lib
n = (512, 512)
R = lib.Registration(n, 4, 1, 1e-2, lib.REG_H1, False, lib.REG_FP64, 0)
R.transport(coefs(n, 1, 0.01), field(n, 7), empty(n))
"""


def test_tuner_takes_the_shorter_tile_each_time(tmp_path):
    # columns of 512 points in double precision: one line per block, with four of them a transport takes 1.3 times
    # as long
    import json
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    for k in range(3):
        cache = tmp_path / f"tune_cache_{k}.json"
        subprocess.run([sys.executable, "-c", TUNED_TRANSPORT % (os.path.dirname(here), here)], check=True, timeout=600,
                       env=dict(os.environ, REG_TUNE_CACHE=str(cache)))
        picks = [v for key, v in json.loads(cache.read_text()).items() if "cols|plain" in key and "|f64|L512|" in key]
        assert picks == [0], picks
