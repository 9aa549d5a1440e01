"""The memory of a gradient with a kept last segment: the backward pass gives the
segment up once it is swept, so that it never holds more than one segment's
states, and a forward pass alone need not keep it."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

N, STEPS, CHECKPOINT = 20_000, 12, 4
STATE = 6 * N * 8                # bytes of one (x, v')
SEGMENT = CHECKPOINT * STATE


@pytest.fixture(scope="module")
def rollout():
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import adjoint as AD, p3t as P
    s = disks.adjoint_disk(N, 7)
    x = torch.as_tensor(np.stack([s["x"], s["y"], s["z"]])).cuda()
    v = torch.as_tensor(np.stack([s["vx"], s["vy"], s["vz"]])).cuda()
    m = torch.as_tensor(s["m"]).cuda()
    prm = P.Params(precision=P.P3T_MIXED)
    ro = AD.cutoffs(prm, x, v, m)
    run = AD.SoftKDK(prm, N, STEPS, CHECKPOINT)
    yield AD, run, (x, v, m, ro)
    run.close()


def _peak(f):
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    base = torch.cuda.memory_allocated()
    out = f()
    torch.cuda.synchronize()
    return torch.cuda.max_memory_allocated() - base, out


def test_backward_holds_one_segment(rollout):
    AD, run, a = rollout
    lam = torch.ones_like(a[0])

    def sweep(kept):
        tape = run.forward(*a)[2]
        if not kept:
            tape["last"] = None
        return run.backward(tape, lam, lam)
    kept, g = _peak(lambda: sweep(True))
    recomputed, h = _peak(lambda: sweep(False))
    # the states of one segment either way; a state or two of temporaries more
    assert kept <= recomputed + 2 * STATE
    assert all(torch.equal(p, q) for p, q in zip(g, h))


def test_forward_alone_keeps_nothing(rollout):
    AD, run, a = rollout
    whole, (_, _, tape) = _peak(lambda: run.forward(*a))
    less, (_, _, bare) = _peak(lambda: run.forward(*a, keep_last=False))
    assert bare["last"] is None and less <= whole - SEGMENT + STATE
    lam = torch.ones_like(a[0])
    g, h = run.backward(tape, lam, lam), run.backward(bare, lam, lam)
    assert all(torch.equal(p, q) for p, q in zip(g, h))
    # a differentiable call without a graph
    x = a[0].clone().requires_grad_()

    def call(grad):
        with torch.set_grad_enabled(grad):
            return AD.soft_kdk(x, a[1], a[2], a[3], run)
    on, y = _peak(lambda: call(True))
    off, z = _peak(lambda: call(False))
    assert torch.equal(y[0], z[0]) and not z[0].requires_grad
    assert off <= on - SEGMENT + STATE
