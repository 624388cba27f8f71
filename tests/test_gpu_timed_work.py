"""The work of the timed pair sums is counted outside the events that time them.

With expansions the pairs that are summed directly are read back from the device. That happens once per geometry, kind
and precision and before anything of the application is queued: an application after it does not wait for the GPU, so
no host time lies between the events of its pair class.
"""
import time

import numpy as np
import pytest

import test_gpu_far as far
import test_gpu_far_close as close

pytestmark = pytest.mark.gpu


def test_counting_the_pairs_does_not_hold_up_timed_applications():
    import torch
    import paper_1811_10270_gb300 as S
    dev = torch.device("cuda")
    up = lambda parts: torch.tensor(np.concatenate([np.ravel(a) for a in parts]), device=dev)
    drops, dens = close.lattice(far.FINER)
    ctx = S.Context(precision=S.DF64)
    ctx.set_drops([p for p, _, _ in drops], up([x for _, x, _ in drops]), [lam for _, _, lam in drops])
    f = up(dens["f"])
    out = torch.empty_like(f)
    ctx.eval_stokes(f, None, out)
    ctx.set_timing(True)
    ctx.eval_stokes(f, None, out)
    work = ctx.kernel_work(S.K_PAIRS_FP64CLASS)
    nt, ns = [(p + 1) * (2 * p + 2) for p in far.FINER], [(2 * p + 2) * (4 * p + 4) for p in far.FINER]
    assert 0.0 < work < 0.9 * far.FLOPS["f"] * sum(t * (sum(ns) - s) for t, s in zip(nt, ns))
    torch.cuda._sleep(int(4e8))         # about 0.2 s of the GPU
    t0 = time.perf_counter()
    ctx.eval_stokes(f, None, out)
    queued = time.perf_counter() - t0
    torch.cuda.synchronize()
    assert queued < 0.1
    assert ctx.kernel_work(S.K_PAIRS_FP64CLASS) == 2.0 * work
    ctx.close()
