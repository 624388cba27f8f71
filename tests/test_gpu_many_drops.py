"""Suspensions of many small drops: what set_drops does per pair of drops stays small beside what it does per drop."""
import time

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def lattice(n, p, spacing=2.6):
    rng = np.random.default_rng(n)
    k = int(np.ceil(n ** (1.0 / 3.0)))
    at = [spacing * np.array([i % k, i // k % k, i // k // k], float) for i in range(n)]
    return torch.tensor(np.concatenate([inputs.perturbed_coef(p, rng, 1.0, c, amp=0.02).ravel() for c in at]), device="cuda")


def test_set_drops_grows_with_the_drops_not_with_their_pairs():
    """Four times the drops, sixteen times the pairs: less than eight times the time (12 times where the pairs are
    classified one after the other on the host)."""
    import paper_1811_10270_gb300 as S
    took = []
    for n in (256, 1024):
        x = lattice(n, 4)
        ctx = S.Context(precision=S.FP32_COMP)
        best = np.inf
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ctx.set_drops([4] * n, x)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        ctx.close()
        took.append(best)
    assert took[1] < 8.0 * took[0], took
