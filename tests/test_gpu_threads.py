"""Two contexts driven from two host threads, each on its own stream, whose launches need different amounts of shared
memory: the opt-in belongs to a kernel, so neither context may lower it for the other.

Operators: translations of order 60 (two drops close enough for it among far ones) and of low order. Row builds:
degrees 56 and 8. Both at once, results equal to those of the contexts alone.
"""
import threading

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def suspension(p, n, spacing):
    rng = np.random.default_rng(n)
    at = [spacing * np.array([i % 3, i // 3 % 3, i // 9], float) for i in range(n)]
    return [inputs.perturbed_coef(p, rng, 1.0, c, amp=0.02) for c in at], [inputs.random_density(p, rng, 3) for _ in range(n)]


def worker(S, p, n, spacing, rounds, rebuild, out, other, key):
    """Applications (and row builds) until the slower of the two threads has done its rounds."""
    try:
        with torch.cuda.stream(torch.cuda.Stream()):
            shapes, dens = suspension(p, n, spacing)
            up = lambda parts: torch.tensor(np.concatenate([a.ravel() for a in parts]), device="cuda")
            x, f = up(shapes), up(dens)
            ctx = S.Context(precision=S.DF64)
            ctx.set_near(False)
            ctx.set_drops([p] * n, x)
            r = torch.empty_like(f)
            ctx.eval_stokes(f, None, r)
            torch.cuda.current_stream().synchronize()
            out[key, "alone"] = r.cpu().numpy()
            other["start"].wait()
            k = 0
            while k < rounds or not other["done"].is_set():
                if rebuild:
                    ctx.set_drops([p] * n, x)
                ctx.eval_stokes(f, None, r)
                k += 1
                if k == rounds:
                    other["mine"].set()
                if k >= 4000:
                    break
            torch.cuda.current_stream().synchronize()
            out[key, "together"] = r.cpu().numpy()
            ctx.close()
    except Exception as e:  # noqa: BLE001 - the thread's failure is the test's
        out[key, "error"] = e
        other["start"].abort()
    finally:
        other["mine"].set()


@pytest.mark.parametrize("what", ["operators", "rows"])
def test_contexts_of_two_threads_do_not_disturb_each_other(what):
    import paper_1811_10270_gb300 as S
    S.lib()
    start, a, b = threading.Barrier(2), threading.Event(), threading.Event()
    jobs = {"large": (14, 27, 3.0, 300, False), "small": (14, 27, 9.0, 300, False)} if what == "operators" else \
        {"large": (56, 1, 3.0, 5, True), "small": (8, 1, 3.0, 50, True)}
    out = {}
    threads = [threading.Thread(target=worker, args=(S, *jobs[k], out, {"start": start, "mine": m, "done": d}, k))
               for k, m, d in (("large", a, b), ("small", b, a))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert not any(t.is_alive() for t in threads)
    for k in jobs:
        if (k, "error") in out:
            raise out[k, "error"]
        np.testing.assert_array_equal(out[k, "alone"], out[k, "together"])
