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


@pytest.mark.parametrize("n,p,precision,kind,expanded", [
    (1024, 4, "FP32_COMP", "f", False), (1024, 4, "FP32_COMP", "fu", False), (128, 6, "FP32_COMP", "f", False),
    (1024, 4, "DF64", "fu", True), (256, 8, "FP32_COMP", "f", True), (64, 8, "DF64", "f", True)])
def test_expansions_are_taken_where_they_pay(n, p, precision, kind, expanded):
    """The direct work of an application against that of every pair: many small drops whose translations cost more
    than the sums they replace (2.6 times at the first size) are summed directly."""
    import paper_1811_10270_gb300 as S
    ctx = S.Context(precision=getattr(S, precision))
    ctx.set_near(False)
    ctx.set_drops([p] * n, lattice(n, p))
    nc, nt, ns = ctx.sizes()
    a, out = (torch.ones(3 * k, device="cuda", dtype=torch.float64) for k in (nc, nt))
    ctx.set_timing(True)
    ctx.eval_stokes(a, a if "u" in kind else None, out, S.OUT_GRID)
    work = sum(ctx.kernel_work(c) for c in (S.K_PAIRS, S.K_PAIRS_FP64CLASS))
    every = {"f": 29.0, "fu": 42.0}[kind] * (nt // n) * (ns // n) * n * (n - 1.0)
    assert (work < 0.5 * every) if expanded else (work == every)
    ctx.close()


def test_pair_terms_are_held_in_parts():
    """1024 drops of degree 4 with their expansions in 8 GB (13.5 where every pair's terms lie side by side)."""
    import paper_1811_10270_gb300 as S
    n, p = 1024, 4
    x = lattice(n, p)
    before = torch.cuda.mem_get_info()[0]
    ctx = S.Context(precision=S.DF64)
    ctx.set_drops([p] * n, x)
    assert before - torch.cuda.mem_get_info()[0] < 8 * 2 ** 30
    ctx.close()


def test_parts_add_up():
    """Sums whose pair terms take several parts, against direct sums: 2^-42 of the sum of magnitudes, which is below
    the sum of the 1/r^2 of a lattice of unit drops, times strengths of which the largest is taken."""
    import paper_1811_10270_gb300 as S
    n, p = 700, 5
    ctx = S.Context(precision=S.DF64)
    ctx.set_near(False)
    ctx.set_drops([p] * n, lattice(n, p))
    nc, nt, ns = ctx.sizes()
    rng = np.random.default_rng(8)
    d = torch.tensor(np.concatenate([inputs.random_density(p, rng)[0] for _ in range(n)]), device="cuda")
    a, b = (torch.empty(nt, device="cuda", dtype=torch.float64) for _ in range(2))
    for which in (S.LAPLACE_DL, S.LAPLACE_SL):
        ctx.set_expansions(True)
        ctx.eval_electric(which, d, a, S.OUT_GRID)
        ctx.set_expansions(False)
        ctx.eval_electric(which, d, b, S.OUT_GRID)
        # |density| < 5; 700 unit spheres at distances from 2.6: sum 4 pi / r / (4 pi) < 700 / 2.6
        assert (a - b).abs().max().item() < 2.0 ** -42 * 5.0 * n / 2.6
    ctx.close()


def test_without_memory_for_the_expansions_every_pair_is_direct():
    """With 2.5 GB left the expansions of 512 drops (3.9 GB where all terms lie side by side) leave the near grids and
    the row build their room, and give back what they took."""
    import paper_1811_10270_gb300 as S
    n, p = 512, 4
    x = lattice(n, p)
    nc = n * (p + 1) ** 2
    d = torch.ones(nc, device="cuda", dtype=torch.float64)
    ctx = S.Context(precision=S.DF64)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - int(2.5 * 2 ** 30), device="cuda", dtype=torch.uint8)
    try:
        ctx.set_drops([p] * n, x)
        out = torch.empty(ctx.sizes()[1], device="cuda", dtype=torch.float64)
        ctx.eval_electric(S.LAPLACE_DL, d, out, S.OUT_GRID)
        assert torch.isfinite(out).all()
    finally:
        del hog
        torch.cuda.empty_cache()
        ctx.close()
