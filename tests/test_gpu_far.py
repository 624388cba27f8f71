"""Sums between well-separated drops through multipole and local expansions, against the oracle.

A suspension of drops of uneven, odd and even degrees in which most pairs are far, one pair is close and one drop is
far from every other: operator values at sampled targets of every drop equal the oracle's regular rule plus
its singular rows. Bounds: the library's stated ones, 1e-10 (FP64 and FP64-class) and 1e-5 (FP32) of the largest
value; the expansions truncate at 3e-15 and 1e-8 of a pair's sum of magnitudes. The direct work the
library reports (kernel_work) shows that the expansions were taken; FP32 sums take them from about ten times as many
pairs on, so that mode runs the same suspension at 1.7 times the degrees.
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu

DEGREES = [16, 5, 21, 9, 12, 14, 18, 7, 20, 11, 17, 15]
FINER = [int(1.7 * p) for p in DEGREES]
FLOPS = {"dl": 19.0, "sl": 11.0, "f": 29.0, "u": 30.0, "fu": 42.0}


def suspension(degrees):
    rng = np.random.default_rng(11)
    drops, centres = [], []
    for i, p in enumerate(degrees):
        a = float(rng.uniform(0.7, 1.1))
        if i == 1:
            c = centres[0] + np.array([0.0, 0.0, 2.3 * 1.0])      # close to drop 0
        elif i == 2:
            c = np.array([40.0, -35.0, 20.0])                     # far from every drop
        else:
            c = 3.6 * np.array([(i % 3) - 1.0, (i // 3 % 2) - 0.5, (i // 6) - 0.5]) + rng.uniform(-0.3, 0.3, 3)
            while centres and min(np.linalg.norm(c - o) for o in centres) < 2.6:
                c = c + np.array([0.9, 1.3, -1.1])
        centres.append(c)
        drops.append((p, inputs.perturbed_coef(p, rng, a, c, amp=0.03), float(rng.uniform(0.5, 8.0))))
    dens = {"scalar": [inputs.random_density(p, rng)[0] for p in degrees], "f": [inputs.random_density(p, rng, 3) for p in degrees],
            "u": [inputs.random_density(p, rng, 3) for p in degrees]}
    return drops, dens


@pytest.fixture(scope="module")
def cases():
    made = {}

    def get(precision):
        degrees = tuple(FINER if precision == "FP32_COMP" else DEGREES)
        if degrees not in made:
            made[degrees] = build(degrees)
        return made[degrees]
    return get


def build(degrees):
    from oracle import operators
    drops, dens = suspension(degrees)
    sysm = operators.System([operators.DropGeom(x, p, lam) for p, x, lam in drops], near=False)
    rng = np.random.default_rng(3)
    sample = [np.sort(rng.choice(d.nt, size=3, replace=False)) for d in sysm.drops]
    ref = {}
    for kind, k in (("dl", "ladl"), ("sl", "lsl")):
        ref[kind] = [sysm.laplace_targets(k, dens["scalar"], i, t) for i, t in enumerate(sample)]
    for kind in ("f", "u", "fu"):
        f = dens["f"] if "f" in kind else None
        u = dens["u"] if "u" in kind else None
        ref[kind] = [sysm.stokes_targets(f, u, i, t) for i, t in enumerate(sample)]
    return drops, dens, sysm, sample, ref


@pytest.mark.parametrize("precision,bound", [("FP64", 1e-10), ("DF64", 1e-10), ("FP32_COMP", 1e-5)])
@pytest.mark.parametrize("kind", ["dl", "sl", "f", "u", "fu"])
def test_far_expansions_match_oracle(cases, kind, precision, bound):
    import torch
    import paper_1811_10270_gb300 as S
    drops, dens, sysm, sample, ref = cases(precision)
    dev = torch.device("cuda")
    up = lambda parts: torch.tensor(np.concatenate([np.ravel(a) for a in parts]), device=dev)
    ctx = S.Context(precision=getattr(S, precision))
    ctx.set_near(False)
    ctx.set_drops([p for p, _, _ in drops], up([x for _, x, _ in drops]), [lam for _, _, lam in drops])
    nt = [d.nt for d in sysm.drops]
    ncomp = 1 if kind in ("dl", "sl") else 3
    out = torch.empty(ncomp * sum(nt), device=dev, dtype=torch.float64)

    def apply():
        if ncomp == 1:
            ctx.eval_electric(S.LAPLACE_SL if kind == "sl" else S.LAPLACE_DL, up(dens["scalar"]), out, S.OUT_GRID)
        else:
            ctx.eval_stokes(up(dens["f"]) if "f" in kind else None, up(dens["u"]) if "u" in kind else None, out, S.OUT_GRID)

    apply()
    ctx.set_timing(True)
    apply()
    cls = S.K_PAIRS if precision == "FP32_COMP" else S.K_PAIRS_FP64CLASS
    work = ctx.kernel_work(cls)
    ctx.set_timing(False)
    got = out.cpu().numpy()
    ns = [d.xs.shape[1] for d in sysm.drops]
    every = FLOPS[kind] * sum(t * (sum(ns) - s) for t, s in zip(nt, ns))
    assert work < 0.5 * every, "every pair summed directly"
    scale = max(np.abs(r).max() for r in ref[kind])
    o = 0
    for i, n in enumerate(nt):
        v = got[o:o + ncomp * n].reshape(ncomp, n)[:, sample[i]]
        o += ncomp * n
        err = np.abs(v - np.reshape(ref[kind][i], (ncomp, -1))).max() / scale
        assert err < bound, (i, drops[i][0], err)
    ctx.close()
