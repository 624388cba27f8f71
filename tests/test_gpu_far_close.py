"""Close drops whose far-side targets take the neighbour's multipole expansion, against the oracle.

Twelve drops on a lattice of spacing 2.45 (gaps of 0.1 to 0.6): neighbours are too close for local expansions, so
the direct work stays below theirs only if groups of targets take the multipole expansions. The degrees are those at
which every kind of sum takes expansions. Bounds as for the other expansions: the library's 1e-10 (FP64 and FP64-class
sums) and 1e-5 (FP32) of the largest value.
"""
import numpy as np
import pytest

import inputs
import test_gpu_far as far

pytestmark = pytest.mark.gpu


def lattice(degrees):
    rng = np.random.default_rng(23)
    drops = []
    for i, p in enumerate(degrees):
        c = 2.45 * np.array([i % 3, i // 3 % 2, i // 6]) + rng.uniform(-0.05, 0.05, 3)
        drops.append((p, inputs.perturbed_coef(p, rng, float(rng.uniform(0.9, 1.05)), c, amp=0.03), float(rng.uniform(0.5, 8.0))))
    dens = {"scalar": [inputs.random_density(p, rng)[0] for p in degrees], "f": [inputs.random_density(p, rng, 3) for p in degrees],
            "u": [inputs.random_density(p, rng, 3) for p in degrees]}
    return drops, dens


@pytest.fixture(scope="module")
def cases():
    plain, far.suspension = far.suspension, lattice
    try:
        yield far.build(far.FINER)
    finally:
        far.suspension = plain


@pytest.mark.parametrize("precision,bound", [("FP64", 1e-10), ("DF64", 1e-10), ("FP32_COMP", 1e-5)])
@pytest.mark.parametrize("kind", ["dl", "sl", "f", "u", "fu"])
def test_close_drops_match_oracle(cases, kind, precision, bound):
    import torch
    import paper_1811_10270_gb300 as S
    drops, dens, sysm, sample, ref = cases
    dev = torch.device("cuda")
    up = lambda parts: torch.tensor(np.concatenate([np.ravel(a) for a in parts]), device=dev)
    ctx = S.Context(precision=getattr(S, precision))
    ctx.set_near(False)
    ctx.set_drops([p for p, _, _ in drops], up([x for _, x, _ in drops]), [lam for _, _, lam in drops])
    nt, ns = [d.nt for d in sysm.drops], [d.xs.shape[1] for d in sysm.drops]
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
    work = ctx.kernel_work(S.K_PAIRS if precision == "FP32_COMP" else S.K_PAIRS_FP64CLASS)
    ctx.set_timing(False)
    at = [np.array([x[c, 0] for c in range(3)]) / np.sqrt(4 * np.pi) for _, x, _ in drops]
    close = far.FLOPS[kind] * sum(nt[i] * ns[j] for i in range(len(nt)) for j in range(len(nt))
                                  if i != j and np.linalg.norm(at[i] - at[j]) < 2.6)
    assert work < 0.9 * close, (work, close)
    got = out.cpu().numpy()
    scale = max(np.abs(r).max() for r in ref[kind])
    o = 0
    for i, n in enumerate(nt):
        v = got[o:o + ncomp * n].reshape(ncomp, n)[:, sample[i]]
        o += ncomp * n
        err = np.abs(v - np.reshape(ref[kind][i], (ncomp, -1))).max() / scale
        assert err < bound, (i, drops[i][0], err)
    ctx.close()
