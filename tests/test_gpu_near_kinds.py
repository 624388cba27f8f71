"""Near-field sums of one Stokes term alone (their own kernels) against the kernel of both terms: S[f] + (lam - 1) D[u]
in one application equals the two applications' sum, at every target, with the correction on and groups of near targets below
and above one, two and three warps. Bounds: the library's stated ones, 1e-10 (FP64, FP64-class) and 1e-5 (FP32) of the
largest value."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,bound", [("FP64", 1e-10), ("DF64", 1e-10), ("FP32_COMP", 1e-5)])
@pytest.mark.parametrize("p,gap", [((6, 5), 0.9), ((9, 12), 0.35), ((14, 11), 0.2), ((20, 17), 0.15)])
def test_single_terms_add_up(p, gap, precision, bound):
    import torch
    import paper_1811_10270_gb300 as S
    rng = np.random.default_rng(sum(p))
    dev = torch.device("cuda")
    up = lambda parts: torch.tensor(np.concatenate([a.ravel() for a in parts]), device=dev)
    x = [inputs.perturbed_coef(q, rng, 1.0, (0.0, 0.0, s * (1.0 + 0.5 * gap)), amp=0.01) for q, s in zip(p, (-1, 1))]
    f, u = ([inputs.random_density(q, rng, 3) for q in p] for _ in range(2))
    ctx = S.Context(precision=getattr(S, precision))
    ctx.set_drops(p, up(x), [3.0, 0.6])
    assert ctx.near_pairs() > 0
    n = 3 * sum((q + 1) * (2 * q + 2) for q in p)
    out = []
    for a, b in ((f, u), (f, None), (None, u)):
        o = torch.empty(n, device=dev, dtype=torch.float64)
        ctx.eval_stokes(None if a is None else up(a), None if b is None else up(b), o, S.OUT_GRID)
        out.append(o.cpu().numpy())
    ctx.close()
    assert np.abs(out[0] - out[1] - out[2]).max() < bound * np.abs(out[0]).max()
