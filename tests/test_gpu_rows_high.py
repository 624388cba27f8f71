"""Singular rows at the degrees where the row build changes form: the folded Fourier stage, seven-digit Legendre stage and
split rotations above degree 39 (40, 41, 47: edges of their K steps; 63: their last degree; 64: two degree tiles of the
Legendre stage, the last degree's rotation on the FP32 pipe), with every stage and with none on the tensor cores, against
the native FP64 build of the same rows, on a drop off the origin. Bound: the one of the other degrees, 1e-11."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def values(S, torch, p, x, dens, f, rows, mask):
    dev = torch.device("cuda")
    ctx = S.Context(precision=S.FP64)
    ctx.set_rows_precision(rows)
    ctx.set_tensor_cores(mask)
    ctx.set_drops([p], torch.tensor(x.ravel(), device=dev), [2.5])
    nt = (p + 1) * (2 * p + 2)
    out = []
    for which in (S.LAPLACE_DL, S.LAPLACE_SL):
        o = torch.empty(nt, device=dev, dtype=torch.float64)
        ctx.eval_electric(which, torch.tensor(dens, device=dev), o, S.OUT_GRID)
        out.append(o.cpu().numpy())
    for a in ((f, None), (None, f)):
        o = torch.empty(3 * nt, device=dev, dtype=torch.float64)
        ctx.eval_stokes(*(None if v is None else torch.tensor(v.ravel(), device=dev) for v in a), o, S.OUT_GRID)
        out.append(o.cpu().numpy())
    ctx.close()
    return out


@pytest.mark.parametrize("p", [39, 40, 41, 47, 63, 64])
def test_rows_match_fp64_build(p):
    import torch
    import paper_1811_10270_gb300 as S
    rng = np.random.default_rng(p)
    x = inputs.perturbed_coef(p, rng, 1.0, (4.0, -3.0, 5.0))
    dens, f = inputs.random_density(p, rng)[0], inputs.random_density(p, rng, 3)
    ref = values(S, torch, p, x, dens, f, S.FP64, 0)
    for mask in (S.TC_ALL, 0, S.TC_FOURIER):
        for a, b in zip(values(S, torch, p, x, dens, f, S.DF64, mask), ref):
            assert np.abs(a - b).max() < 1e-11 * np.abs(b).max(), mask
