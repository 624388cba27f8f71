"""Singular rows at the degrees whose row build has its own tensor-core form: folded Fourier stage, seven-digit Legendre
stage and split rotations from degree 40 on (40, 41, 47: edges of their K steps; 63: their last degree block; 64: two degree
tiles of the Legendre stage, the last degree's rotation on the FP32 pipe). Seven digits hold more than a double-float's
sums keep, so against the native FP64 rows the build with every stage on the tensor cores is as close as the
double-float build of the same rows (no stage on them): the root mean square error of the operator values at most 1.5 times
as large, and never above 1e-10 of the largest value. The drop is centred: off the origin the FP64 rows are those of
a drop displaced by the rounding of their rotation of the centre."""
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


@pytest.mark.parametrize("p", [40, 41, 47, 63, 64])
def test_tensor_core_rows_as_close_as_double_float(p):
    import torch
    import paper_1811_10270_gb300 as S
    rng = np.random.default_rng(p)
    x = inputs.perturbed_coef(p, rng, 1.0, (0.0, 0.0, 0.0))
    dens, f = inputs.random_density(p, rng)[0], inputs.random_density(p, rng, 3)
    ref = values(S, torch, p, x, dens, f, S.FP64, 0)
    plain = values(S, torch, p, x, dens, f, S.DF64, 0)
    rms = lambda a: float(np.sqrt(np.mean(a * a)))
    for mask in (S.TC_ALL, S.TC_FOURIER | S.TC_LEGENDRE, S.TC_ROTATION):
        for a, b, r in zip(values(S, torch, p, x, dens, f, S.DF64, mask), plain, ref):
            assert rms(a - r) <= 1.5 * rms(b - r), (mask, rms(a - r), rms(b - r))
            assert np.abs(a - r).max() < 1e-10 * np.abs(r).max(), mask
