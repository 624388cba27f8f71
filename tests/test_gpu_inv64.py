"""Powers of 1/r in FP64: single pairs over the range of distances, the inner one and what lies outside it."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1811_10270_gb300 as pkg
    if not os.path.exists(pkg.LIB_PATH):
        from paper_1811_10270_gb300 import build
        build.build()
    pkg.lib()
    return pkg


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("lo,hi", [(-1, 1), (-49, 49), (-70, -45), (45, 70)])
def test_single_pairs_over_distances(S, which, lo, hi):
    """One source, targets on a line through it at |r| from 2^lo to 2^hi, the normal along the line: exactly
    1 / (4 pi r) and 1 / (4 pi r^2). r^2 has a relative error of 2.5 and its power (k/2 of that) one of 4 more
    roundings at most: 8 units of 2^-53 for k = 1, 12 for k = 3."""
    rng = np.random.default_rng(100 + hi)
    r = np.exp2(rng.uniform(lo, hi, 4096)) * rng.uniform(0.5, 1.0, 4096)
    u = np.array([2.0, -3.0, 6.0]) / 7.0
    x = r[None] * u[:, None]
    tgt = torch.tensor(np.concatenate([x, np.repeat(u[:, None], r.size, 1)]), device="cuda").contiguous()
    src = torch.tensor([[0.0], [0.0], [0.0], [1.0]], device="cuda", dtype=torch.float64)
    out = torch.empty(r.size, device="cuda", dtype=torch.float64)
    assert S.pairs_laplace_noalloc(which, tgt, src, out) == 0
    xl, ul = x.astype(np.longdouble), u.astype(np.longdouble)
    d2 = (xl * xl).sum(0)
    ref = (1 / np.sqrt(d2) if which == 1 else (xl * ul[:, None]).sum(0) / (d2 * np.sqrt(d2))) * np.longdouble("0.0795774715459476678844418816862571810")
    err = np.abs(out.cpu().numpy() / ref - 1).astype(float)
    assert err.max() < (8 if which == 1 else 12) * 2.0**-53


def test_coincident_and_infinite_points(S):
    """A target on the source and one infinitely far away: as the quotients have it in floating point."""
    tgt = torch.zeros(6, 2, device="cuda", dtype=torch.float64)
    tgt[0, 1] = float("inf")
    tgt[3] = 1.0
    src = torch.tensor([[0.0], [0.0], [0.0], [1.0]], device="cuda", dtype=torch.float64)
    out = torch.empty(2, device="cuda", dtype=torch.float64)
    assert S.pairs_laplace_noalloc(1, tgt, src, out) == 0
    assert out[0].item() == float("inf") and out[1].item() == 0.0
    assert S.pairs_laplace_noalloc(0, tgt, src, out) == 0
    assert torch.isnan(out).all()
