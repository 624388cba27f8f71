"""Shapes that are not finite are refused by set_drops, whichever coefficient it is, and the refusal leaves no way into the
sums between drops.

The degree-0 coefficients give a drop's centre; the modes of the Stokes preconditioner, in which the other
coefficients show, do not hold them.
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1811_10270_gb300 as pkg
    pkg.lib()
    return pkg


def drops(degrees):
    return [inputs.sphere_coef(p, 1.0, (0.0, 0.0, 3.0 * i)) for i, p in enumerate(degrees)]


def device(shapes):
    return torch.tensor(np.concatenate([x.ravel() for x in shapes]), device="cuda")


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("degrees,where", [([4], (0, 0)), ([4], (0, 2)), ([4, 3], (1, 1)), ([4, 3], (0, 0))])
def test_a_centre_that_is_not_finite_is_refused(S, degrees, where, value):
    shapes = drops(degrees)
    shapes[where[0]][where[1], 0] = value
    ctx = S.Context(precision=S.FP64)
    with pytest.raises(S.ShbimError):
        ctx.set_drops(degrees, device(shapes))
    # the context takes the sound shapes afterwards
    ctx.set_drops(degrees, device(drops(degrees)))
    ctx.close()


def operators(S, ctx, n):
    """One call of every kind of sum between drops on densities of n coefficients."""
    d, u = torch.ones(n, device="cuda", dtype=torch.float64), torch.ones(3 * n, device="cuda", dtype=torch.float64)
    out, out3 = torch.empty_like(d), torch.empty_like(u)
    return [lambda: ctx.eval_electric(S.LAPLACE_DL, d, out), lambda: ctx.eval_electric(S.LAPLACE_SL, d, out),
            lambda: ctx.eval_stokes(u, None, out3), lambda: ctx.eval_stokes(None, u, out3), lambda: ctx.eval_stokes(u, u, out3)]


@pytest.mark.parametrize("precision", ["FP64", "FP32_COMP", "DF64"])
def test_a_failed_layout_leaves_no_drops(S, precision):
    """Lists and near pairs of the layout before are not used on the buffers of the one that failed."""
    ctx = S.Context(precision=getattr(S, precision))
    close = [inputs.sphere_coef(6, 1.0, (0.0, 0.0, 2.2 * i)) for i in range(5)]
    ctx.set_drops([6] * 5, device(close))
    assert ctx.near_pairs() > 0
    bad = drops([4, 3])
    bad[1][:] = 0.0                     # no surface: refused after the layout has been made
    with pytest.raises(S.ShbimError):
        ctx.set_drops([4, 3], device(bad))
    assert ctx.near_pairs() == 0 and ctx.sizes() == (0, 0, 0)
    for call in operators(S, ctx, 25 + 16):
        with pytest.raises(S.ShbimError, match="no drops set"):
            call()
    ctx.set_drops([4, 3], device(drops([4, 3])))
    for call in operators(S, ctx, 25 + 16):
        call()
    ctx.close()


def test_refused_shapes_of_the_same_layout_are_not_summed(S):
    ctx = S.Context(precision=S.FP64)
    ctx.set_drops([4, 3], device(drops([4, 3])))
    bad = drops([4, 3])
    bad[1][:] = 0.0
    with pytest.raises(S.ShbimError):
        ctx.set_drops([4, 3], device(bad))
    for call in operators(S, ctx, 25 + 16):
        with pytest.raises(S.ShbimError, match="set_drops failed"):
            call()
    ctx.set_drops([4, 3], device(drops([4, 3])))
    for call in operators(S, ctx, 25 + 16):
        call()
    ctx.close()


def test_more_drops_than_the_lists_hold_are_refused(S):
    """Before anything is allocated: the drop set of before stays."""
    ctx = S.Context(precision=S.FP64)
    ctx.set_drops([4, 3], device(drops([4, 3])))
    n = 65536
    with pytest.raises(S.ShbimError, match="65535"):
        ctx.set_drops([1] * n, torch.zeros(n * 3 * 4, device="cuda", dtype=torch.float64))
    for call in operators(S, ctx, 25 + 16):
        call()
    ctx.close()
