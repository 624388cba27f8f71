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
