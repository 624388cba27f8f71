"""The Stokes preconditioner's basis from the device: shapes at the edges of its two ways."""
import os

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
    if not os.path.exists(pkg.LIB_PATH):
        from paper_1811_10270_gb300 import build
        build.build()
    pkg.lib()
    return pkg


def solve(S, degrees, shapes, lam, precondition):
    dev = torch.device("cuda")
    rng = np.random.default_rng(5)
    x = torch.tensor(np.concatenate([s.ravel() for s in shapes]), device=dev)
    rhs = torch.tensor(np.concatenate([inputs.random_density(p, rng, 3).ravel() for p in degrees]), device=dev)
    ctx = S.Context(precision=S.FP64, gmres_tol=1e-12)
    ctx.set_stokes_preconditioner(precondition)
    ctx.set_drops(degrees, x, lam)
    u = torch.zeros_like(rhs)
    ctx.gmres_solve(S.SYS_STOKES, rhs, u)
    ctx.close()
    return u.cpu().numpy()


@pytest.mark.parametrize("degrees,shift", [([1], 0.0), ([5, 16], 0.0), ([9, 4], 300.0)])
def test_preconditioned_solution_is_the_plain_one(S, degrees, shift):
    """GMRES to 1e-12 with and without the preconditioner: the solutions differ by the residuals times the
    condition of the system (below 1e4 for these viscosity ratios and shapes), 1e-8 relative."""
    rng = np.random.default_rng(2)
    shapes, lam = [], []
    for i, p in enumerate(degrees):
        shapes.append(inputs.perturbed_coef(p, rng, 1.0, (shift + 3.0 * i, 0.0, 0.0), amp=0.03 if p > 1 else 0.0))
        lam.append(20.0 / (i + 1))
    a, b = solve(S, degrees, shapes, lam, True), solve(S, degrees, shapes, lam, False)
    assert np.linalg.norm(a - b) < 1e-8 * np.linalg.norm(b)


def needle(aspect):
    """A sphere squeezed toward the line through (1, 1, 1): at small aspects the rotations are nearly dependent."""
    x = inputs.sphere_coef(6, 1.0, (0.0, 0.0, 0.0))
    d = np.ones((3, 1)) / np.sqrt(3.0)
    along = d * (d * x).sum(0)
    return along + aspect * (x - along)


@pytest.mark.parametrize("aspect", [0.3, 3e-4])
def test_needles_are_accepted(S, aspect):
    ctx = S.Context(precision=S.FP64)
    ctx.set_drops([6], torch.tensor(needle(aspect).ravel(), device="cuda"))
    ctx.close()


@pytest.mark.parametrize("bad", ["zero", "nan", "line"])
def test_shapes_without_a_basis_are_refused(S, bad):
    x = needle(0.0)
    if bad == "zero":
        x[:] = 0.0
    elif bad == "nan":
        x[1, 7] = float("nan")
    ctx = S.Context(precision=S.FP64)
    with pytest.raises(S.ShbimError):
        ctx.set_drops([6], torch.tensor(x.ravel(), device="cuda"))
    ctx.close()
