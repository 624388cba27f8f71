"""Expansions between drops against direct sums of the library, at every target and for every kind of sum.

Errors are taken against the direct sums in native FP64 and relative to the sum of magnitudes at each target,
sum |strength| / r^k / (4 pi) over the other drops' nodes (k = 1 for single layers, 2 for double layers). Bounds:

* FP64: 1e-14. The truncation is 3e-15 of strengths over gaps; sums of 1e4 to 1e5 roundings of 2^-53, random
  from term to term, stay below the rest.
* FP64-class: 2^-42, the rounding of one direct term (2^-44, and 2^-42 on quantised positions).
* FP32: 2^-22, the rounding of one direct term (four roundings of 2^-24).

Orders ten too low would show at 3e-15 and 1e-8 times 0.6^-10 = 165 and more.
"""
import numpy as np
import pytest

import inputs
import test_gpu_far as far
import test_gpu_far_close as close

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BOUND = {"FP64": 1e-14, "DF64": 2.0 ** -42, "FP32_COMP": 2.0 ** -22}
KINDS = ["dl", "sl", "f", "u", "fu"]


def densities(degrees, rng):
    return {"scalar": [inputs.random_density(p, rng)[0] for p in degrees], "f": [inputs.random_density(p, rng, 3) for p in degrees],
            "u": [inputs.random_density(p, rng, 3) for p in degrees]}


def elongated():
    """Ellipsoids of aspect 3 and drops of radius 0.3 to 1.8 side by side."""
    rng = np.random.default_rng(41)
    drops = []
    for i in range(14):
        p = [21, 15, 18, 24][i % 4]
        r = [1.8, 0.3, 1.0, 0.5][i % 4]
        x = inputs.perturbed_coef(p, rng, r, (0.0, 0.0, 0.0), amp=0.02)
        x[2] *= 3.0 if i % 3 == 0 else 1.0
        x[:, 0] = np.sqrt(4.0 * np.pi) * np.array([6.0 * (i % 3), 5.5 * (i // 3 % 3), 12.0 * (i // 9)])
        drops.append((p, x, float(rng.uniform(0.5, 8.0))))
    return drops, densities([p for p, _, _ in drops], rng)


def many(n):
    """n small drops (lists of the planner at and past multiples of a warp)."""
    rng = np.random.default_rng(n)
    drops = []
    for i in range(n):
        c = 2.7 * np.array([i % 4, i // 4 % 4, i // 16]) + rng.uniform(-0.1, 0.1, 3)
        drops.append((6 + i % 3, inputs.perturbed_coef(6 + i % 3, rng, float(rng.uniform(0.8, 1.1)), c, amp=0.03), float(rng.uniform(0.5, 8.0))))
    return drops, densities([p for p, _, _ in drops], rng)


SETS = {"suspension": lambda: far.suspension(far.FINER), "close": lambda: close.lattice(far.FINER), "elongated": elongated,
        "33 drops": lambda: many(33), "64 drops": lambda: many(64)}


def magnitudes(drops, dens):
    """Per kind the sum of magnitudes at every target."""
    from oracle import operators, sh
    geo = [operators.DropGeom(x, p, lam) for p, x, lam in drops]
    up = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    src = [up(d.xs) for d in geo]
    tgt = [up(d.x0) for d in geo]
    val = {}
    for name in ("scalar", "f", "u"):
        val[name] = []
        for d, c in zip(geo, dens[name]):
            v = np.sqrt((sh.sht_inverse(np.atleast_2d(c), d.p, d.q) ** 2).sum(0)) * d.ws
            val[name].append(up(v * (6.0 * abs(d.lam - 1.0) if name == "u" else 1.0)))
    out = {k: [] for k in KINDS}
    for i, t in enumerate(tgt):
        one, two, f, u = (torch.zeros(t.shape[1], device="cuda", dtype=torch.float64) for _ in range(4))
        for j, s in enumerate(src):
            if j == i:
                continue
            ri = torch.cdist(t.T.contiguous(), s.T.contiguous(), compute_mode="donot_use_mm_for_euclid_dist").reciprocal_()
            one += ri @ val["scalar"][j]
            f += ri @ val["f"][j]
            ri *= ri
            two += ri @ val["scalar"][j]
            u += ri @ val["u"][j]
        for k, v in zip(KINDS, (two, one, f, u, f + u)):
            out[k].append(v.cpu().numpy() / (4.0 * np.pi))
    return out


@pytest.fixture(scope="module")
def made():
    kept = {}

    def get(name):
        if name not in kept:
            drops, dens = SETS[name]()
            kept[name] = (drops, dens, magnitudes(drops, dens))
        return kept[name]
    return get


def device(parts):
    return torch.tensor(np.concatenate([np.ravel(a) for a in parts]), device="cuda")


def apply(S, ctx, kind, dens, nt):
    ncomp = 1 if kind in ("dl", "sl") else 3
    out = torch.empty(ncomp * sum(nt), device="cuda", dtype=torch.float64)
    if ncomp == 1:
        ctx.eval_electric(S.LAPLACE_SL if kind == "sl" else S.LAPLACE_DL, device(dens["scalar"]), out, S.OUT_GRID)
    else:
        ctx.eval_stokes(device(dens["f"]) if "f" in kind else None, device(dens["u"]) if "u" in kind else None, out, S.OUT_GRID)
    return out.cpu().numpy()


def others(S, ctx, kind, dens, nt):
    """Per drop the values at its targets of all other drops' densities: its own is zero, so that the self rows, whose
    values are many times as large for a drop far from the others, add nothing that has to be rounded."""
    ncomp, o, out = (1 if kind in ("dl", "sl") else 3), 0, []
    for i, n in enumerate(nt):
        rest = {k: [np.zeros_like(a) if j == i else a for j, a in enumerate(v)] for k, v in dens.items()}
        out.append(apply(S, ctx, kind, rest, nt)[o:o + ncomp * n].reshape(ncomp, n))
        o += ncomp * n
    return out


def made_of_expansions(S, ctx, kind, dens, nt, degrees):
    """Whether the direct work of an application is less than that of every pair."""
    ctx.set_timing(True)
    apply(S, ctx, kind, dens, nt)
    work = sum(ctx.kernel_work(c) for c in (S.K_PAIRS, S.K_PAIRS_FP64CLASS))
    ctx.set_timing(False)
    ns = [(2 * p + 2) * (4 * p + 4) for p in degrees]
    return work < 0.95 * far.FLOPS[kind] * sum(t * (sum(ns) - s) for t, s in zip(nt, ns))


@pytest.mark.parametrize("name", list(SETS))
def test_expansions_are_as_close_as_direct_sums(made, name):
    import paper_1811_10270_gb300 as S
    drops, dens, mags = made(name)
    degrees, shapes, lam = [p for p, _, _ in drops], device([x for _, x, _ in drops]), [l for _, _, l in drops]
    nt = [(p + 1) * (2 * p + 2) for p in degrees]
    ref, taken = {}, {p: set() for p in BOUND}
    for precision in ("FP64", "DF64", "FP32_COMP"):
        ctx = S.Context(precision=getattr(S, precision))
        ctx.set_near(False)
        ctx.set_drops(degrees, shapes, lam)
        for kind in KINDS:
            got = others(S, ctx, kind, dens, nt)
            if precision == "FP64":
                ctx.set_expansions(False)
                assert not made_of_expansions(S, ctx, kind, dens, nt, degrees)
                ref[kind] = others(S, ctx, kind, dens, nt)
                ctx.set_expansions(True)
            if made_of_expansions(S, ctx, kind, dens, nt, degrees):
                taken[precision].add(kind)
            worst = max((np.abs(g - r).max(0) / m).max() for g, r, m in zip(got, ref[kind], mags[kind]))
            print(name, precision, kind, "%.2e" % worst, kind in taken[precision])
            assert worst < BOUND[precision], (precision, kind, worst)
        ctx.close()
    # few small drops: in FP64 alone the expansions pay
    assert taken["FP64"] and (taken["DF64"] or "drops" in name), taken


def test_expansions_follow_the_shapes_through_captured_graphs(made):
    """Solves before and after the drops have moved (other lists, other orders), operators captured in graphs: the
    same as in a fresh context. The near correction adds in no fixed order and is off; the Givens rotations stay on the
    host (a context's first solve starts there, its later ones on the device, with another hypotenuse)."""
    import paper_1811_10270_gb300 as S
    drops, dens, _ = made("suspension")
    degrees, lam = [p for p, _, _ in drops], [l for _, _, l in drops]
    moved = [x.copy() for _, x, _ in drops]
    for i, x in enumerate(moved):
        x[:, 0] *= 1.0 + 0.1 * (i % 3)
    rhs = device(dens["u"])

    def solve(ctx, shapes):
        ctx.set_drops(degrees, device(shapes), lam)
        out = torch.zeros_like(rhs)
        ctx.gmres_solve(S.SYS_STOKES, rhs, out)
        return out.cpu().numpy()

    def context():
        ctx = S.Context(precision=S.DF64, gmres_tol=1e-10)
        ctx.set_near(False)
        ctx.set_device_gmres(False)
        return ctx
    used, fresh = context(), context()
    first = solve(used, [x for _, x, _ in drops])
    second = solve(used, moved)
    assert np.abs(first - second).max() > 1e-6 * np.abs(first).max()
    np.testing.assert_array_equal(second, solve(fresh, moved))
    np.testing.assert_array_equal(first, solve(used, [x for _, x, _ in drops]))
    used.close()
    fresh.close()


def in_long_double(kind, drops, dens, i, targets):
    """Sums over the other drops at targets of drop i, in long double on the oracle's sources."""
    from oracle import operators, sh
    LD = np.longdouble
    geo = [operators.DropGeom(x, p, lam) for p, x, lam in drops]
    out = []
    for t in targets:
        x0, n0, v = geo[i].x0[:, t].astype(LD), geo[i].n0[:, t].astype(LD), np.zeros(1 if kind == "dl" else 3, LD)
        for j, d in enumerate(geo):
            if j == i:
                continue
            r = [x0[c] - d.xs[c].astype(LD) for c in range(3)]
            ri = 1 / np.sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2])
            if kind == "dl":
                q = (sh.sht_inverse(dens["scalar"][j], d.p, d.q) * d.ws).astype(LD)
                v[0] += (q * ri ** 3 * sum(r[c] * n0[c] for c in range(3))).sum()
            else:
                q = sh.sht_inverse(dens["u"][j], d.p, d.q).astype(LD) * d.ws.astype(LD)
                w = ri ** 5 * sum(r[c] * q[c] for c in range(3)) * sum(r[c] * d.ns[c].astype(LD) for c in range(3))
                v += np.array([(w * r[c]).sum() for c in range(3)]) * (-6 * (LD(d.lam) - 1))
        out.append(v * LD("0.0795774715459476678844418816862571810"))
    return np.stack(out, 1)


@pytest.mark.parametrize("kind", ["dl", "u"])
def test_fp64_sums_at_a_distant_drop_are_rounded_not_truncated(made, kind):
    """At a drop 57 radii away every source lies in one direction and the truncation's bound is nearly reached. Allowed:
    1e-15 of the sum of magnitudes, five roundings (the oracle's positions there are rounded to 1e-16 of the distance)."""
    import paper_1811_10270_gb300 as S
    drops, dens, mags = made("suspension")
    degrees = [p for p, _, _ in drops]
    nt = [(p + 1) * (2 * p + 2) for p in degrees]
    ctx = S.Context(precision=S.FP64)
    ctx.set_near(False)
    ctx.set_drops(degrees, device([x for _, x, _ in drops]), [l for _, _, l in drops])
    assert made_of_expansions(S, ctx, kind, dens, nt, degrees)
    got = others(S, ctx, kind, dens, nt)[2]
    ctx.close()
    targets = np.arange(7, nt[2], nt[2] // 24)
    ref = in_long_double(kind, drops, dens, 2, targets)
    err = np.abs(got[:, targets] - ref).max(0).astype(float) / mags[kind][2][targets]
    print(kind, "%.2e" % err.max())
    assert err.max() < 1e-15
