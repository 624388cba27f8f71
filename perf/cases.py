"""Timed cases of the library: what a simulation of surfactant-covered drops asks of it, call by call.

A time step of the method rebuilds the operators of the current drop shapes (set_drops), applies the Laplace
and Stokes layer operators inside GMRES and once each for its right-hand sides, and now and then
reparametrises the surfaces; around it stand the transforms and the warm-start network. The cases take each of
these through the package's public calls: single drops (where launches count), two close drops of degree
32, and batches of up to 64 drops of degrees 16 to 48 in a box, in the three arithmetic modes (the default
native FP64, double-float, and single precision with compensated sums, the operator of the inner
GMRES iterations). Shapes, surfactant, densities and box are of the recipe of the repository's inputs:
perturbed spheres of radius 0.8 to 1.2, gaps of at least about 0.2, densities N(0,1)/(n+1).

`exact` restates the discretised operators in plain torch, in 64 bits: harmonics evaluated at points, the
regular rule, the rotated-pole rule by direct evaluation at rotated nodes, the upsampled rule at near targets.
"""
import math

import numpy as np
import torch

import paper_1811_10270_gb300 as lib

PRECISION = {"fp64": lib.FP64, "fp32": lib.FP32_COMP, "df64": lib.DF64}
MIXED = "16,24,32,48"


def listed():
    return [
        # the smallest full step: one drop of degree 16, native FP64 (launches and latency)
        {"name": "step_one_p16", "call": "step", "drops": 1, "degrees": "16", "precision": "fp64"},
        # two drops 0.1 apart at degree 32: the step of a pair interaction run, mixed precision
        {"name": "step_two_p32", "call": "step", "drops": 2, "degrees": "32", "precision": "fp32"},
        # a small suspension of uneven degrees: one whole step, mixed precision
        {"name": "step_12_mixed", "call": "step", "drops": 12, "degrees": MIXED, "precision": "fp32"},
        # the electric GMRES operator of a 64-drop suspension, single precision with compensated sums
        {"name": "electric_dl_fp32_64", "call": "electric", "which": "dl", "drops": 64, "degrees": MIXED, "precision": "fp32"},
        # the Stokes GMRES operator of the same suspension
        {"name": "stokes_d_fp32_64", "call": "stokes", "which": "u", "drops": 64, "degrees": MIXED, "precision": "fp32"},
        # the Stokes right-hand side of the same suspension: a one-shot sum in double-float
        {"name": "stokes_s_df64_64", "call": "stokes", "which": "f", "drops": 64, "degrees": MIXED, "precision": "df64"},
        # many small drops of an odd degree: charge potential in double-float
        {"name": "electric_sl_df64_40p11", "call": "electric", "which": "sl", "drops": 40, "degrees": "11", "precision": "df64"},
        # a solve with the default context (native FP64) on a handful of drops
        {"name": "solve_fp64_6p16", "call": "solve", "which": "electric", "drops": 6, "degrees": "16", "precision": "fp64"},
        # mixed-precision Stokes solve of two close drops, refined to 1e-10 (training data of the network)
        {"name": "refine_stokes_two_p32", "call": "refine", "which": "stokes", "drops": 2, "degrees": "32", "precision": "fp32"},
        # new shapes, their operators and one application of each: degrees up to the largest, 64
        {"name": "geometry_16_to_64", "call": "geometry", "drops": 4, "degrees": "16,31,48,64", "precision": "df64"},
        # synthesis of vector fields on the upsampled grids and their projection back
        {"name": "sht_16_mixed", "call": "sht", "drops": 16, "degrees": MIXED, "precision": "fp64"},
        # gradients of the warm-start network for two drops of degree 8, batch 64
        {"name": "network_gradients_p8", "call": "network", "drops": 2, "degrees": "8", "precision": "fp32", "batch": 64},
    ]


def draw(rng):
    while True:
        call = rng.choice(["step", "electric", "electric", "electric", "stokes", "stokes", "stokes", "geometry", "solve", "refine", "sht", "reparametrize", "network"])
        lo, hi = {"step": (1, 12), "solve": (1, 8), "refine": (1, 8), "geometry": (1, 12), "network": (1, 2), "reparametrize": (1, 16)}.get(call, (1, 64))
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        top = {"network": 12, "solve": 32}.get(call, 48)
        kinds = rng.randint(1, 4)
        degrees = ",".join(str(int(round(math.exp(rng.uniform(math.log(6), math.log(top)))))) for _ in range(min(kinds, n)))
        case = {"call": call, "drops": n, "degrees": degrees, "precision": rng.choice(["fp64", "fp32", "df64"])}
        if call in ("refine", "network"):
            case["precision"] = "fp32"
        if call in ("solve", "refine"):
            case["which"] = rng.choice(["electric", "stokes"])
        if call == "electric":
            case["which"] = rng.choice(["dl", "sl"])
        if call == "stokes":
            case["which"] = rng.choice(["f", "u", "fu"])
        if call == "network":
            case["batch"] = rng.randint(1, 96)
        # no more than the largest listed case, in target-source pairs weighted by their arithmetic and in
        # entries of the singular-rule weights
        S = _sizes(case)
        applications = {"solve": 12, "refine": 24, "step": 60}.get(call, 1) if call != "sht" else 0
        weight = {"fp64": 60.0, "df64": 8.0, "fp32": 1.0}[case["precision"]] * (2.0 if call != "electric" else 1.0)
        rows = S["row_nodes"] * {"step": 2}.get(call, 1)
        if applications * weight * S["pairs"] < 8e11 and rows < 1.5e9:
            return case


# ---------------------------------------------------------------- inputs


def _degrees(case):
    d = [int(x) for x in case["degrees"].split(",")]
    return [d[i % len(d)] for i in range(case["drops"])]


def _nodes(q):
    return (q + 1) * (2 * q + 2)


def _sizes(case):
    ps = _degrees(case)
    nt, ns = [_nodes(p) for p in ps], [_nodes(2 * p + 1) for p in ps]
    return {"coef": sum((p + 1) ** 2 for p in ps), "targets": sum(nt), "sources": sum(ns),
            "pairs": float(sum(nt)) * sum(ns) - sum(a * float(b) for a, b in zip(nt, ns)),
            "row_nodes": sum(a * float(b) for a, b in zip(nt, ns)),
            "self_work": sum(a * float(b) * (p + 1) ** 2 for p, a, b in zip(ps, nt, ns)),
            "rows": sum(a * 14.0 * (p + 1) ** 2 for p, a in zip(ps, nt))}


def _place(rng, radii):
    """Centres in a box of the suspension's density (64 drops in a 12 x 12 x 12 box), nominal gaps >= 0.4."""
    n = len(radii)
    box = 12.0 * max(n / 64.0, 0.05) ** (1.0 / 3.0)
    while True:
        at = np.zeros((0, 3))
        for i in range(n):
            for _ in range(4000):
                c = rng.uniform(-box / 2 + radii[i], box / 2 - radii[i], size=3) if box > 2 * radii[i] else rng.uniform(-0.1, 0.1, size=3)
                if i == 0 or np.all(np.linalg.norm(at - c, axis=1) >= radii[:i] + radii[i] + 0.4):
                    at = np.vstack([at, c])
                    break
            else:
                break
        if len(at) == n:
            return at
        box *= 1.1


def _shape(rng, p, radius, centre):
    """A sphere plus N(0,1) 0.05 / n^2 radius on every position coefficient of degree 1 to 8."""
    c = np.zeros((3, (p + 1) ** 2))
    k = math.sqrt(4.0 * math.pi / 3.0) * radius
    c[0, 3], c[1, 1], c[2, 2] = -k, -k, k
    c[:, 0] = math.sqrt(4.0 * math.pi) * np.asarray(centre)
    for n in range(1, min(8, p) + 1):
        c[:, n * n:(n + 1) ** 2] += rng.standard_normal((3, 2 * n + 1)) * 0.05 / (n * n) * radius
    return c


def _surfactant(rng, p):
    g = np.zeros((p + 1) ** 2)
    g[0] = math.sqrt(4.0 * math.pi)
    top = (min(4, p) + 1) ** 2
    g[1:top] = rng.uniform(-0.2, 0.2, size=top - 1) / 24.0
    return g


def _density(rng, p, ncomp):
    n = np.floor(np.sqrt(np.arange((p + 1) ** 2)))
    return rng.standard_normal((ncomp, (p + 1) ** 2)) / (n + 1.0)


def _inputs(case, seed):
    """Numpy inputs of a case, from the seed alone."""
    rng = np.random.default_rng([seed, case["drops"]])
    ps = _degrees(case)
    n = len(ps)
    radii = rng.uniform(0.8, 1.2, size=n) if n > 2 else np.ones(n)
    lam = rng.uniform(0.5, 10.0, size=n) if n > 2 else np.full(n, 5.0 if n == 2 else 1.0)
    if n > 2:
        x = [_shape(rng, p, r, c) for p, r, c in zip(ps, radii, _place(rng, radii))]
    else:
        x = [_shape(rng, p, 1.0, (0.0, 0.0, 0.0)) for p in ps]
        if n == 2:  # one above the other, 0.1 between their extremes along the axis
            z = [_on_grid(torch.tensor(c[2:]), p, p, False)[0][0] for c, p in zip(x, ps)]
            gap = 0.1 + float(z[0].max()) - float(z[1].min())
            x[0][2, 0] -= 0.5 * gap * math.sqrt(4.0 * math.pi)
            x[1][2, 0] += 0.5 * gap * math.sqrt(4.0 * math.pi)
    return {"p": ps, "lam": lam.tolist(), "x": x, "gamma": [_surfactant(rng, p) for p in ps],
            "scalar": [_density(rng, p, 1)[0] for p in ps], "f": [_density(rng, p, 3) for p in ps],
            "u": [_density(rng, p, 3) for p in ps], "rng": rng}


def _device(parts):
    return torch.tensor(np.concatenate([np.asarray(a).ravel() for a in parts]), device="cuda")


def _like(t, n):
    return torch.empty(n, device="cuda", dtype=torch.float64)


def prepare(case, seed):
    I = _inputs(case, seed)
    call = case["call"]
    if call == "network":
        return _prepare_network(case, I)
    s = {"case": case, "p": I["p"], "lam": I["lam"], "x": _device(I["x"])}
    tol = 1e-10 if call == "refine" else 1e-8
    ctx = s["ctx"] = lib.Context(precision=PRECISION[case["precision"]], R=2.0, gmres_tol=tol)
    # the layout and the operators of these shapes; a geometry or step case builds them again in its pass
    ctx.set_drops(s["p"], s["x"], s["lam"])
    nc, nt, ns = s["sizes"] = ctx.sizes()
    if call == "step":
        s["phys"] = lib.phys(R=2.0, Q=0.5, Ca_E=0.1, beta=0.2, x_s=0.5, E_u=(0.0, 0.0, 1.0))
        s["gamma"], s["x_out"], s["gamma_out"] = _device(I["gamma"]), _like(s, 3 * nc), _like(s, nc)
    elif call == "electric":
        s["density"], s["out"] = _device(I["scalar"]), _like(s, nc)
    elif call == "stokes":
        s["f"] = _device(I["f"]) if "f" in case["which"] else None
        s["u"] = _device(I["u"]) if "u" in case["which"] else None
        s["out"] = _like(s, 3 * nc)
    elif call in ("solve", "refine"):
        stokes = case["which"] == "stokes"
        s["rhs"] = _device(I["f"] if stokes else I["scalar"])
        s["out"] = torch.empty_like(s["rhs"])
    elif call == "geometry":
        s["density"], s["f"], s["u"] = _device(I["scalar"]), _device(I["f"]), _device(I["u"])
        s["at"], s["electric"], s["stokes"] = _like(s, 7 * nt), _like(s, nc), _like(s, 3 * nc)
    elif call == "sht":
        s["fields"] = [d for d in range(len(s["p"])) for _ in range(3)]
        s["coef"], s["grid"], s["back"] = _device(I["u"]), _like(s, 3 * ns), _like(s, 3 * nc)
    elif call == "reparametrize":
        s["gamma"] = _device(I["gamma"])
        s["x_out"], s["gamma_out"] = torch.empty_like(s["x"]), torch.empty_like(s["gamma"])
    return s


def _prepare_network(case, I):
    """The warm-start network of the case's drops: features to the guesses of both solves, width 512."""
    nc = sum((p + 1) ** 2 for p in I["p"])
    widths = [4 * nc + 7 + len(I["p"]), 512, 512, 512, 4 * nc]
    rng, net = I["rng"], lib.MLP(widths, max_batch=case["batch"])
    layers = []
    for l, (a, b) in enumerate(zip(widths[:-1], widths[1:])):
        layers.append((rng.uniform(-1, 1, size=(b, a)).astype(np.float32) / math.sqrt(a), np.zeros(b, np.float32)))
        net.set_layer(l, *layers[-1])
    x, t = (rng.standard_normal((case["batch"], w)).astype(np.float32) for w in (widths[0], widths[-1]))
    return {"case": case, "net": net, "layers": layers, "x": torch.tensor(x, device="cuda"), "t": torch.tensor(t, device="cuda"),
            "y": torch.empty(case["batch"], widths[-1], device="cuda")}


def run(s):
    case = s["case"]
    call = case["call"]
    if call == "network":
        net = s["net"]
        loss = net.train_step(s["x"], s["t"], 1e-3, update=False)
        net.forward(s["x"], s["y"])
        return {"loss": loss, "y": s["y"], "gradients": [net.get_layer(l)[2:] for l in range(len(net.widths) - 1)]}
    ctx = s["ctx"]
    if call == "step":
        err, _ = ctx.step(s["phys"], s["x"], s["gamma"], 1e-2, s["x_out"], s["gamma_out"])
        return {"x": s["x_out"], "gamma": s["gamma_out"], "error": err}
    if call == "electric":
        ctx.eval_electric(lib.LAPLACE_SL if case["which"] == "sl" else lib.LAPLACE_DL, s["density"], s["out"])
        return _as_summed(case, s["out"])
    if call == "stokes":
        ctx.eval_stokes(s["f"], s["u"], s["out"])
        return _as_summed(case, s["out"])
    if call == "solve":
        ctx.gmres_solve(lib.SYS_STOKES if case["which"] == "stokes" else lib.SYS_ELECTRIC, s["rhs"], s["out"])
        return _as_summed(case, s["out"])
    if call == "refine":
        ctx.gmres_solve_refined(lib.SYS_STOKES if case["which"] == "stokes" else lib.SYS_ELECTRIC, s["rhs"], s["out"])
        return s["out"]
    if call == "geometry":
        ctx.set_drops(s["p"], s["x"], s["lam"])
        ctx.target_geometry(s["at"])
        ctx.eval_electric(lib.LAPLACE_DL, s["density"], s["electric"])
        ctx.eval_stokes(s["f"], s["u"], s["stokes"])
        return {"targets": s["at"], "electric": _as_summed(case, s["electric"]), "stokes": _as_summed(case, s["stokes"])}
    if call == "sht":
        ctx.sht(lib.SHT_INVERSE, lib.GRID_UP, s["fields"], s["coef"], s["grid"])
        ctx.sht(lib.SHT_FORWARD, lib.GRID_UP, s["fields"], s["grid"], s["back"])
        return {"grid": s["grid"], "back": s["back"]}
    s["x_out"].copy_(s["x"])
    s["gamma_out"].copy_(s["gamma"])
    energies = ctx.reparametrize(s["x_out"], s["gamma_out"], steps=20)
    return {"x": s["x_out"], "gamma": s["gamma_out"], "energies": np.array(energies)}


def _as_summed(case, out):
    """The values of a single-precision sum carry single precision, and are handed on as such."""
    return out.float() if case["precision"] == "fp32" else out


def work(case):
    """What a pass cannot do without: coefficients in and out, every geometry node (position, normal, weight) once
    where sums over other drops are formed, and the singular rows where an operator is applied or built; flops of
    the singular rows' products and of the transforms by latitude (Legendre sums, then Fourier sums), per
    density. The sums between drops are left out of the flops: they are the part whose cost depends on the
    method that forms them."""
    call, S = case["call"], _sizes(case)
    if call == "network":
        w = [4 * S["coef"] + 7 + case["drops"], 512, 512, 512, 4 * S["coef"]]
        mk = sum(a * b for a, b in zip(w[:-1], w[1:]))
        return {"bytes": 2 * mk + 4 * mk + 4 * case["batch"] * (w[0] + 2 * w[-1]), "flops": 8.0 * mk * case["batch"]}
    per_drop = [(p, 2 * p + 1) for p in _degrees(case)]
    sht_up = sum(2.0 * (q + 1) * ((p + 1) ** 2 + (p + 1) * (2 * q + 2)) for p, q in per_drop)
    sht_base = sum(2.0 * (p + 1) * ((p + 1) ** 2 + (p + 1) * (2 * p + 2)) for p, _ in per_drop)
    if call == "sht":
        return {"bytes": 8.0 * 3 * (2 * S["coef"] + 2 * S["sources"]), "flops": 3 * 2 * sht_up}
    if call == "reparametrize":
        return {"bytes": 8.0 * 8 * S["coef"], "flops": 20 * 12 * sht_up}
    grid = 8.0 * 7 * (S["targets"] + (S["sources"] if case["drops"] > 1 else 0))
    def applied(scalar):
        comps = 1 if scalar else 3
        return {"bytes": 8.0 * (2 * comps * S["coef"] + S["rows"] / 14 * (1 if scalar else 6)) + grid,
                "flops": 2 * S["rows"] / 14 * (1 if scalar else 9) + comps * (sht_up + sht_base)}
    built = {"bytes": 8.0 * (3 * S["coef"] + S["rows"]), "flops": 14 * S["targets"] / max(1, case["drops"]) * sht_up}
    e, t = applied(True), applied(False)
    if call == "electric":
        return e
    if call == "stokes":
        return t
    if call in ("solve", "refine"):
        return e if case["which"] == "electric" else t
    parts = [built, e, t] if call == "geometry" else [built, built] + 4 * [e] + 4 * [t]
    return {k: sum(x[k] for x in parts) for k in ("bytes", "flops")}


# ---------------------------------------------------------------- the same in 64 bits, plain torch


def _legendre_blocks(top, ct, st):
    """For m = 0, 1, .. top: the normalised Legendre functions of order m, degrees m .. top, stacked."""
    sect = torch.full_like(ct, 1.0 / math.sqrt(4.0 * math.pi))
    for m in range(top + 1):
        if m:
            sect = -math.sqrt((2.0 * m + 1.0) / (2.0 * m)) * st * sect
        block = [sect]
        if m < top:
            block.append(math.sqrt(2.0 * m + 3.0) * ct * sect)
        for n in range(m + 2, top + 1):
            a = math.sqrt((4.0 * n * n - 1.0) / (n * n - m * m))
            b = math.sqrt(((n - 1.0) ** 2 - m * m) / (4.0 * (n - 1.0) ** 2 - 1.0))
            block.append(a * (ct * block[-1] - b * block[-2]))
        yield torch.stack(block)


def _at_points(coef, p, ct, st, ph, derivs=True):
    """Fields [K, (p+1)^2] at points: values, d/dtheta and (1/sin) d/dphi, each [K, points] (the last two None
    without derivs). Division-free forms of the derivatives hold at the poles too."""
    dev = ct.device
    coef = coef.to(dev)
    out = [torch.zeros(coef.shape[0], ct.numel(), dtype=torch.float64, device=dev) for _ in range(3 if derivs else 1)]
    gen = _legendre_blocks(p + 1 if derivs else p, ct, st)
    lower, here = None, next(gen)
    for m in range(p + 1):
        upper = next(gen, None)
        n = torch.arange(m, p + 1, dtype=torch.float64, device=dev)
        i = (n * n + n).long()
        cc, cs = coef[:, i + m], coef[:, i - m]
        if m == 0:
            out[0] += cc @ here[: p + 1]
            if derivs:
                out[1][:] += (cc[:, 1:] * torch.sqrt(n * (n + 1))[1:]) @ upper[:p]
        else:
            r2, c, s = math.sqrt(2.0), torch.cos(m * ph), torch.sin(m * ph)
            out[0] += r2 * ((cc @ here[: p + 1 - m]) * c + (cs @ here[: p + 1 - m]) * s)
            if derivs:
                up, down = 0.5 * torch.sqrt((n - m) * (n + m + 1)), 0.5 * torch.sqrt((n + m) * (n - m + 1))
                k = -0.5 * torch.sqrt((2 * n + 1) / (2 * n + 3))
                mu, md = k * torch.sqrt((n + m + 1) * (n + m + 2)), k * torch.sqrt((n - m + 1) * (n - m + 2))

                def both(q):
                    dth = (q * up)[:, 1:] @ upper[: p - m] - (q * down) @ lower[1: p + 2 - m]
                    msin = (q * mu) @ upper[: p + 1 - m] + (q * md) @ lower[2: p + 3 - m]
                    return dth, msin
                (dc, mc), (ds, ms) = both(cc), both(cs)
                out[1] += r2 * (dc * c + ds * s)
                out[2] += r2 * (ms * c - mc * s)
        lower, here = here, upper
    return out if derivs else [out[0], None, None]


def _grid(q, dev):
    t, w = np.polynomial.legendre.leggauss(q + 1)
    t, w = torch.tensor(t[::-1].copy(), device=dev), torch.tensor(w[::-1].copy(), device=dev)
    ph = math.pi * torch.arange(2 * q + 2, dtype=torch.float64, device=dev) / (q + 1)
    return t, (math.pi / (q + 1)) * w, ph


def _on_grid(coef, p, q, derivs=True):
    t, _, ph = _grid(q, coef.device)
    k = ph.numel()
    ct = t.repeat_interleave(k)
    return _at_points(coef, p, ct, torch.sqrt(1 - ct * ct), ph.repeat(q + 1), derivs)


def _weights(q, dev):
    return _grid(q, dev)[1].repeat_interleave(2 * q + 2)


def _project(values, p, q):
    """Inner products of grid values [K, nodes] with the harmonics up to degree p."""
    t, w, ph = _grid(q, values.device)
    v = values.reshape(values.shape[0], q + 1, 2 * q + 2) * w[None, :, None]
    out = torch.zeros(values.shape[0], (p + 1) ** 2, dtype=torch.float64, device=values.device)
    for m, block in enumerate(_legendre_blocks(p, t, torch.sqrt(1 - t * t))):
        n = torch.arange(m, p + 1, device=values.device)
        scale = 1.0 if m == 0 else math.sqrt(2.0)
        out[:, n * n + n + m] = scale * (v @ torch.cos(m * ph)) @ block.T
        if m:
            out[:, n * n + n - m] = scale * (v @ torch.sin(m * ph)) @ block.T
    return out


def _normals(xt, xp):
    c = torch.linalg.cross(xt, xp, dim=0)
    J = torch.sqrt((c * c).sum(0))
    return c / J, J


class _Drop:
    def __init__(self, p, x, lam):
        self.p, self.q, self.lam = p, 2 * p + 1, lam
        self.coef = torch.tensor(x, device="cuda")
        self.x0, a, b = _on_grid(self.coef, p, p)
        self.n0, self.J0 = _normals(a, b)
        self.sources = self.nodes(self.q)
        self.spacing = math.sqrt(float(self.sources[2].sum()) / self.sources[0].shape[1])

    def nodes(self, q):
        """Positions, normals and weights of the drop's degree-q grid."""
        x, a, b = _on_grid(self.coef, self.p, q)
        n, J = _normals(a, b)
        return x, n, _weights(q, "cuda") * J

    def strengths(self, coef, q):
        return _on_grid(coef, self.p, q, False)[0]


def _term(kind, d, n0, n, dens):
    """Kernel times density at displacements d [3, T, S]: [1 or 3, T, S]."""
    r2 = (d * d).sum(0)
    ri = torch.rsqrt(r2)
    if kind == "sl":
        return (ri * dens[0])[None]
    if kind == "dl":
        return ((d * n0[:, :, None]).sum(0) * ri * ri * ri * dens[0])[None]
    dd = (d * dens).sum(0)
    if kind == "f":
        return ri * dens + d * (dd * ri ** 3)
    return d * (-6.0 * dd * (d * n).sum(0) * ri ** 5)


def _sum_over(kind, x0, n0, x, n, w, dens):
    step = max(1, int(2e7) // x.shape[1])
    out = [_term(kind, x0[:, a:a + step, None] - x[:, None], n0[:, a:a + step], n[:, None], dens[:, None]) @ w
           for a in range(0, x0.shape[1], step)]
    return torch.cat(out, 1) / (4.0 * math.pi)


def _self_values(d, kinds, dens):
    """The rotated-pole rule at every target of drop d; dens {kind: coefficients}. {kind: values}."""
    t, w, ph = _grid(d.q, "cuda")
    p0, p1, tot = torch.ones_like(t), t.clone(), torch.ones_like(t) + t
    for n in range(1, d.q):
        p0, p1 = p1, ((2 * n + 1) * t * p1 - n * p0) / (n + 1)
        tot = tot + p1
    mu = (w * torch.sqrt(2 * (1 - t)) * tot).repeat_interleave(ph.numel()) / (4.0 * math.pi)
    ct, p2 = t.repeat_interleave(ph.numel()), ph.repeat(t.numel())
    st = torch.sqrt(1 - ct * ct)
    node = torch.stack([st * torch.cos(p2), st * torch.sin(p2), ct])
    tb, _, pb = _grid(d.p, "cuda")
    th, fi = torch.arccos(tb).repeat_interleave(pb.numel()), pb.repeat(tb.numel())
    step = max(1, int(1.5e6) // node.shape[1])
    out = {k: [] for k in kinds}
    for a in range(0, th.numel(), step):
        c, s, cf, sf = (f[:, None] for f in (torch.cos(th[a:a + step]), torch.sin(th[a:a + step]), torch.cos(fi[a:a + step]), torch.sin(fi[a:a + step])))
        m = c.shape[0]
        u, z = c * node[0] + s * node[2], -s * node[0] + c * node[2]
        X, Y = cf * u - sf * node[1], sf * u + cf * node[1]
        rct, rst, rph = z.reshape(-1), torch.sqrt(X * X + Y * Y).reshape(-1), torch.atan2(Y, X).reshape(-1)
        x, xa, xb = _at_points(d.coef, d.p, rct, rst, rph)
        n, J = _normals(xa, xb)
        shape = (3, m, -1)
        dx = d.x0[:, a:a + step, None] - x.reshape(shape)
        weight = J.reshape(m, -1) * mu
        for k in kinds:
            v = _at_points(dens[k], d.p, rct, rst, rph, False)[0].reshape(dens[k].shape[0], m, -1)
            out[k].append((_term(k, dx, d.n0[:, a:a + step], n.reshape(shape), v) * weight).sum(-1))
    return {k: torch.cat(v, 1) for k, v in out.items()}


def _near(di, dj):
    """Targets of drop i closer than six source spacings to a node of drop j."""
    x, lim = dj.sources[0], 6.0 * dj.spacing
    step = max(1, int(2e7) // x.shape[1])
    d2 = torch.cat([((di.x0[:, a:a + step, None] - x[:, None]) ** 2).sum(0).min(1).values for a in range(0, di.x0.shape[1], step)])
    return torch.nonzero(torch.sqrt(d2) < lim)[:, 0]


def _layer(drops, dens):
    """Galerkin coefficients of the sum over kinds in dens {kind: [coefficients per drop]} ('u' with its contrast)."""
    parts = []
    scaled = {k: [(c * (d.lam - 1.0) if k == "u" else c) for c, d in zip(v, drops)] for k, v in dens.items()}
    on_grid = {k: [d.strengths(c, d.q) for c, d in zip(v, drops)] for k, v in scaled.items()}
    for i, d in enumerate(drops):
        own = _self_values(d, list(dens), {k: scaled[k][i] for k in dens})
        total = sum(own.values())
        for j, e in enumerate(drops):
            if i == j:
                continue
            near = _near(d, e)
            for k in dens:
                total = total + _sum_over(k, d.x0, d.n0, *e.sources, on_grid[k][j])
                if near.numel():
                    qf = 4 * (e.q + 1) - 1
                    x0, n0 = d.x0[:, near], d.n0[:, near]
                    total[:, near] += _sum_over(k, x0, n0, *e.nodes(qf), e.strengths(scaled[k][j], qf)) - _sum_over(k, x0, n0, *e.sources, on_grid[k][j])
        parts.append(_project(total, d.p, d.p).reshape(-1))
    return torch.cat(parts)


def _bf16(a):
    return torch.tensor(a).bfloat16().double() if isinstance(a, np.ndarray) else a.float().bfloat16().double()


def exact(case, seed):
    call, S = case["call"], _sizes(case)
    I = _inputs(case, seed)
    if call == "network":
        s = _prepare_network(case, I)
        W, h = [_bf16(w).cuda() for w, _ in s["layers"]], [_bf16(s["x"])]
        for l, w in enumerate(W):
            z = h[-1] @ w.T
            h.append(_bf16(torch.tanh(z)) if l + 1 < len(W) else z)
        d = (h[-1] - s["t"].double()) / case["batch"]
        loss, g = 0.5 * float((d * d).sum()) * case["batch"], []
        for l in range(len(W) - 1, -1, -1):
            d = d * (1 - h[l + 1] ** 2) if l + 1 < len(W) else d
            g.append((d.T @ h[l], d.sum(0)))
            d = d @ W[l]
        return {"loss": loss, "y": h[-1], "gradients": g[::-1]}
    dev = [torch.tensor(a, device="cuda") for a in I["u"]]
    if call == "sht":
        grid = [_on_grid(c, p, 2 * p + 1, False)[0] for c, p in zip(dev, I["p"])]
        return {"grid": torch.cat([g.reshape(-1) for g in grid]), "back": torch.cat([_project(g, p, 2 * p + 1).reshape(-1) for g, p in zip(grid, I["p"])])}
    if call == "reparametrize":
        return _exact_flow(I)
    if call not in ("electric", "stokes", "geometry") or S["self_work"] > 6e10 or S["pairs"] > 4e9:
        return None
    drops = [_Drop(p, x, lam) for p, x, lam in zip(I["p"], I["x"], I["lam"])]
    scalar = [torch.tensor(a[None], device="cuda") for a in I["scalar"]]
    f = [torch.tensor(a, device="cuda") for a in I["f"]]
    if call == "electric":
        return _layer(drops, {case["which"]: scalar})
    if call == "stokes":
        return _layer(drops, {k: {"f": f, "u": dev}[k] for k in case["which"]})
    at = torch.cat([torch.cat([getattr(d, a)[c] for d in drops]) for a in ("x0", "n0") for c in range(3)] + [d.J0 for d in drops])
    return {"targets": at, "electric": _layer(drops, {"dl": scalar}), "stokes": _layer(drops, {"f": f, "u": dev})}


def _exact_flow(I):
    """Twenty tangential steps of the reparametrisation, energy exponent 4, step 0.5 / p^4."""
    X, G, E = [], [], np.zeros(21)
    for p, x, g in zip(I["p"], I["x"], I["gamma"]):
        q, tau = 2 * p + 1, 0.5 / float(p) ** 4
        both = torch.tensor(np.vstack([x, g[None]]), device="cuda")
        n4 = torch.floor(torch.sqrt(torch.arange((p + 1) ** 2, dtype=torch.float64, device="cuda") + 1e-9)) ** 4
        E[0] += float((n4 * both[:3] ** 2).sum())
        for k in range(20):
            v, a, b = _on_grid(both, p, q)
            n, _ = _normals(a[:3], b[:3])
            h = _on_grid(n4 * both[:3], p, q, False)[0]
            t = h - (h * n).sum(0) * n
            aa, ab, bb = ((u * w).sum(0) for u, w in ((a[:3], a[:3]), (a[:3], b[:3]), (b[:3], b[:3])))
            at, bt = (a[:3] * t).sum(0), (b[:3] * t).sum(0)
            dg = (a[3] * (bb * at - ab * bt) + b[3] * (aa * bt - ab * at)) / (aa * bb - ab * ab)
            both = _project(torch.cat([v[:3] - tau * t, (v[3] - tau * dg)[None]]), p, q)
            E[k + 1] += float((n4 * both[:3] ** 2).sum())
        X.append(both[:3].reshape(-1))
        G.append(both[3])
    return {"x": torch.cat(X), "gamma": torch.cat(G), "energies": E}
