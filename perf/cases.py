"""Performance cases of the drop solver: the calls a simulation of surfactant-laden drops makes, through
the package's public entry points, over the sizes of the seeded workloads of inputs.py and the bench.

Kinds of a case
  apply       one layer-operator apply (the matvec of the solve) on a geometry that is kept
  rhs         the right-hand side 2 u_inf + S[f] on a geometry that is kept
  solve       right-hand side and GMRES solve of the boundary integral equation
  setup       a new shape: geometry, interfacial force, right-hand side (each stage of a time step)
  surfactant  explicit and diffusive surfactant rates and the implicit diffusion stage
  velocity    the velocity at fluid points among the drops
  step        one coupled drop/surfactant time step (Alg. 1)

Values of a mixed-precision apply carry single precision (its pair sums and self term run in FP32), so
they are returned as float32; everything else is returned as the calls give it, in float64.

exact() restates the method (arXiv 1707.02156) in plain torch in 64 bits: spherical-harmonic bases
evaluated at points, the singular rule with the target at the pole (Thm 1), the regular and upsampled
rules, the interpolation next to a surface (Sec. 2.3), the Galerkin projection, and the surface calculus
of the force and the surfactant.
"""
import math

import numpy as np
import torch

from paper_1707_02156_gb300 import api

PRECISION = {"fp64": api.BIE_FP64, "mixed": api.BIE_MIXED, "df": api.BIE_DF}
ELASTICITY, SHEAR, INV_PE, DT = 0.2, 1.0, 0.1, 0.01


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def _case(name, kind, shape, n, degrees, **more):
    c = {"name": name, "kind": kind, "shape": shape, "n": n, "degrees": degrees, "double_quadrature": False, "up": 2,
         "precision": "mixed", "layer": "double", "gap": 0.0, "points": 0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one FP64 single-layer apply on a sphere of degree 16
        _case("sphere_apply_fp64", "apply", "sphere", 1, "16", precision="fp64", layer="single"),
        # the matvec of a single-drop solve: degree 32 with the quadrature grid twice as fine
        _case("drop_matvec_mixed", "apply", "drop", 1, "32", double_quadrature=True),
        # the velocity of a single drop in shear: double-float right-hand side, mixed solve to 1e-10
        _case("drop_solve", "solve", "drop", 1, "32", double_quadrature=True),
        # two drops nearly touching: the near-singular rule in every matvec of the solve
        _case("pair_solve", "solve", "pair", 2, "32", up=4, gap=0.05),
        # a batch of drops of uneven degree: the matvec over several degree groups
        _case("uneven_matvec_mixed", "apply", "spheres", 20, "16,24,32,48"),
        # the matvec of a many-drop run: the FP32 pair sums
        _case("many_matvec_mixed", "apply", "deformed", 192, "24"),
        # the right-hand side of a many-drop solve: the double-float pair sums
        _case("many_rhs_df", "rhs", "deformed", 80, "24", precision="df", layer="single"),
        # the matvec in plain FP64 on a small batch
        _case("batch_matvec_fp64", "apply", "spheres", 16, "16,24", precision="fp64"),
        # every stage of every time step sets up a new shape
        _case("new_shapes", "setup", "deformed", 64, "24", precision="df", layer="single"),
        # the surfactant's share of a time step
        _case("surfactant_stage", "surfactant", "deformed", 48, "16,24,32"),
        # the flow field among the drops, some points right at the surfaces
        _case("flow_field", "velocity", "deformed", 64, "24", points=16411),
        # a whole time step of a small run
        _case("small_step", "step", "deformed", 8, "16"),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "rhs", "solve", "setup", "surfactant", "velocity", "step"])
    if kind == "apply" and rng.random() < 0.5 or kind == "solve" and rng.random() < 0.5:  # one drop
        p = rng.randint(8, 36)
        fine = p <= 28 and rng.random() < 0.5
        return _case("", kind, rng.choice(["sphere", "drop"]) if kind == "apply" else "drop", 1, str(p),
                     double_quadrature=fine, precision=rng.choice(["fp64", "mixed", "df"]) if kind == "apply" else "mixed",
                     layer=rng.choice(["single", "double"]))
    if kind == "solve":
        return _case("", kind, "pair", 2, str(rng.randint(12, 30)), up=rng.choice([2, 3, 4]), gap=rng.uniform(0.04, 0.15))
    if kind == "step":
        return _case("", kind, "deformed", _log(rng, 2, 8), str(rng.randint(8, 15)))
    if kind == "apply" and rng.random() < 0.4:
        ps = sorted(rng.sample(range(8, 41), rng.randint(2, 5)))
        return _case("", kind, "spheres", _log(rng, 3, 20), ",".join(map(str, ps)), up=rng.choice([1, 2, 3]),
                     precision=rng.choice(["mixed", "mixed", "df"]), layer=rng.choice(["single", "double"]))
    if kind == "apply":
        return _case("", kind, "deformed", _log(rng, 3, 150), str(rng.randint(10, 24)), precision="mixed",
                     layer=rng.choice(["single", "double"]))
    if kind == "rhs":
        return _case("", kind, "deformed", _log(rng, 2, 64), str(rng.randint(10, 24)), precision="df", layer="single")
    if kind == "setup":
        ps = sorted(rng.sample(range(8, 25), rng.randint(1, 3)))
        return _case("", kind, "deformed", _log(rng, 2, 56), ",".join(map(str, ps)), precision="df", layer="single")
    if kind == "surfactant":
        ps = sorted(rng.sample(range(8, 33), rng.randint(1, 3)))
        return _case("", kind, "deformed", _log(rng, 2, 44), ",".join(map(str, ps)))
    return _case("", "velocity", "deformed", _log(rng, 2, 60), str(rng.randint(12, 24)), points=_log(rng, 200, 15000))


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _nc(p):
    return (p + 1) * (p + 1)


def _degrees(p):
    return np.floor(np.sqrt(np.arange(_nc(p)) + 0.5)).astype(np.int64)


def _band(rng, p, ncomp):
    """Random band-limited fields, coefficients ~ N(0, 1)/(n+1)^2."""
    return rng.standard_normal((ncomp, _nc(p))) / (_degrees(p) + 1.0) ** 2


def _unit_sphere(p):
    u = np.zeros((3, _nc(p)))
    s = math.sqrt(2.0 * math.pi / 3.0)
    u[0, 3], u[1, 1], u[2, 2] = -s, s, math.sqrt(4.0 * math.pi / 3.0)
    return u


def _noise(rng, p, lo, hi, amplitude):
    """Perturbation of degrees lo..hi whose components are bounded by amplitude."""
    n = _degrees(p)
    m = np.arange(_nc(p)) - n * (n + 1)
    d = rng.standard_normal((3, _nc(p))) * ((n >= lo) & (n <= hi))
    fac = np.where(m == 0, 1.0, 2.0) * np.sqrt((2 * n + 1) / (4.0 * math.pi))
    a = np.abs(d) * fac  # |(Re, Im)| <= |Re| + |Im|
    return d * (amplitude / max(1e-300, a.sum(axis=1).max()))


def _rotation(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    return q * np.sign(np.linalg.det(q))


def _place(rng, radii, gap):
    """Random sequential addition in a cube at the bench's volume fraction, the largest first."""
    n = len(radii)
    box = 2.6 + 25.6 * (n / 512.0) ** (1.0 / 3.0)
    order = np.argsort(-radii)
    at = np.zeros((n, 3))
    while True:
        done = 0
        for i in order:
            for _ in range(400):
                c = rng.uniform(radii[i], box - radii[i], size=(16, 3))
                if done:
                    d = np.linalg.norm(c[:, None] - at[order[:done]][None], axis=2)
                    c = c[np.all(d >= radii[order[:done]] + radii[i] + gap, axis=1)]
                if len(c):
                    at[i] = c[0]
                    done += 1
                    break
            else:
                break
        if done == n:
            return at
        box *= 1.04


def _inputs(case, seed):
    """Host arrays: degrees, quadrature degrees, shapes, densities, surfactant, viscosity ratios."""
    rng = np.random.default_rng([seed, 1707])
    choice = [int(v) for v in str(case["degrees"]).split(",")]
    n, shape = case["n"], case["shape"]
    ps = [choice[0]] * n if len(choice) == 1 else [int(v) for v in rng.permutation([choice[i % len(choice)] for i in range(n)])]
    pqs = [2 * p + 1 if case["double_quadrature"] else p for p in ps]
    lam = rng.uniform(0.2, 5.0, size=n)
    xs = []
    if shape == "sphere":
        xs = [_unit_sphere(ps[0])]
    elif shape == "drop":
        xs = [_unit_sphere(ps[0]) + _noise(rng, ps[0], 1, 6, 0.05)]
        lam[:] = 5.0
    elif shape == "pair":
        # nearly spherical drops on the z axis; the deformation moves the gap by less than half of it
        for k in range(2):
            x = _unit_sphere(ps[0]) + _noise(rng, ps[0], 2, 4, 0.2 * case["gap"])
            x[2, 0] += math.sqrt(4.0 * math.pi) * (1.0 + 0.5 * case["gap"]) * (1 - 2 * k)
            xs.append(x)
        lam[:] = 0.5
    else:
        if shape == "spheres":
            radii = rng.uniform(0.8, 1.2, size=n)
            forms = [r * _unit_sphere(p) for r, p in zip(radii, ps)]
        else:
            axes = rng.uniform(0.7, 1.3, size=(n, 3))
            radii = axes.max(axis=1) + 0.1
            forms = [_rotation(rng) @ np.diag(a) @ _unit_sphere(p) + _noise(rng, p, 2, 8, 0.1) for a, p in zip(axes, ps)]
        for x, c in zip(forms, _place(rng, radii, 0.5)):
            x[:, 0] += math.sqrt(4.0 * math.pi) * c
            xs.append(x)
    dens = [_band(rng, p, 3) for p in ps]
    gam = []
    for p in ps:
        g = 0.1 * _band(rng, p, 1)
        g[0, 0] = math.sqrt(4.0 * math.pi)
        gam.append(g)
    far = []  # u_inf = (shear z, 0, 0)
    for x in xs:
        u = np.zeros_like(x)
        u[0] = SHEAR * x[2]
        far.append(u)
    return {"p": ps, "pq": pqs, "lam": lam, "x": xs, "dens": dens, "gamma": gam, "far": far, "rng": rng}


def _points(inp, count):
    """Fluid points: most uniform in the drops' box outside every bounding sphere, one in eight 0.06 off a
    surface, along the ray from the drop's centre."""
    rng, xs, ps = inp["rng"], inp["x"], inp["p"]
    cen = np.array([x[:, 0] for x in xs]) / math.sqrt(4.0 * math.pi)
    near = count // 8
    got = []
    s = rng.standard_normal((near, 3))
    s /= np.linalg.norm(s, axis=1)[:, None]
    owner = rng.integers(0, len(ps), size=near)
    for p in sorted(set(ps)):
        sel = [k for k in range(near) if ps[owner[k]] == p]
        if sel:
            B = _basis(torch.tensor(s[sel]), p)[0].numpy()
            at = np.stack([xs[owner[k]] @ B[i] for i, k in enumerate(sel)])
            ray = at - cen[owner[sel]]
            got.append(at + 0.06 * ray / np.linalg.norm(ray, axis=1)[:, None])
    lo, hi = cen.min(axis=0) - 2.0, cen.max(axis=0) + 2.0
    left = count - near
    while left > 0:
        c = rng.uniform(lo, hi, size=(2 * left + 64, 3))
        ok = np.ones(len(c), dtype=bool)
        for k in range(len(ps)):
            ok &= np.sum((c - cen[k]) ** 2, axis=1) > 1.6 ** 2
        c = c[ok][:left]
        left -= len(c)
        got.append(c)
    return np.ascontiguousarray(np.concatenate(got).T)


def _flat(blocks):
    return torch.tensor(np.concatenate([np.asarray(b).reshape(-1) for b in blocks]), device="cuda")


_CONTEXTS = {}


def _context(up):
    """A program keeps one context (plan tables per degree) and makes its geometries in it."""
    if up not in _CONTEXTS:
        _CONTEXTS[up] = api.Context(0, upsample=up)
    return _CONTEXTS[up]


def prepare(case, seed):
    inp = _inputs(case, seed)
    kind = case["kind"]
    s = {"case": case, "p": inp["p"], "pq": inp["pq"], "lam": [float(v) for v in inp["lam"]], "ctx": _context(case["up"]),
         "x": _flat(inp["x"]), "f": _flat(inp["dens"]), "prec": PRECISION[case["precision"]]}
    if kind in ("apply", "rhs", "solve", "velocity"):
        s["geo"] = s["ctx"].geometry(s["p"], s["pq"], s["x"], s["lam"])
        s["out"] = torch.zeros_like(s["f"])
    if kind in ("rhs", "solve", "setup"):
        s["far"] = _flat(inp["far"])
        s["b"] = torch.zeros_like(s["f"])
    if kind in ("setup", "surfactant", "step"):
        s["gamma"] = _flat(inp["gamma"])
    if kind == "surfactant":
        s["fe"], s["fi"], s["y"] = (torch.zeros_like(s["gamma"]) for _ in range(3))
    if kind == "setup":
        s["force"] = torch.zeros_like(s["f"])
    if kind == "velocity":
        s["u"] = _flat([_band(inp["rng"], p, 3) for p in inp["p"]])
        pts = torch.tensor(_points(inp, case["points"]), device="cuda")
        far = torch.zeros_like(pts)
        far[0] = SHEAR * pts[2]
        s.update(points=pts, points_far=far, v=torch.zeros_like(pts))
    if kind == "step":
        s["u0"], s["x1"], s["g1"] = torch.zeros_like(s["x"]), torch.zeros_like(s["x"]), torch.zeros_like(s["gamma"])
    return s


def _as_computed(s, t):
    return t.float() if s["case"]["precision"] == "mixed" else t


def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"]
    if kind == "apply":
        g = s["geo"]
        (g.apply_single if s["case"]["layer"] == "single" else g.apply_double)(s["f"], s["out"], precision=s["prec"])
        return _as_computed(s, s["out"])
    if kind == "rhs":
        return s["geo"].rhs(s["far"], s["f"], s["b"], precision=api.BIE_DF)
    if kind == "solve":
        s["geo"].rhs(s["far"], s["f"], s["b"], precision=api.BIE_DF)
        s["out"].zero_()
        s["geo"].solve(s["b"], s["out"], precision=api.BIE_MIXED, tol=1e-10)
        return {"b": s["b"], "u": s["out"]}
    if kind == "setup":
        g = ctx.geometry(s["p"], s["pq"], s["x"], s["lam"])
        g.interfacial_force(s["gamma"], ELASTICITY, 0.0, s["force"])
        g.rhs(s["far"], s["force"], s["b"], precision=api.BIE_DF)
        g.close()
        return {"force": s["force"], "b": s["b"]}
    if kind == "surfactant":
        api.surfactant_rates(ctx, s["p"], s["x"], s["f"], s["gamma"], INV_PE, s["fe"], s["fi"])
        api.surfactant_implicit(ctx, s["p"], s["x"], s["gamma"], 0.5 * DT * INV_PE, s["y"])
        return {"fe": s["fe"], "fi": s["fi"], "y": s["y"]}
    if kind == "velocity":
        s["geo"].velocity_at(s["points"], s["f"], s["u"], s["v"], uinf=s["points_far"], precision=s["prec"])
        return _as_computed(s, s["v"])
    api.coupled_step(ctx, s["p"], s["pq"], s["x"], s["gamma"], s["u0"], False, ELASTICITY, 0.0, s["lam"], SHEAR, INV_PE, DT,
                     s["x1"], s["g1"])
    return {"x": s["x1"], "gamma": s["g1"], "u": s["u0"]}


# ------------------------------------------------------------------------------------------------
# work
# ------------------------------------------------------------------------------------------------
def work(case):
    """Bytes: densities, shapes and the self rule's operator (6 symmetric 3x3 entries per target and
    coefficient, what an apply has to read of a kept geometry) read once, results written once.  Flops:
    that operator's products and about 30 per inter-drop pair."""
    choice = [int(v) for v in str(case["degrees"]).split(",")]
    n = case["n"]
    ps = [choice[i % len(choice)] for i in range(n)]
    word = 4 if case["precision"] == "mixed" else 8
    nt = [2 * _nc(p) for p in ps]
    coef = sum(3 * 8 * _nc(p) for p in ps)
    self_b, self_f = sum(6 * t * _nc(p) * word for t, p in zip(nt, ps)), sum(18 * t * _nc(p) for t, p in zip(nt, ps))
    pairs = sum(nt) ** 2 - sum(t * t for t in nt)
    kind = case["kind"]
    if kind in ("apply", "rhs"):
        return {"bytes": 2 * coef + self_b + 7 * 8 * sum(nt) * (n > 1), "flops": self_f + 30 * pairs}
    if kind == "solve":  # one operator and one right-hand side, about 15 matvecs
        return {"bytes": 2 * self_b + 4 * coef, "flops": 16 * (self_f + 30 * pairs)}
    if kind == "setup":
        # the rotated grids and kernel weights of every target, one right-hand side
        rot = sum(t * 2 * (p + 1) ** 3 * 12 for t, p in zip(nt, ps))
        return {"bytes": 4 * coef + 2 * self_b, "flops": 4 * rot + self_f + 30 * pairs}
    if kind == "surfactant":
        grid = sum(8 * (p + 1) ** 2 for p in ps)
        return {"bytes": 4 * coef, "flops": sum(60 * 4 * (p + 1) * (p + 1) ** 2 for p in ps) * 8 + 400 * grid}
    if kind == "velocity":
        return {"bytes": 2 * coef + 9 * 8 * case["points"] + 7 * 8 * sum(nt), "flops": 60 * case["points"] * sum(nt)}
    rot = sum(t * 2 * (p + 1) ** 3 * 12 for t, p in zip(nt, ps))
    return {"bytes": 8 * coef + 4 * self_b, "flops": 2 * (4 * rot + 16 * (self_f + 30 * pairs))}


# ------------------------------------------------------------------------------------------------
# the method in plain torch, 64 bits
# ------------------------------------------------------------------------------------------------
def _gauss(P):
    t, w = np.polynomial.legendre.leggauss(P + 1)
    return t, w


def _legendre(ct, st, p):
    """Orthonormal associated Legendre functions with the Condon-Shortley phase, {(n, m): values}; for
    m > 0 those divided by sin(theta), which stay finite at the poles."""
    P = {}
    d = torch.full_like(ct, math.sqrt(1.0 / (4.0 * math.pi)))
    for m in range(p + 2):
        P[m, m] = d
        if m + 1 <= p + 1:
            P[m + 1, m] = math.sqrt(2.0 * m + 3.0) * ct * d
        for n in range(m + 2, p + 1):
            a = math.sqrt((4.0 * n * n - 1.0) / (n * n - m * m))
            b = math.sqrt(((n - 1.0) ** 2 - m * m) / (4.0 * (n - 1.0) ** 2 - 1.0))
            P[n, m] = a * (ct * P[n - 1, m] - b * P[n - 2, m])
        d = -math.sqrt(1.0 + 1.0 / (2.0 * (m + 1))) * d if m == 0 else -math.sqrt(1.0 + 1.0 / (2.0 * (m + 1))) * st * d
    return P


def _basis(s, p, order=0):
    """Real-packed basis at unit vectors s [..., 3]: B [..., (p+1)^2] with f = B c; for order 1 also its
    derivatives by theta and by phi, the latter divided by sin(theta) (the tangent derivatives, finite at
    the poles); for order 2 the derivatives t, p, tt, tp, pp as they are (not at the poles)."""
    ct = s[..., 2]
    st = torch.sqrt(s[..., 0] ** 2 + s[..., 1] ** 2)
    at = st > 0
    cp = torch.where(at, s[..., 0] / torch.where(at, st, 1.0), 1.0)
    sp = torch.where(at, s[..., 1] / torch.where(at, st, 1.0), 0.0)
    P = _legendre(ct, st, p)
    outs = [torch.zeros(s.shape[:-1] + (_nc(p),), dtype=s.dtype, device=s.device) for _ in range([1, 3, 6][order])]
    cm, sm = torch.ones_like(ct), torch.zeros_like(ct)
    for m in range(p + 1):
        f = 1.0 if m == 0 else 2.0
        for n in range(m, p + 1):
            q = P[n, m] * st if m else P[n, m]
            th = [q]
            if order:
                d = m * ct * P[n, m] if m else torch.zeros_like(q)
                if n > m:
                    d = d + math.sqrt((n - m) * (n + m + 1.0)) * P[n, m + 1] * st
                th.append(d)
            if order == 2:
                th.append(-ct / st * th[1] + (m * m / (st * st) - n * (n + 1.0)) * q)
            c, i = n * (n + 1) + m, n * (n + 1) - m
            # (theta order, phi order) of each output
            for o, (a, b) in zip(outs, ((0, 0), (1, 0), (0, 1), (2, 0), (1, 1), (0, 2))):
                if b and not m:
                    continue
                v = P[n, m] if order == 1 and b else th[a]
                re = [cm, -m * sm, -m * m * cm][b]
                im = [-sm, -m * cm, m * m * sm][b]
                if m:
                    o[..., i] = f * v * im
                o[..., c] = f * v * re
        cm, sm = cm * cp - sm * sp, sm * cp + cm * sp
    return outs


def _grid(P, dev):
    """Unit vectors [j][k] of the degree-P grid and its weights pi/(P+1) w_j."""
    t, w = _gauss(P)
    t, w = torch.tensor(t, device=dev), torch.tensor(w, device=dev)
    ph = math.pi / (P + 1) * torch.arange(2 * P + 2, device=dev, dtype=torch.float64)
    st = torch.sqrt((1 - t) * (1 + t))
    s = torch.stack([st[:, None] * torch.cos(ph), st[:, None] * torch.sin(ph), t[:, None].expand(-1, len(ph))], dim=-1)
    wt = (math.pi / (P + 1) * w)[:, None].expand(-1, len(ph))
    return s.reshape(-1, 3), wt.reshape(-1).contiguous()


def _analysis(B, wt, p):
    """Matrix of the Galerkin projection, coefficients from grid values, given the basis there."""
    n = torch.tensor(_degrees(p), device=B.device)
    m = torch.arange(_nc(p), device=B.device) - n * (n + 1)
    return (B[:, : _nc(p)] * torch.where(m == 0, 1.0, 0.5).to(B.dtype)).T * wt


def _kernel(xh, nw, w, kind):
    """Symmetric 3x3 kernel weights [..., 6] (xx yy zz xy xz yz): nw = area vector times weight, w = its norm."""
    r2 = (xh * xh).sum(-1)
    if kind == 0:
        ri = torch.rsqrt(r2)
        d, c = w * ri, w * ri / r2
    else:
        d = torch.zeros_like(r2)
        c = -6.0 * (xh * nw).sum(-1) / (r2 * r2 * torch.sqrt(r2))
    x, y, z = xh.unbind(-1)
    return torch.stack([d + c * x * x, d + c * y * y, d + c * z * z, c * x * y, c * x * z, c * y * z], dim=-1)


SYM = ((0, 3, 4), (3, 1, 5), (4, 5, 2))


class _Exact:
    """The operators of a set of drops (tensors in float64)."""

    def __init__(self, inp, up, dev):
        self.dev, self.up, self.p, self.pq, self.lam = dev, up, inp["p"], inp["pq"], inp["lam"]
        self.x = [torch.tensor(np.asarray(x), device=dev) for x in inp["x"]]
        self.n = len(self.p)
        self.tables = {}
        self.std = [self._sources(j, self.p[j]) for j in range(self.n)]
        self.ups = None
        self.h = []
        for j in range(self.n):
            y, area, _ = self._surface(j, 2 * self.p[j] + 1)
            vol = (self._tab(self.p[j], 2 * self.p[j] + 1)["wt"] * (y * area).sum(-1)).sum().item() / 3.0
            self.h.append((3.0 * vol / (4.0 * math.pi)) ** (1.0 / 3.0) * math.pi / (self.p[j] + 1))
        self.dense = {}

    def _tab(self, p, P, order=1):
        key = (p, P, order)
        if key not in self.tables:
            s, wt = _grid(P, self.dev)
            self.tables[key] = {"s": s, "wt": wt, "B": _basis(s, p, order)}
        return self.tables[key]

    def _surface(self, j, P):
        t = self._tab(self.p[j], P)
        y, yt, yp = (b @ self.x[j].T for b in t["B"])
        return y, torch.linalg.cross(yt, yp), t

    def _sources(self, j, P):
        """Positions, weighted area vectors, weights and the basis of drop j's grid of degree P."""
        y, area, t = self._surface(j, P)
        nw = area * t["wt"][:, None]
        return {"y": y, "nw": nw, "w": nw.norm(dim=-1), "B": t["B"][0]}

    def upsampled(self, j):
        if self.ups is None:
            self.ups = {}
        if j not in self.ups:
            self.ups[j] = self._sources(j, self.up * (self.p[j] + 1) - 1)
        return self.ups[j]

    # ---- the singular rule of Thm 1 ----
    def _weights(self, pq):
        """The weights w^s_j at every point of the degree-pq grid."""
        t, w = _gauss(pq)
        P = np.zeros((pq + 1, pq + 1))
        P[0], P[1] = 1.0, t
        for n in range(1, pq):
            P[n + 1] = ((2 * n + 1) * t * P[n] - n * P[n - 1]) / (n + 1)
        ws = math.pi / (pq + 1) * w * 2.0 * np.sqrt((1.0 - t) / 2.0) * P.sum(axis=0)
        return torch.tensor(np.repeat(ws, 2 * pq + 2), device=self.dev)

    def _turned(self, p, P):
        """The points R_y(theta_a) s of the degree-P grid for every latitude a of the degree-p grid, [a][q][3]."""
        s = _grid(P, self.dev)[0]
        ct = torch.tensor(_gauss(p)[0], device=self.dev)[:, None]
        st = torch.sqrt((1.0 - ct) * (1.0 + ct))
        return torch.stack([ct * s[:, 0] + st * s[:, 2], s[:, 1].expand(p + 1, -1), ct * s[:, 2] - st * s[:, 0]], dim=-1)

    def _phase(self, c, p, sign=1.0):
        """e^{i m phi_b} c for every longitude of the degree-p grid, [b][k][(p+1)^2], c [k] or [b][k] (sign -1:
        the transpose): the coefficients of f(R_z(phi_b) s)."""
        n = torch.tensor(_degrees(p), device=self.dev)
        m = torch.arange(_nc(p), device=self.dev) - n * (n + 1)
        ph = math.pi / (p + 1) * torch.arange(2 * p + 2, device=self.dev, dtype=torch.float64)[:, None] * m.abs()
        co, si = torch.cos(ph)[:, None], (-sign * torch.sign(m) * torch.sin(ph))[:, None]
        return c * co + c[..., n * (n + 1) - m] * si

    def _rotate(self, c, p):
        """Coefficients of f(R_z(phi_b) R_y(theta_a) s) for every target of the degree-p grid, [a b][k][(p+1)^2]."""
        key = ("rotation", p)
        if key not in self.tables:
            tab = self._tab(p, p)
            A, B = _analysis(tab["B"][0], tab["wt"], p), _basis(self._turned(p, p), p)[0]
            self.tables[key] = [A[n * n:(n + 1) ** 2] @ B[..., n * n:(n + 1) ** 2] for n in range(p + 1)]
        g = self._phase(c, p)
        out = torch.empty((p + 1,) + g.shape, device=self.dev, dtype=torch.float64)
        for n, D in enumerate(self.tables[key]):
            out[..., n * n:(n + 1) ** 2] = (g[..., n * n:(n + 1) ** 2].reshape(-1, 2 * n + 1) @ D.transpose(1, 2)).reshape(out[..., n * n:(n + 1) ** 2].shape)
        return out.flatten(0, 1)

    def _synthesis(self, c, p, P, derivatives):
        """Values [t][k][q] on the degree-P grid from coefficients [t][k][(p+1)^2] (and the tangent derivatives)."""
        key = ("synthesis", p, P)
        if key not in self.tables:
            s = _grid(P, self.dev)[0].reshape(P + 1, -1, 3)[:, 0]
            T = torch.zeros(3, p + 1, p + 1, P + 1, device=self.dev, dtype=torch.float64)  # [kind][m][n][j]
            for k, b in enumerate(_basis(s, p, 1)):
                for n in range(p + 1):
                    for m in range(n + 1):
                        T[k, m, n] = -b[:, n * (n + 1) - m] if k == 2 else b[:, n * (n + 1) + m]
            ph = math.pi / (P + 1) * torch.outer(torch.arange(p + 1, device=self.dev), torch.arange(2 * P + 2, device=self.dev)).double()
            self.tables[key] = T, torch.cat([torch.cos(ph), -torch.sin(ph)]), torch.cat([-torch.sin(ph), -torch.cos(ph)])
        T, E0, E1 = self.tables[key]
        m, n = torch.meshgrid(torch.arange(p + 1, device=self.dev), torch.arange(p + 1, device=self.dev), indexing="ij")
        keep = (n >= m).double()
        lead = c.shape[:-1]
        c = c.reshape(-1, _nc(p))
        re = (c[:, (n * (n + 1) + m).clamp(max=_nc(p) - 1)] * keep).transpose(0, 1)  # [m][t k][n]
        im = (c[:, (n * (n + 1) - m).clamp(min=0)] * keep * (m > 0)).transpose(0, 1)
        both = torch.cat([re, im], dim=1)
        outs = []
        for k, E in ((0, E0), (1, E0), (2, E1))[:3 if derivatives else 1]:
            h = both @ T[k]  # [m][2 t k][j]
            h = torch.cat(h.split(len(c), dim=1), dim=0).permute(1, 2, 0)  # [t k][j][2 (p+1)]
            outs.append((h @ E).reshape(lead + (-1,)))
        return outs

    def _rotated_geometry(self, j):
        """x0 - x' and the weighted area vectors on every target's rotated grid, [t][q][3]."""
        p, pq = self.p[j], self.pq[j]
        y, yt, yp = (v.transpose(1, 2) for v in self._synthesis(self._rotate(self.x[j], p), p, pq, True))
        return self.std[j]["y"][:, None] - y, torch.linalg.cross(yt, yp) * self._weights(pq)[:, None]

    def self_values(self, kind, dens):
        """Raw values [target][3] of every drop's own integral; dens: list of [3][(p+1)^2]."""
        out = []
        for j in range(self.n):
            xh, area = self._rotated_geometry(j)
            q = self._synthesis(self._rotate(dens[j], self.p[j]), self.p[j], self.pq[j], False)[0].transpose(1, 2)
            out.append(self._contract(xh, area, q, kind).sum(1))
        return out

    @staticmethod
    def _contract(xh, nw, q, kind, w=None):
        """Kernel times density: w G q (single) or -6 (q.xh)(xh.nw) xh / r^5 (double)."""
        r2 = (xh * xh).sum(-1)
        xq = (xh * q).sum(-1)
        if kind == 0:
            w = nw.norm(dim=-1) if w is None else w
            ri = torch.rsqrt(r2) * w
            return q * ri[..., None] + xh * (xq * ri / r2)[..., None]
        return xh * (-6.0 * xq * (xh * nw).sum(-1) / (r2 * r2 * torch.sqrt(r2)))[..., None]

    def self_matrix(self, kind, j):
        """The same as a matrix [target][3][3][(p+1)^2]."""
        p, pq = self.p[j], self.pq[j]
        if (kind, j) not in self.dense:
            M = torch.empty(2 * _nc(p), 6, _nc(p), device=self.dev, dtype=torch.float64)
            xh, area = self._rotated_geometry(j)
            K = _kernel(xh, area, area.norm(dim=-1), kind).transpose(1, 2).contiguous()
            B, nb = _basis(self._turned(p, pq), p)[0], 2 * p + 2
            for a in range(p + 1):
                rows = (K[a * nb:(a + 1) * nb].reshape(-1, K.shape[-1]) @ B[a]).reshape(nb, 6, -1)
                M[a * nb:(a + 1) * nb] = self._phase(rows, p, -1.0)
            self.dense[kind, j] = M
        return self.dense[kind, j]

    # ---- inter-drop rules ----
    def _regions(self, pts, j):
        """0, 1, 2 of each point with respect to drop j (Sec. 2.3)."""
        cen = self.x[j][:, 0] / math.sqrt(4.0 * math.pi)
        d = (pts - cen).norm(dim=1)
        reg = torch.zeros(len(pts), dtype=torch.long, device=self.dev)
        close = torch.nonzero(d <= (self.std[j]["y"] - cen).norm(dim=1).max() * 1.1 + 5.0 * self.h[j] + 0.1)[:, 0]
        y = self.upsampled(j)["y"] if len(close) else None
        for k in range(0, len(close), 512):
            sel = close[k:k + 512]
            m = (pts[sel][:, None] - y[None]).norm(dim=2).min(dim=1).values
            reg[sel] = (m <= 5.0 * self.h[j]).long() + (m <= self.h[j]).long()
        return reg

    def _sum(self, pts, src, dens, kind):
        """Regular rule at points [n][3] from a drop's sources."""
        q = src["B"] @ dens.T
        out = torch.empty_like(pts)
        per = max(1, int(1.5e8 // len(q)))
        for k in range(0, len(pts), per):
            out[k:k + per] = self._pairs(pts[k:k + per], src, q, kind)
        return out

    @staticmethod
    def _pairs(pts, src, q, kind):
        y, nw, w = src["y"], src["nw"], src["w"]
        d = [pts[:, c:c + 1] - y[None, :, c] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        xq = d[0] * q[:, 0] + d[1] * q[:, 1] + d[2] * q[:, 2]
        if kind == 0:
            ri = torch.rsqrt(r2)
            c = xq * ri * ri
            ri *= w
            c *= ri
            return ri @ q + torch.stack([(c * d[k]).sum(1) for k in range(3)], dim=1)
        r2 = torch.rsqrt(r2)
        c = xq * (d[0] * nw[:, 0] + d[1] * nw[:, 1] + d[2] * nw[:, 2]) * r2
        r2 *= r2
        c *= r2
        c *= r2 * -6.0
        return torch.stack([(c * d[k]).sum(1) for k in range(3)], dim=1)

    def _closest(self, pts, js):
        """Closest points of the drops js (of one degree) as rows of the basis there, and positions."""
        p = self.p[js[0]]
        y, x = torch.stack([self.std[j]["y"] for j in js]), torch.stack([self.x[j].T for j in js])
        k = torch.cat([((q[:, None] - y[i]) ** 2).sum(-1).argmin(dim=1) for i, q in enumerate(pts)])
        x = x[torch.cat([torch.full((len(q),), i, device=self.dev) for i, q in enumerate(pts)])]
        s, pts = self._tab(p, p)["s"][k].clone(), torch.cat(pts)

        def at(b):
            return torch.bmm(b[:, None], x)[:, 0]

        for _ in range(18):  # Gauss-Newton in the tangent plane of the parameter sphere
            B, Bt, Bp = _basis(s, p, 1)
            ct, st = s[:, 2:], torch.sqrt(s[:, :1] ** 2 + s[:, 1:2] ** 2)
            e1 = torch.cat([s[:, :2] * ct / st, -st], dim=1)
            e2 = torch.cat([-s[:, 1:2], s[:, :1], torch.zeros_like(st)], dim=1) / st
            J = torch.stack([at(Bt), at(Bp)], dim=2)
            a = torch.linalg.solve(J.transpose(1, 2) @ J, J.transpose(1, 2) @ (pts - at(B))[:, :, None])[:, :, 0]
            s = s + a[:, :1] * e1 + a[:, 1:] * e2
            s = s / s.norm(dim=1, keepdim=True)
        B = _basis(s, p)[0]
        return B, at(B)

    def plan(self, points):
        """The region of every point of points[j] with respect to drop j, and the interpolation's data."""
        plans = []
        for j, pts in enumerate(points):
            reg = self._regions(pts, j)
            plans.append({r: torch.nonzero(reg == k)[:, 0] for k, r in enumerate(("far", "mid", "near"))})
        for p in sorted(set(self.p)):
            js = [j for j in range(self.n) if self.p[j] == p and len(plans[j]["near"])]
            if not js:
                continue
            near = [points[j][plans[j]["near"]] for j in js]
            B, xs = self._closest(near, js)
            size = [len(q) for q in near]
            for j, q, b, x in zip(js, near, B.split(size), xs.split(size)):
                d0 = (q - x).norm(dim=1)
                e = (q - x) / d0[:, None]
                nodes = [0.0] + [self.h[j] * math.sqrt(l) for l in range(1, 9)]
                lag = []
                for l in range(9):
                    v = torch.ones_like(d0)
                    for k in range(9):
                        if k != l:
                            v = v * (d0 - nodes[k]) / (nodes[l] - nodes[k])
                    lag.append(v)
                chk = [x + nodes[l] * e for l in range(1, 9)]
                plans[j].update(B=b, lag=lag, chk=chk, reg=[self._regions(c, j) for c in chk])
        return plans

    def _near(self, plan, j, kind, dens, self_coef):
        """Interpolation through the exterior limit at x* and eight check points."""
        v = plan["B"] @ self_coef.T
        if kind == 1:
            v = v - 4.0 * math.pi * (plan["B"] @ dens.T)
        out = plan["lag"][0][:, None] * v
        for l in range(8):
            c, reg = plan["chk"][l], plan["reg"][l]
            for far, src in ((True, self.std[j]), (False, self.upsampled(j))):
                sel = torch.nonzero((reg == 0) == far)[:, 0]
                if len(sel):
                    out[sel] += plan["lag"][l + 1][sel][:, None] * self._sum(c[sel], src, dens, kind)
        return out

    def _add_from(self, out, pts, j, kind, weight, dens, self_coef, P):
        """out += weight * integral over drop j at the points."""
        if len(P["far"]):
            out[P["far"]] += weight * self._sum(pts[P["far"]], self.std[j], dens, kind)
        if len(P["mid"]):
            out[P["mid"]] += weight * self._sum(pts[P["mid"]], self.upsampled(j), dens, kind)
        if len(P["near"]):
            out[P["near"]] += weight * self._near(P, j, kind, dens, self_coef)

    def weight(self, kind, j):
        return -1.0 / (4.0 * math.pi) if kind == 0 else (self.lam[j] - 1.0) / (4.0 * math.pi)

    def project(self, vals, j):
        t = self._tab(self.p[j], self.p[j])
        return (_analysis(t["B"][0], t["wt"], self.p[j]) @ vals).T

    def apply(self, kind, dens, plans, dense=False):
        if dense:
            own = []
            for j in range(self.n):
                M = self.self_matrix(kind, j)
                v = M.reshape(-1, _nc(self.p[j])) @ dens[j].T
                v = v.reshape(-1, 6, 3)
                own.append(torch.stack([sum(v[:, SYM[a][b], b] for b in range(3)) for a in range(3)], dim=1))
        else:
            own = self.self_values(kind, dens)
        total = [self.weight(kind, j) * own[j] for j in range(self.n)]
        if self.n > 1:
            coef = [self.project(v, j) for j, v in enumerate(own)]
            pts = torch.cat([s["y"] for s in self.std])
            at = np.cumsum([0] + [len(v) for v in own])
            rest = [torch.cat([torch.arange(0, at[j]), torch.arange(at[j + 1], at[-1])]).to(self.dev) for j in range(self.n)]
            if not plans:
                plans.extend(self.plan([pts[r] for r in rest]))
            both = torch.cat(total)
            for j, r in enumerate(rest):
                v = torch.zeros(len(r), 3, device=self.dev, dtype=torch.float64)
                self._add_from(v, pts[r], j, kind, self.weight(kind, j), dens[j], coef[j], plans[j])
                both[r] += v
            total = [both[at[j]:at[j + 1]] for j in range(self.n)]
        return [self.project(v, j) for j, v in enumerate(total)]

    def velocity(self, pts, dens, u):
        out, plans = torch.zeros_like(pts), self.plan([pts] * self.n)
        for kind, d in ((0, dens), (1, u)):
            coef = [self.project(v, j) for j, v in enumerate(self.self_values(kind, d))]
            for j in range(self.n):
                self._add_from(out, pts, j, kind, 0.5 * self.weight(kind, j), d[j], coef[j], plans[j])
        return out

    # ---- surface calculus on the grid of degree 2p+1 ----
    def calculus(self, j):
        p = self.p[j]
        t = self._tab(p, 2 * p + 1, 2)
        y, yt, yp, ytt, ytp, ypp = (b @ self.x[j].T for b in t["B"])
        G, F, E = (yt * yt).sum(1), (yt * yp).sum(1), (yp * yp).sum(1)
        W2 = E * G - F * F
        return {"t": t, "d": (y, yt, yp, ytt, ytp, ypp), "g": (E / W2, -F / W2, G / W2), "W2": W2,
                "A": _analysis(t["B"][0], t["wt"], p), "EFG": (E, F, G)}

    def force(self, j, gamma):
        c = self.calculus(j)
        y, yt, yp, ytt, ytp, ypp = c["d"]
        n = torch.linalg.cross(yt, yp) / torch.sqrt(c["W2"])[:, None]
        gtt, gtp, gpp = c["g"]
        K = 0.5 * (gtt * (ytt * n).sum(1) + 2.0 * gtp * (ytp * n).sum(1) + gpp * (ypp * n).sum(1))
        g, gt, gp = (b @ gamma for b in c["t"]["B"][:3])
        st, sp = -ELASTICITY * gt, -ELASTICITY * gp
        grad = (gtt * st + gtp * sp)[:, None] * yt + (gtp * st + gpp * sp)[:, None] * yp
        return (c["A"] @ (-2.0 * ((1.0 - ELASTICITY * g) * K)[:, None] * n - grad)).T

    def surfactant(self, j, u, gamma, a):
        """Explicit rate -Gamma div u, diffusive rate and the implicit stage (I - a lap) y = Gamma."""
        c = self.calculus(j)
        y, yt, yp, ytt, ytp, ypp = c["d"]
        gtt, gtp, gpp = c["g"]
        B = c["t"]["B"]
        ut, up = B[1] @ u.T, B[2] @ u.T
        div = gtt * (yt * ut).sum(1) + gtp * ((yt * up).sum(1) + (yp * ut).sum(1)) + gpp * (yp * up).sum(1)
        trace = gtt[:, None] * ytt + 2.0 * gtp[:, None] * ytp + gpp[:, None] * ypp
        bt, bp = (trace * yt).sum(1), (trace * yp).sum(1)
        lap = (gtt[:, None] * B[3] + 2.0 * gtp[:, None] * B[4] + gpp[:, None] * B[5]
               - (gtt * bt + gtp * bp)[:, None] * B[1] - (gtp * bt + gpp * bp)[:, None] * B[2])
        L = c["A"] @ lap
        eye = torch.eye(len(L), device=self.dev, dtype=torch.float64)
        return c["A"] @ (-(B[0] @ gamma) * div), INV_PE * (L @ gamma), torch.linalg.solve(eye - a * L, gamma)


def _gmres(op, b, tol=1e-13, steps=60):
    V, H = [b / b.norm()], torch.zeros(steps + 1, steps, dtype=torch.float64)
    for k in range(steps):
        w = op(V[k])
        for _ in range(2):
            for i, v in enumerate(V):
                h = (v @ w).item()
                H[i, k] += h
                w = w - h * v
        H[k + 1, k] = w.norm().item()
        e = torch.zeros(k + 2, dtype=torch.float64)
        e[0] = b.norm().item()
        y = torch.tensor(np.linalg.lstsq(H[:k + 2, :k + 1].numpy(), e.numpy(), rcond=None)[0])
        if (H[:k + 2, :k + 1] @ y - e).norm() <= tol * e[0] or H[k + 1, k] <= 1e-15:
            break
        V.append(w / H[k + 1, k].item())
    return sum(c.item() * v for c, v in zip(y, V))


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return None  # two solves and the surfactant scheme around them
    inp = _inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"

    def on(blocks):
        return [torch.tensor(np.asarray(b), device=dev) for b in blocks]

    E = _Exact(inp, case["up"], dev)
    dens, far, plans = on(inp["dens"]), on(inp["far"]), []
    flat = lambda blocks: torch.cat([b.reshape(-1) for b in blocks])  # noqa: E731
    if kind == "apply":
        return flat(E.apply(0 if case["layer"] == "single" else 1, dens, plans))
    if kind == "rhs":
        return 2.0 * flat(far) + flat(E.apply(0, dens, plans))
    if kind == "setup":
        force = [E.force(j, g[0]) for j, g in enumerate(on(inp["gamma"]))]
        return {"force": flat(force), "b": 2.0 * flat(far) + flat(E.apply(0, force, plans))}
    if kind == "surfactant":
        got = [E.surfactant(j, dens[j], g[0], 0.5 * DT * INV_PE) for j, g in enumerate(on(inp["gamma"]))]
        return {k: flat([r[i] for r in got]) for i, k in enumerate(("fe", "fi", "y"))}
    if kind == "velocity":
        u = on([_band(inp["rng"], p, 3) for p in inp["p"]])
        pts = torch.tensor(_points(inp, case["points"]), device=dev)
        v = E.velocity(pts.T.contiguous(), dens, u).T.contiguous()
        v[0] += SHEAR * pts[2]
        return v
    b = 2.0 * flat(far) + flat(E.apply(0, dens, plans, dense=True))
    E.dense.clear()
    size = [3 * _nc(p) for p in E.p]
    scale = torch.cat([torch.full((k,), E.lam[j] + 1.0, device=dev, dtype=torch.float64) for j, k in enumerate(size)])

    def system(u):
        parts = [v.reshape(3, -1) for v in torch.split(u, size)]
        return scale * u - flat(E.apply(1, parts, plans, dense=True))

    return {"b": b, "u": _gmres(system, b)}
