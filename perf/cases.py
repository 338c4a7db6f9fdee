"""Performance cases of the Yin-Yang gravity solver.

A case is one call of a user's time step: Phi, or Phi and -grad Phi, of the
densities a simulation holds on the GPU, on a grid handle it keeps, in one of
the library's arithmetic forms; or one batched step over several fields.

listed()  the grids of the package (tiny, mid, production and the batched
          fields), the one-degree spherical polar grid and a ragged grid of
          high degree, each in a form that such a grid is solved in
draw()    another grid of the same ranges, odd sizes among them
prepare() the grid handle with its tables, the densities and the output arrays
run()     one solve through yy.Grid.potential / yy.Batch.potential
work()    the densities read once and the results written once, and the
          multiply-adds of the two separable sums
exact()   the same solve from the method's definitions in plain float64 torch

Densities are the package's analytic ones, evaluated on the GPU: a steep
proto-neutron-star profile with an angular perturbation of degree <= 4
("core"), an oblate, rotation-like body with cell noise ("oblate"), and two
homogeneous spheres ("spheres").
"""

import math

import numpy as np
import torch

from paper_1806_04593_gb300 import inputs, yy

PRECISIONS = ("fp64_ozaki", "fp64", "fp32", "fp16x2", "bf16x3", "tf32")


def _case(name, n_r, r_min, n_theta, n_phi, l_max, precision, gradient, *, grid="yinyang", buffer=0, density="core"):
    """`buffer`: width of the patches' buffer zones in cells, in theta and in phi."""
    return {"name": name, "grid": grid, "n_r": n_r, "r_min": r_min, "n_theta": n_theta, "n_phi": n_phi, "buffer": buffer,
            "l_max": l_max, "precision": precision, "gradient": gradient, "density": density}


def listed():
    return [
        # a small validation grid, solved again and again: the call's latency
        _case("tiny_fp64", 32, 1e-3, 16, 48, 8, "fp64", True, buffer=2, density="spheres"),
        # two-degree production-like runs in the paper's arithmetic, in single precision, and Phi alone (an energy diagnostic)
        _case("mid_fp64", 200, 1e-3, 45, 135, 15, "fp64", True, density="oblate"),
        _case("mid_fp32", 200, 1e-3, 45, 135, 15, "fp32", True, density="oblate"),
        _case("mid_ozaki_phi", 200, 1e-3, 45, 135, 15, "fp64_ozaki", False, density="oblate"),
        # the one-degree stellar-core grid, gravity source terms of every time step: each form that is offered for it
        _case("production_ozaki", 550, 1e-4, 90, 270, 25, "fp64_ozaki", True),
        _case("production_fp64", 550, 1e-4, 90, 270, 25, "fp64", True),
        _case("production_fp32", 550, 1e-4, 90, 270, 25, "fp32", True),
        _case("production_fp16x2", 550, 1e-4, 90, 270, 25, "fp16x2", True),
        _case("production_bf16x3_phi", 550, 1e-4, 90, 270, 25, "bf16x3", False),
        # the full spherical polar grid that the paper compares with, one-degree cells
        _case("polar_ozaki", 300, 1e-4, 180, 360, 25, "fp64_ozaki", True, grid="polar"),
        # sizes that fit no tile, high degree
        _case("ragged_ozaki", 317, 1e-3, 61, 185, 40, "fp64_ozaki", True, buffer=1, density="oblate"),
        # many independent fields of uneven size per step
        {"name": "batch_fp16x2", "grid": "batch", "fields": 16, "first_seed": 100, "precision": "fp16x2", "gradient": True},
    ]


def _cells(case):
    """(cells x orders) summed over the fields, the azimuthal work of one evaluated field."""
    if case["grid"] == "batch":
        return sum(2 * s.n_r * s.n_ang * (2 * s.lmax + 1) for s, _, _ in inputs.batched_specs(case["fields"], case["first_seed"]))
    patches = 1 if case["grid"] == "polar" else 2
    return patches * case["n_r"] * case["n_theta"] * case["n_phi"] * (2 * case["l_max"] + 1)


def draw(rng):
    most = _cells(_case("", 550, 1e-4, 90, 270, 25, "fp64", True))
    between = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    if rng.random() < 0.1:
        return {"grid": "batch", "fields": between(3, 16), "first_seed": rng.randrange(200, 100000),
                "precision": rng.choice(("fp16x2", "fp64_ozaki", "bf16x3")), "gradient": rng.random() < 0.7}
    while True:
        grid = "polar" if rng.random() < 0.2 else "yinyang"
        n_theta = between(16, 180 if grid == "polar" else 90)
        square = 2 * n_theta if grid == "polar" else 3 * n_theta          # about square cells
        n_phi = square if rng.random() < 0.4 else max(24, square + rng.randint(-9, 9))
        case = _case("", between(30, 600), rng.choice((1e-4, 1e-3, 1e-2)), n_theta, n_phi, between(6, min(60, n_theta)),
                     rng.choices(PRECISIONS, (30, 20, 15, 20, 10, 5))[0], rng.random() < 0.7, grid=grid,
                     buffer=0 if grid == "polar" else rng.choice((0, 0, 1, 2)), density=rng.choice(("core", "oblate")))
        del case["name"]
        if _cells(case) <= most:
            return case


# ---------------------------------------------------------------------------
# the grid and its densities
# ---------------------------------------------------------------------------

def _spec(case):
    r_edges = np.logspace(math.log10(case["r_min"]), 0.0, case["n_r"] + 1)
    n_t, n_p, b = case["n_theta"], case["n_phi"], case["buffer"]
    if case["grid"] == "polar":
        return inputs.polar_grid(r_edges, n_t, n_p, case["l_max"])
    # n cells span the patch's range and a buffer of b cells on either side
    d_t, d_p = 0.5 * math.pi / (n_t - 2 * b), 1.5 * math.pi / (n_p - 2 * b)
    return inputs.GridSpec("case", r_edges, n_t, n_p, b * d_t, b * d_p, case["l_max"])


def _fields(case):
    """[(spec, density kind, perturbation)] of the case's fields."""
    if case["grid"] == "batch":
        return [(s, "core", e) for s, _, e in inputs.batched_specs(case["fields"], case["first_seed"])]
    return [(_spec(case), case["density"], 0.02)]


def _patches(spec):
    return ("yin",) if spec.polar else ("yin", "yang")


def _densities(spec, kind, eps_scale, seed):
    """The density of each patch, [n_r][n_theta][n_phi] float64 on the GPU."""
    rng = np.random.default_rng(seed)
    noise = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    r_c, units = inputs.cell_centres(spec)
    r = put(r_c)[:, None, None]
    powers = [(a, b, d - a - b) for d in range(1, 5) for a in range(d + 1) for b in range(d + 1 - a)]
    eps = rng.normal(0.0, eps_scale, len(powers))
    where = rng.uniform(-0.3, 0.3, 3)
    out = []
    for q in _patches(spec):
        x, y, z = (put(c) for c in units[q])
        if kind == "core":
            angular = 1.0 + sum(float(e) * x ** a * y ** b * z ** c for e, (a, b, c) in zip(eps, powers))
            rho = (torch.exp(-r / 0.02) + 1e-4 * r ** -2.5) * angular
        elif kind == "oblate":
            rho = (1.0 + r * r * ((x * x + y * y) / 0.04 + z * z / 0.0225)) ** -2
            rho = rho * (1.0 + 0.05 * torch.randn(rho.shape, generator=noise, dtype=torch.float64, device="cuda"))
        else:
            away = (r * x - where[0]) ** 2 + (r * y - where[1]) ** 2 + (r * z - where[2]) ** 2
            rho = (r <= 0.3).double() + 5.0 * (away <= 0.01).double()
        out.append(rho.contiguous())
    return out


def prepare(case, seed):
    fields = _fields(case)
    rho = [_densities(spec, kind, eps, seed * 1000 + f) for f, (spec, kind, eps) in enumerate(fields)]
    phi = [[torch.empty_like(x) for x in r] for r in rho]
    grad = [[torch.empty((3,) + tuple(x.shape), dtype=x.dtype, device=x.device) for x in r] for r in rho] if case["gradient"] else None
    if case["grid"] == "batch":
        solver = yy.Batch([spec for spec, _, _ in fields])
    else:
        solver = yy.Grid.from_spec(fields[0][0])
    solver.prepare(case["precision"])
    return {"case": case, "solver": solver, "rho": rho, "phi": phi, "grad": grad}


def run(state):
    case, rho, phi, grad = state["case"], state["rho"], state["phi"], state["grad"]
    stream = torch.cuda.current_stream()
    if case["grid"] == "batch":
        side = lambda a, q: None if a is None else [x[q] for x in a]  # noqa: E731
        state["solver"].potential(side(rho, 0), side(rho, 1), side(phi, 0), side(phi, 1), side(grad, 0), side(grad, 1),
                                  prec=case["precision"], stream=stream)
        return {"phi": phi, "grad": grad}
    other = lambda a: a[1] if len(a) > 1 else None  # noqa: E731
    g = grad[0] if grad else [None, None]
    state["solver"].potential(rho[0][0], other(rho[0]), phi[0][0], other(phi[0]), g[0], other(g),
                              prec=case["precision"], stream=stream)
    return {"phi": phi, "grad": grad}


def work(case):
    outs = 4 if case["gradient"] else 1
    n_bytes, flops = 0, 0
    for spec, _, _ in _fields(case):
        cells = (1 if spec.polar else 2) * spec.n_r * spec.n_ang
        n_bytes += 8 * cells * (1 + outs)
        polar = (1 if spec.polar else 2) * spec.n_r * spec.n_theta * (spec.lmax + 1) ** 2
        flops += 2 * (1 + outs) * (cells * (2 * spec.lmax + 1) + polar)
    return {"bytes": n_bytes, "flops": flops}


# ---------------------------------------------------------------------------
# the solve in plain float64
# ---------------------------------------------------------------------------

def _legendre(l_max, theta):
    """K_lm P_l^m(cos theta) with 4 pi / (2 l + 1) K^2 = N^(lm), Condon-Shortley phase: [l][m][...]."""
    x, s = torch.cos(theta), torch.sin(theta)
    P = torch.zeros((l_max + 1, l_max + 1) + tuple(theta.shape), dtype=torch.float64, device=theta.device)
    P[0, 0] = 1.0 / math.sqrt(4.0 * math.pi)
    for m in range(1, l_max + 1):
        P[m, m] = -math.sqrt((2 * m + 1) / (2.0 * m) * (2.0 if m == 1 else 1.0)) * s * P[m - 1, m - 1]
    for l in range(1, l_max + 1):
        m = torch.arange(l, dtype=torch.float64, device=theta.device).reshape((l,) + (1,) * theta.dim())
        P[l, :l] = torch.sqrt((4.0 * l * l - 1) / (l * l - m * m)) * x * P[l - 1, :l]
        if l > 1:
            P[l, :l - 1] -= torch.sqrt((2 * l + 1) * ((l - 1) ** 2 - m[:-1] ** 2) / ((2 * l - 3) * (l * l - m[:-1] ** 2))) * P[l - 2, :l - 1]
    return P


def _modes(l_max):
    """(l, m, sine?) of the real harmonics."""
    return [(l, m, s) for l in range(l_max + 1) for m in range(l + 1) for s in ((0, 1) if m else (0,))]


def _weights(spec, te, pe):
    """Share of each cell that counts for its own patch: 1 - f / 2, f the part of its solid angle inside the other patch.
    At fixed phi the other patch's domain is |sin(theta) sin(phi)| <= c and not (cos(phi) > 0 and |cot(theta)| < t cos(phi)),
    that is |cos(theta)| >= h(phi); the area above h is integrated in phi between the kinks."""
    if spec.polar:
        return torch.ones((spec.n_theta, spec.n_phi), dtype=torch.float64, device="cuda")
    c, t = math.cos(math.pi / 4 - spec.delta_theta), math.tan(math.pi / 4 - spec.delta_phi)
    nt, npp = spec.n_theta, spec.n_phi
    lo, hi = pe[:-1].expand(nt, npp), pe[1:].expand(nt, npp)
    kinks = [lo, hi]

    def add(v, sine):
        v = torch.as_tensor(v, dtype=torch.float64, device=pe.device).expand(nt, npp)
        a = torch.asin(v.clamp(-1, 1)) if sine else torch.acos(v.clamp(-1, 1))
        kinks.extend((a, -a, math.pi - a, a - math.pi) if sine else (a, -a))

    add(c, True)
    add(0.0, False)
    for e in (te[:-1, None], te[1:, None]):
        add(c / torch.sin(e), True)
        add(torch.cos(e) / torch.sin(e) / t, False)
        add(-torch.cos(e) / torch.sin(e) / t, False)
    add(math.sqrt((1 - c * c) / (1 + c * c * t * t)), False)
    k = torch.sort(torch.stack([torch.minimum(torch.maximum(v, lo), hi) for v in kinks], -1), -1).values
    x, g = (torch.from_numpy(v).to(pe.device) for v in np.polynomial.legendre.leggauss(24))
    # phi = mid + half sin(pi u / 2): smooth through square-root ends
    u, du = torch.sin(0.5 * math.pi * x), g * 0.5 * math.pi * torch.cos(0.5 * math.pi * x)
    area = torch.zeros((nt, npp), dtype=torch.float64, device=pe.device)
    top, bot = torch.cos(te[:-1, None, None]), torch.cos(te[1:, None, None])
    for i in range(k.shape[-1] - 1):
        half = 0.5 * (k[..., i + 1] - k[..., i])
        ph = (0.5 * (k[..., i + 1] + k[..., i]))[..., None] + half[..., None] * u
        sp, cp = torch.sin(ph).abs(), torch.cos(ph)
        h = torch.sqrt(((sp - c) * (sp + c)).clamp(min=0)) / sp.clamp(min=c)
        b = t * cp.clamp(min=0)
        h = torch.maximum(h, b / torch.sqrt(1 + b * b))
        inside = (top - torch.maximum(h, bot)).clamp(min=0) + (torch.minimum(-h, top) - bot).clamp(min=0)
        inside = torch.where(h <= 0, top - bot, inside)
        area += half * (inside * du).sum(-1)
    return 1.0 - 0.5 * area / ((torch.cos(te[:-1]) - torch.cos(te[1:]))[:, None] * (pe[1:] - pe[:-1]))


def _moments(spec, rho, te, pe, modes, w):
    """sum over the cells of rho w int K P sin(theta) dtheta int {cos, sin}(m phi) dphi, [n_r][modes]."""
    L = spec.lmax
    x, g = (torch.from_numpy(v).to(te.device) for v in np.polynomial.legendre.leggauss(L + 32))
    half = 0.5 * (te[1:] - te[:-1])[:, None]
    th = 0.5 * (te[1:] + te[:-1])[:, None] + half * x
    T = (_legendre(L, th) * (half * g * torch.sin(th))).sum(-1)                             # [l][m][j]
    m = torch.arange(1, L + 1, dtype=torch.float64, device=te.device)[:, None]
    C = torch.cat([(pe[1:] - pe[:-1])[None], (torch.sin(m * pe[1:]) - torch.sin(m * pe[:-1])) / m])
    S = torch.cat([torch.zeros_like(pe[1:])[None], (torch.cos(m * pe[:-1]) - torch.cos(m * pe[1:])) / m])
    rho = rho * w
    F = (rho @ C.T, rho @ S.T)                                                              # [i][j][m]
    return torch.stack([F[s][:, :, k] @ T[l, k] for l, k, s in modes], 1)


def _radial(spec, A, modes):
    """Coefficients of each harmonic in Phi / (-G) and its radial derivative at the outer edges, from the moments A."""
    r = torch.from_numpy(spec.r_edges).to(A.device)
    rm, rp = r[:-1], r[1:]
    i = torch.arange(spec.n_r, device=A.device)
    inner, outer = i[None, :] <= i[:, None], i[None, :] > i[:, None]
    U, D = torch.empty_like(A), torch.empty_like(A)
    deg = torch.tensor([l for l, _, _ in modes], device=A.device)
    for l in range(spec.lmax + 1):
        at = deg == l
        q = (rp[None, :] / rp[:, None]) ** (l + 1) * (rp ** 2 * (1 - (rm / rp) ** (l + 3)) / (l + 3))[None, :]
        c = torch.where(inner, q, 0.0) @ A[:, at]
        if l < 2:
            shell = rm ** l * (rp ** (2 - l) - rm ** (2 - l)) / (2 - l)
        else:
            shell = rm ** 2 * (torch.log(rp / rm) if l == 2 else (1 - (rm / rp) ** (l - 2)) / (l - 2))
        p = (rp[:, None] / rm[None, :]) ** l * shell[None, :]
        d = torch.where(outer, p, 0.0) @ A[:, at]
        k = 4.0 * math.pi / (2 * l + 1)
        U[:, at], D[:, at] = k * (c + d), k * (l * d - (l + 1) * c) / rp[:, None]
    return U, D


def _evaluate(spec, U, D, modes, theta, phi, gradient):
    """-Phi / G at the angles, and -grad Phi / G there in the frame's Cartesian components."""
    L = spec.lmax
    P = _legendre(L + 1, theta)
    m = torch.arange(L + 2, dtype=torch.float64, device=theta.device)[:, None]
    cs = (torch.cos(m * phi), torch.sin(m * phi))
    l_of, m_of = (torch.tensor([q[k] for q in modes], device=theta.device) for k in (0, 1))
    sine = torch.tensor([q[2] for q in modes], device=theta.device)[:, None] == 1
    own = torch.where(sine, cs[1][m_of], cs[0][m_of])
    Pm = P[l_of, m_of]
    out = [U @ (Pm * own)]
    if not gradient:
        return out[0], None
    # d/dtheta by the neighbours in m, and m / sin(theta) by those of degree l + 1 (both finite at the poles)
    lf, mf = l_of.double(), m_of.double()
    two = lambda k: torch.where(k == 0, 2.0, 1.0).double()  # noqa: E731  (a harmonic of m = 0 carries 1 where the others carry sqrt 2)
    up = P[l_of, m_of + 1] * torch.sqrt((lf - mf) * (lf + mf + 1))[:, None]
    down = torch.where((m_of > 0)[:, None], P[l_of, (m_of - 1).clamp(min=0)], 0.0)
    down = down * torch.sqrt((lf + mf) * (lf - mf + 1) * two((m_of - 1).clamp(min=0)))[:, None]
    dP = torch.where((m_of == 0)[:, None], up * 0.5 ** 0.5, 0.5 * (up - down))
    k = torch.sqrt((2 * lf + 1) / (2 * lf + 3))[:, None]
    a = P[l_of + 1, m_of + 1] * torch.sqrt((lf + mf + 1) * (lf + mf + 2))[:, None]
    b = P[l_of + 1, (m_of - 1).clamp(min=0)] * torch.sqrt((lf - mf + 1) * (lf - mf + 2) * two((m_of - 1).clamp(min=0)))[:, None]
    mP = torch.where((m_of > 0)[:, None], -0.5 * k * (a + b), 0.0)
    turned = torch.where(sine, cs[0][m_of], -cs[1][m_of])
    r = torch.from_numpy(spec.r_edges[1:]).to(U.device)[:, None]
    g = (D @ (Pm * own), U @ (dP * own) / r, U @ (mP * turned) / r)
    st, ct, sp, cp = torch.sin(theta), torch.cos(theta), torch.sin(phi), torch.cos(phi)
    e = ((st * cp, st * sp, ct), (ct * cp, ct * sp, -st), (-sp, cp, torch.zeros_like(st)))
    return out[0], [sum(g[i] * e[i][x] for i in range(3)) for x in range(3)]


def _solve(spec, rho, gradient):
    te, pe = (torch.from_numpy(v).cuda() for v in inputs.angular_cell_edges(spec))
    modes = _modes(spec.lmax)
    w = _weights(spec, te, pe)
    coef = [_radial(spec, _moments(spec, x, te, pe, modes, w), modes) for x in rho]
    th, ph = torch.meshgrid(0.5 * (te[1:] + te[:-1]), 0.5 * (pe[1:] + pe[:-1]), indexing="ij")
    th, ph = th.reshape(-1), ph.reshape(-1)
    phi = [torch.empty_like(x) for x in rho]
    grad = [torch.empty((3,) + tuple(x.shape), dtype=x.dtype, device=x.device) for x in rho] if gradient else None
    step = max(1, (1 << 25) // len(modes))
    for at in range(0, th.numel(), step):
        t, p = th[at:at + step], ph[at:at + step]
        # the same points in the other patch's frame, (x, y, z) -> (-x, z, y)
        to = torch.acos((torch.sin(t) * torch.sin(p)).clamp(-1, 1))
        po = torch.atan2(torch.cos(t), -torch.sin(t) * torch.cos(p))
        st, ct, sp, cp = torch.sin(t), torch.cos(t), torch.sin(p), torch.cos(p)
        for q in range(len(rho)):
            f, v = _evaluate(spec, *coef[q], modes, t, p, gradient)
            if len(rho) > 1:
                f2, v2 = _evaluate(spec, *coef[1 - q], modes, to, po, gradient)
                f = f + f2
                v = [v[0] - v2[0], v[1] + v2[2], v[2] + v2[1]] if gradient else None
            phi[q].reshape(spec.n_r, -1)[:, at:at + step] = -spec.G * f
            if gradient:
                e = ((st * cp, st * sp, ct), (ct * cp, ct * sp, -st), (-sp, cp, torch.zeros_like(st)))
                for i in range(3):
                    grad[q].reshape(3, spec.n_r, -1)[i, :, at:at + step] = spec.G * sum(v[x] * e[i][x] for x in range(3))
    return phi, grad


def exact(case, seed):
    got = [_solve(spec, _densities(spec, kind, eps, seed * 1000 + f), case["gradient"])
           for f, (spec, kind, eps) in enumerate(_fields(case))]
    return {"phi": [p for p, _ in got], "grad": [g for _, g in got] if case["gradient"] else None}
