"""Performance cases of the QBX library: what a user of the framework runs,
through its public entry points.

  listed()             the cases, by use
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  what a program holds before the call: curve, plan, densities
  run(state)           one pass; returns every output whole
  work(case)           bytes and floating-point operations the call cannot do without
  exact(case, seed)    the same outputs from plain torch in 64 bits (no code of the library)

A case is a dict: kind ("apply", "batch", "cfie", "solve", "shape", "field"),
the curve and its M panels, the grid pair (q_tgt, q_src), wavenumber
kre + i kim, order p, side and limit, operators, right-hand sides.
"""
import math

import numpy as np
import torch

import paper_1207_4461_gb300 as qbx

_SIDE = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}
_LIMIT = {"lim": qbx.LIMIT_ONE_SIDED, "pv": qbx.LIMIT_PV}
_OP = {"S": qbx.OP_S, "D": qbx.OP_D, "G": qbx.OP_GRAD_S, "R": qbx.OP_R, "H": qbx.OP_GRAD_D}


def _case(name, kind, curve, M, k, p, **kw):
    c = {"kind": kind, "curve": curve, "M": M, "levels": 0, "kre": float(complex(k).real), "kim": float(complex(k).imag),
         "p": p, "q_tgt": 16, "q_src": 64, "side": "two", "limit": "pv", "ops": "S", "nrhs": 1, "eta": 0.0}
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one curve of moderate size inside another program's loop: the latency of a call
        _case("apply_small", "apply", "starfish", 32, 5.0, 8, side="int", ops="SD"),
        # all layer potentials of a well-resolved curve in one pass (the benchmark workload)
        _case("apply_large", "apply", "starfish", 256, 20.0, 12, side="two", ops="SDG"),
        # one operator, several densities, one-sided, an odd panel count and grid pair
        _case("apply_ragged", "apply", "fourier", 93, 11.0, 10, side="ext", ops="D", nrhs=3, q_tgt=12, q_src=40),
        # lossy medium
        _case("apply_lossy", "apply", "starfish", 128, 20 + 1j, 12, side="two", ops="SDG"),
        # direct evaluation of distant pairs at the caller's request (near-only QBX)
        _case("apply_near_only", "apply", "starfish", 256, 20.0, 12, side="two", ops="SDG", eta=8.0),
        # the hypersingular operator grad D of a Neumann problem
        _case("hypersingular", "apply", "ellipse", 128, 10.0, 10, side="two", ops="H"),
        # many curves of uneven size, 32 densities each, one persistent launch
        _case("batch", "batch", "fourier", 256, 40.0, 10, side="int", limit="lim", ops="SD", nrhs=32, curves=12),
        # the matrix-free solver's matvec for 64 incident waves, corner-refined mesh
        _case("matvec_64", "cfie", "teardrop", 256, 30.0, 14, levels=8, nrhs=64),
        # assembled scattering solve, whole: matrix, GMRES to 1e-10, 16 incident waves
        _case("scatter_solve", "solve", "teardrop", 72, 12.0, 10, levels=5, nrhs=16),
        # one shape-optimisation step of S: geometry, value, gradients of density and curve samples
        _case("shape_step", "shape", "starfish", 128, 10.0, 10, side="int", ops="S"),
        # the same of D on a smaller curve
        _case("shape_step_d", "shape", "fourier", 63, 6.0, 8, side="ext", limit="pv", ops="D"),
        # the field around a solved density: distant points by the smooth rule, close ones by expansions
        _case("field", "field", "starfish", 128, 16.0, 10, side="ext", ops="D", points=12000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["batch", "cfie", "solve", "shape", "shape", "field"])
    k = round(math.exp(rng.uniform(0.0, math.log(40.0))), 3)
    curve = rng.choice(["starfish", "fourier", "ellipse"])
    p = rng.randint(6, 14)
    if kind == "apply":
        M = _log_int(rng, 16, 256)
        q = rng.choice([(16, 64), (16, 64), (12, 40), (8, 32), (16, 48)])
        kw = {"side": rng.choice(["int", "ext", "two"]), "limit": rng.choice(["lim", "pv"]), "q_tgt": q[0], "q_src": q[1],
              "ops": rng.choice(["S", "D", "G", "SD", "SDG", "SDG", "DG", "R", "H"]), "nrhs": rng.choice([1, 1, 1, 2, 3, 5])}
        kim = 0.0
        if rng.random() < 0.25:
            kim = round(rng.uniform(0.02, 0.1) * k, 4)
            M = min(M, 128)
        if kw["ops"] == "H":
            M = min(M, 128)
        if kw["nrhs"] > 1:
            M = min(M, 160)
        if not {"R", "H"} & set(kw["ops"]) and rng.random() < 0.15:
            kw["eta"] = round(rng.uniform(4.0, 12.0), 2)
        return _case(None, "apply", curve, M, k + 1j * kim, p, **kw)
    if kind == "batch":
        return _case(None, "batch", "fourier", _log_int(rng, 48, 224), k, rng.randint(6, 10), side=rng.choice(["int", "ext"]), limit="lim",
                     ops=rng.choice(["S", "D", "SD"]), nrhs=rng.choice([4, 12, 16, 32]), curves=rng.randint(5, 11))
    if kind == "cfie":
        return _case(None, "cfie", "teardrop", _log_int(rng, 48, 224), k, p, levels=rng.randint(2, 8), nrhs=rng.choice([1, 5, 16, 33, 64]))
    if kind == "solve":
        return _case(None, "solve", "teardrop", rng.randint(40, 80), min(k, 16.0), rng.randint(8, 12), levels=rng.randint(2, 6),
                     nrhs=rng.choice([1, 4, 9, 16]))
    if kind == "shape":
        return _case(None, "shape", curve, _log_int(rng, 24, 120), min(k, 16.0), rng.randint(6, 10), side=rng.choice(["int", "ext"]),
                     limit=rng.choice(["lim", "pv"]), ops=rng.choice(["S", "D"]))
    return _case(None, "field", curve, _log_int(rng, 24, 128), k, rng.randint(6, 12), side=rng.choice(["int", "ext"]), ops=rng.choice(["S", "D"]),
                 points=_log_int(rng, 500, 12000))


# ----------------------------------------------------------------------------
# Curves: t -> (gamma, gamma'), panel edges
# ----------------------------------------------------------------------------
def _polar(t, r, dr):
    c, s = np.cos(t), np.sin(t)
    return np.stack([r * c, r * s], -1), np.stack([dr * c - r * s, dr * s + r * c], -1)


def _curve(case, rng):
    kind = case["curve"]
    if kind == "starfish":
        return lambda t: _polar(t, 1.0 + 0.25 * np.cos(5 * t), -1.25 * np.sin(5 * t))
    if kind == "ellipse":
        return lambda t: (np.stack([np.cos(t), 0.5 * np.sin(t)], -1), np.stack([-np.sin(t), 0.5 * np.cos(t)], -1))
    if kind == "fourier":
        a, b = rng.uniform(-0.04, 0.04, 8), rng.uniform(-0.04, 0.04, 8)
        m = np.arange(1, 9.0)
        return lambda t: _polar(t, 1.0 + np.cos(np.outer(t, m)) @ a + np.sin(np.outer(t, m)) @ b,
                                -np.sin(np.outer(t, m)) @ (m * a) + np.cos(np.outer(t, m)) @ (m * b))
    pi = math.pi

    def teardrop(t):   # corner at t = 0 = 2 pi
        u = t / (2 * pi)
        x, y = 1.7 * (np.sin(pi * u) - 0.5), 0.85 * np.cos(pi * u) * (pi * u - pi) * pi * u
        dx = 1.7 * pi * np.cos(pi * u)
        dy = 0.85 * (-pi * np.sin(pi * u) * (pi * u - pi) * pi * u + np.cos(pi * u) * pi * (2 * pi * u - pi))
        return np.stack([x, y], -1), np.stack([dx, dy], -1) / (2 * pi)
    return teardrop


def _edges(M, levels):
    """M panels equal in t, of which 2 levels come from bisecting the two next to t = 0 = 2 pi."""
    e = np.linspace(0.0, 2 * math.pi, M - 2 * levels + 1)
    if levels == 0:
        return e
    h = e[1]
    left = [h / 2 ** j for j in range(levels, 0, -1)]
    return np.concatenate([[0.0], left, e[1:-1], [2 * math.pi - v for v in reversed(left)], [2 * math.pi]])


def _dens(n, nrhs, seed, dev="cuda"):
    """Seeded CN(0, 1) densities."""
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return torch.randn(n, nrhs, dtype=torch.complex128, device=dev, generator=g)


def _waves(x, y, k, nrhs):
    """Incident plane waves from nrhs directions, -u_inc on the curve."""
    th = torch.arange(nrhs, dtype=torch.float64, device=x.device) * (2 * math.pi / nrhs) + 0.3
    ph = k.real * (x[:, None] * torch.cos(th) + y[:, None] * torch.sin(th))
    return -torch.polar(torch.ones_like(ph), ph)


def _sizes(case, seed):
    """Panel counts (16..M, uneven, by the case alone) and wavenumbers (1..kre) of a batch's curves."""
    n = case["curves"]
    M = np.round(np.linspace(min(16, case["M"]), case["M"], n)).astype(int)
    M = np.random.default_rng(case["M"]).permutation(np.maximum(M - (np.arange(n) * 7) % 4, 1))
    ks = np.random.default_rng(seed + 71).uniform(1.0, max(case["kre"], 1.5), n)
    return [int(m) for m in M], [float(v) for v in ks]


def _k(case):
    return complex(case["kre"], case["kim"]) if case["kim"] else case["kre"]


def _ncomp(ops):
    return sum(2 if o in "GH" else 1 for o in ops)


# ----------------------------------------------------------------------------
# prepare / run
# ----------------------------------------------------------------------------
def prepare(case, seed):
    rng = np.random.default_rng(seed)
    M, qt, qs, p, nrhs = case["M"], case["q_tgt"], case["q_src"], case["p"], case["nrhs"]
    kind = case["kind"]
    s = {"case": case, "k": _k(case), "side": _SIDE[case["side"]], "limit": _LIMIT[case["limit"]]}
    if kind == "batch":
        Ms, ks = _sizes(case, seed)
        plan = qbx.Plan(qt, qs, n_src=qs * max(Ms), n_ctr=qt * max(Ms), ncoef=2, nrhs=nrhs)
        geoms = [qbx.qbx_geometry(plan, _curve(case, rng), _edges(m, 0)) for m in Ms]
        dens = [_dens(g.n_tgt, nrhs, seed + 1009 * i) for i, g in enumerate(geoms)]
        s.update(plan=plan, batch=qbx.Batch(plan, geoms, ks, p, [_OP[o] for o in case["ops"]], s["side"], s["limit"], dens))
        return s
    cur, edges = _curve(case, rng), _edges(M, case["levels"])
    need = qbx.qbx_workspace_bytes(M * qs, 2 * M * qt, 4, nrhs)
    if kind == "shape":
        need = max(need, qbx.qbx_shape_adjoint_workspace_bytes(M, qt, qs, p, nrhs))
    if kind == "field":
        need = max(qbx.qbx_workspace_bytes(M * qs, 2 * M * qt, 2 * p + 1, nrhs), qbx.qbx_workspace_bytes(M * qs, case["points"], 2, nrhs))
    plan = qbx.Plan(qt, qs, workspace_bytes=need)
    s.update(plan=plan)
    if kind == "shape":
        up = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
        t_t, t_s = qbx.panel_nodes(edges, qt), qbx.panel_nodes(edges, qs)
        s.update(edges=edges, samples=[up(a).requires_grad_() for a in (*cur(t_t), *cur(t_s))],
                 dens=_dens(M * qt, nrhs, seed).requires_grad_(), goal=_dens(M * qt, nrhs, seed + 5))
        return s
    g = qbx.qbx_geometry(plan, cur, edges)
    s.update(g=g)
    if kind == "solve":
        s["dens"] = _waves(g["tgt_x"], g["tgt_y"], complex(s["k"]), nrhs) + 0.05 * _dens(g.n_tgt, nrhs, seed)
        return s
    s["dens"] = _dens(g.n_tgt, nrhs, seed)
    if kind == "field":
        far, near = _points(case, seed, {n: g[n] for n in ("ctr_x", "ctr_y", "ctr_r")}, g.n_tgt)
        s.update(far=far, near=near)
    return s


def _points(case, seed, g, n):
    """A ring of distant points and points inside expansion disks of the side."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 17)
    m = case["points"]
    u = torch.rand(m, 2, dtype=torch.float64, device="cuda", generator=gen)
    rad = (1.7 + 1.3 * u[:, 0]) if case["side"] == "ext" else 0.25 * u[:, 0]
    th = 2 * math.pi * u[:, 1]
    far = torch.stack([rad * torch.cos(th), rad * torch.sin(th)], 1)
    v = torch.rand(n, 2, dtype=torch.float64, device="cuda", generator=gen)
    o = n if case["side"] == "ext" else 0
    rr, th = 0.8 * g["ctr_r"][o:o + n] * v[:, 0], 2 * math.pi * v[:, 1]
    near = torch.stack([g["ctr_x"][o:o + n] + rr * torch.cos(th), g["ctr_y"][o:o + n] + rr * torch.sin(th)], 1)
    return far, near


def run(s):
    c, plan, k, p = s["case"], s["plan"], s["k"], s["case"]["p"]
    kind, ops = c["kind"], c["ops"]
    if kind == "batch":
        return [[o[j] for j in sorted(o)] for o in s["batch"].apply()]
    if kind == "shape":
        x, d = s["samples"], s["dens"]
        if ops == "S":
            u = qbx.apply_s_shape_autograd(plan, s["edges"], *x, d, s["side"], k, p)
        else:
            u = qbx.apply_d_shape_autograd(plan, s["edges"], *x, d, s["side"], s["limit"], k, p)
        loss = (u - s["goal"]).abs().square().sum()
        return [loss.detach(), u.detach(), *torch.autograd.grad(loss, [d, *x])]
    g = s["g"]
    if kind == "apply":
        if ops in "RH" or (len(ops) == 1 and not c["eta"]):
            return [qbx.qbx_apply(plan, g, _OP[ops], s["side"], s["limit"], k, p, s["dens"])]
        out = qbx.qbx_apply_ops(plan, g, [_OP[o] for o in ops], s["side"], s["limit"], k, p, s["dens"], eta=c["eta"] or None)
        return [out[_OP[o]] for o in ops]
    if kind == "cfie":
        return [qbx.qbx_apply_cfie(plan, g, k, k, p, s["dens"])]
    if kind == "solve":
        A = qbx.qbx_assemble_cfie(plan, g, k, k, p)
        mu, iters, _ = qbx.qbx_solve_exterior_dirichlet(plan, g, k, k, p, s["dens"], tol=1e-10, restart=60, maxiter=240, A=A)
        return [A, mu, iters]
    wd = qbx.qbx_upsample(plan, g, s["dens"])
    far = qbx.qbx_far(plan, g, _OP[ops], k, wd, s["far"])
    at = qbx.qbx_assign_centres(plan, g, s["side"], s["near"])
    alpha = qbx.qbx_form_locals(plan, g, _OP[ops], s["side"], k, p, wd)
    x, y = s["near"][:, 0].contiguous(), s["near"][:, 1].contiguous()
    return [far, at, qbx.qbx_eval_locals(plan, g, s["side"], k, p, alpha, ex=x, ey=y, ectr=at)]


def work(case):
    """Each input read and each output written once; one complex multiply-add
    (8 operations) per target, source, component and right-hand side: the
    discrete operator applied once, its entries taken as given."""
    M, qt, qs, nrhs = case["M"], case["q_tgt"], case["q_src"], case["nrhs"]
    kind = case["kind"]
    if kind == "batch":
        Ms = _sizes(case, 0)[0]
        n, pairs = sum(Ms), float(qt * qs * sum(m * m for m in Ms))
    else:
        n, pairs = M, float(M * qt) * (M * qs)
    comp = _ncomp(case["ops"])
    geo = n * (qt * 5 + qs * 5) * 8.0
    io = n * qt * nrhs * 16.0 * (1 + comp)
    flops = 8.0 * pairs * comp * nrhs
    if kind == "solve":   # matrix out, then one product (the least a solve can do)
        io += 16.0 * (M * qt) ** 2
        flops = 8.0 * pairs + 8.0 * (M * qt) ** 2 * nrhs
    if kind == "shape":   # value, transposed value, gradients of sources and centres
        io += n * (qt + qs) * 4 * 8.0
        flops = 8.0 * pairs * 6
    if kind == "field":
        io += case["points"] * 32.0
        flops = 8.0 * (case["points"] * M * qs + pairs)
    return {"bytes": geo + io, "flops": flops}


# ----------------------------------------------------------------------------
# exact: the same quantities in plain torch, 64 bits
# ----------------------------------------------------------------------------
class _Hankel(torch.autograd.Function):
    """H0(k rho), H1(k rho) for real k > 0 as complex tensors, differentiable
    in rho (torch.special.bessel_* on the GPU is good to 1e-7 only)."""

    @staticmethod
    def forward(ctx, rho, k):
        z = k * rho
        h0, h1 = _hankel_complex(torch.complex(z, torch.zeros_like(z)))
        ctx.save_for_backward(z, h0, h1)
        ctx.k = k
        return h0, h1

    @staticmethod
    def backward(ctx, g0, g1):
        z, h0, h1 = ctx.saved_tensors
        d = (g0.conj() * (-h1)).real + (g1.conj() * (h0 - h1 / z)).real
        return ctx.k * d, None


def _hankel_complex(z):
    """H0, H1 at complex z, Im z > 0: the ascending series for |z| < 3, above
    it H_n(z) = (2/(pi z))^(1/2) e^(i(z - n pi/2 - pi/4)) / Gamma(n + 1/2)
    int_0^inf e^-t t^(n-1/2) (1 + i t/(2z))^(n-1/2) dt (DLMF 10.9.11 family)
    with t = u^2 by the trapezoidal rule."""
    small = z.abs() < 3.0
    zs = torch.where(small, z, torch.ones_like(z))
    t = -0.25 * zs * zs
    j0, y0, j1, y1 = (torch.zeros_like(z) for _ in range(4))
    term, psi, psi2 = torch.ones_like(z), -0.57721566490153286061, 1.0 - 0.57721566490153286061
    for m in range(26):
        if m:
            term = term * t / (m * m)
            psi += 1.0 / m
            psi2 += 1.0 / (m + 1)
        j0, y0 = j0 + term, y0 + psi * term
        j1, y1 = j1 + term / (m + 1), y1 + (psi + psi2) * term / (m + 1)
    L = torch.log(0.5 * zs)
    j1 = 0.5 * zs * j1
    h0 = j0 + 1j * (2 / math.pi) * (L * j0 - y0)
    h1 = j1 + 1j * (2 / math.pi * L * j1 - 2 / math.pi / zs - zs / (2 * math.pi) * y1)
    zl = torch.where(small, torch.full_like(z, 3.0), z)
    s0, s1 = torch.zeros_like(z), torch.zeros_like(z)
    h = 0.22
    for i in range(0, 30):
        u2 = (i * h) ** 2
        w = 2.0 * h * math.exp(-u2) * (0.5 if i == 0 else 1.0)
        q = torch.sqrt(1.0 + 1j * u2 / (2.0 * zl))
        s0 = s0 + w / q
        if i:
            s1 = s1 + w * u2 * q
    pre = torch.sqrt(2.0 / (math.pi * zl)) * torch.exp(1j * (zl - math.pi / 4)) / math.sqrt(math.pi)
    return torch.where(small, h0, pre * s0), torch.where(small, h1, -2j * pre * s1)


def _bessel_cols(z, n):
    """J_0..J_n at z (vector) by backward recurrence, normalised by J_0 + 2 sum J_2k = 1."""
    top = 2 * ((n + 30 + int(1.2 * float(z.detach().abs().max()))) // 2)
    f1, f = torch.zeros_like(z), torch.full_like(z, 1e-60)
    norm, cols = 2 * f, []
    for m in range(top, 0, -1):
        f1, f = f, (2.0 * m / z) * f - f1
        big = f.detach().abs() > 1e100
        sc = torch.where(big, 1e-100, torch.ones_like(f.detach().abs()))
        f, f1, norm, cols = f * sc, f1 * sc, norm * sc, [v * sc for v in cols]
        if m - 1 <= n:
            cols.append(f)
        if (m - 1) % 2 == 0:
            norm = norm + (f if m == 1 else 2 * f)
    return [v / norm for v in reversed(cols)]


def _gl(q):
    return np.polynomial.legendre.leggauss(q)


def _interp(qt, qs):
    xt, wt = _gl(qt)
    vt = np.polynomial.legendre.legvander(xt, qt - 1)
    proj = (np.arange(qt) + 0.5)[:, None] * (vt * wt[:, None]).T
    return np.polynomial.legendre.legvander(_gl(qs)[0], qt - 1) @ proj


def _geometry(case, cur, edges, dev, samples=None):
    """Nodes, normals, weights, centres; differentiable in the curve samples."""
    qt, qs = case["q_tgt"], case["q_src"]
    mid, half = 0.5 * (edges[1:] + edges[:-1]), 0.5 * (edges[1:] - edges[:-1])
    nodes = lambda q: (mid[:, None] + half[:, None] * _gl(q)[0]).reshape(-1)
    up = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    if samples is None:
        samples = [up(a) for a in (*cur(nodes(qt)), *cur(nodes(qs)))]
    gt, dgt, gs, dgs = samples
    nrm = lambda d: torch.stack([d[:, 1], -d[:, 0]], 1) / torch.linalg.vector_norm(d, dim=1, keepdim=True)
    wgt = lambda d, q: torch.linalg.vector_norm(d, dim=1) * up(np.outer(half, _gl(q)[1]).reshape(-1))
    g = {"xt": gt, "nt": nrm(dgt), "wt": wgt(dgt, qt), "xs": gs, "ns": nrm(dgs), "ws": wgt(dgs, qs)}
    g["h"] = g["ws"].reshape(-1, qs).sum(1)
    r = 0.5 * g["h"].repeat_interleave(qt)
    g["r"] = torch.cat([r, r])
    g["c"] = torch.cat([gt - r[:, None] * g["nt"], gt + r[:, None] * g["nt"]])
    g["P"] = up(_interp(qt, qs))
    return g


def _cplx(v):
    return torch.complex(v[:, 0], v[:, 1])


def _kernels(case, g, c, x, what, eta=0.0):
    """Truncated Graf kernels (with i/4) of centres c and targets x against
    every source: {name: [n_c, n_s]} for the names in what (S D R G H)."""
    k, p = _k(case), case["p"]
    xs = g["xs"]
    d = xs[None, :, :] - c[:, None, :]
    rho = torch.sqrt(d[..., 0] ** 2 + d[..., 1] ** 2)
    z = k * rho
    h0, h1 = _Hankel.apply(rho, k) if not case["kim"] else _hankel_complex(z)
    em = torch.complex(d[..., 0] / rho, -d[..., 1] / rho)   # e^{-i theta_s}
    far = None
    if eta:
        xc = x - c
        far = rho.detach() >= eta * torch.sqrt(xc[:, 0] ** 2 + xc[:, 1] ** 2)[:, None]
        h0, h1 = h0.masked_fill(far, 0.0), h1.masked_fill(far, 0.0)
    H = [h0, h1]
    for l in range(1, p + 1):
        H.append((2.0 * l / z) * H[l] - H[l - 1])
    ph, cols = torch.ones_like(em), {0: h0}
    for l in range(1, p + 2):
        ph = ph * em
        cols[l] = H[l] * ph
        cols[-l] = (-1) ** l * H[l] * ph.conj()
    E = torch.stack([cols[l] for l in range(-p - 1, p + 2)], 1)   # [C, 2p+3, S]
    dx = x - c
    rx = torch.sqrt(dx[:, 0] ** 2 + dx[:, 1] ** 2)
    J = _bessel_cols(k * rx, p + 1)
    ep = torch.complex(dx[:, 0] / rx, dx[:, 1] / rx)
    pw, J = [torch.ones_like(ep)], [j.to(torch.complex128) for j in J]
    for l in range(1, p + 2):
        pw.append(pw[-1] * ep)
    cl = {l: J[l] * pw[l] if l >= 0 else (-1) ** (-l) * J[-l] * pw[-l].conj() for l in range(-p - 1, p + 2)}

    def weights(shift_t, shift_s):   # sum over |l| <= p of c_{l+shift_t} E_{l+shift_s}
        zero = torch.zeros_like(pw[0])
        return torch.stack([cl[m - shift_s + shift_t] if abs(m - shift_s) <= p else zero for m in range(-p - 1, p + 2)], 1)

    jobs = []
    add = lambda st, ss: (jobs.append(weights(st, ss)), len(jobs) - 1)[1]
    idx = {}
    for o in what:
        idx[o] = ([add(0, 0)] if o == "S" else [add(0, -1), add(0, 1)] if o in "DR" else [add(-1, 0), add(1, 0)] if o == "G" else
                  [add(-1, -1), add(-1, 1), add(1, -1), add(1, 1)])
    R = torch.bmm(torch.stack(jobs, 1), E)
    nu = {"D": _cplx(g["ns"]), "H": _cplx(g["ns"]), "R": 1j * _cplx(g["ns"])}
    out = {}
    for o in what:
        r = [R[:, i] for i in idx[o]]
        if o == "S":
            out[o] = 0.25j * r[0]
        elif o in "DR":
            out[o] = 0.125j * k * (nu[o].conj() * r[0] - nu[o] * r[1])
        else:
            if o == "G":
                a, b = k * r[0], -k * r[1]                       # (dx - i dy), (dx + i dy)
            else:
                a = 0.5 * k * k * (nu[o].conj() * r[0] - nu[o] * r[1])
                b = -0.5 * k * k * (nu[o].conj() * r[2] - nu[o] * r[3])
            out[o + "x"], out[o + "y"] = 0.125j * (a + b), 0.125j * 1j * (a - b)
    if eta:
        for n, v in _smooth(case, g, x, what).items():
            out[n] = out[n] + torch.where(far, v, torch.zeros_like(v))
    return out


def _smooth(case, g, x, what):
    """Kernels of the plain rule at points x."""
    k = _k(case)
    d = x[:, None, :] - g["xs"][None, :, :]
    rho = torch.sqrt(d[..., 0] ** 2 + d[..., 1] ** 2)
    h0, h1 = _Hankel.apply(rho, k) if not case["kim"] else _hankel_complex(k * rho)
    out = {}
    if "S" in what:
        out["S"] = 0.25j * h0
    if "D" in what:
        out["D"] = 0.25j * k * h1 * ((d * g["ns"]).sum(-1) / rho)
    if "G" in what:
        out["Gx"], out["Gy"] = (-0.25j * k * h1 * (d[..., i] / rho) for i in (0, 1))
    return out


def _upsample(case, g, dens):
    u = torch.einsum("ji,mir->mjr", g["P"].to(torch.complex128), dens.reshape(case["M"], case["q_tgt"], -1))
    return u.reshape(-1, dens.shape[1]) * g["ws"][:, None]


def _jumps(case, g, name, val, sg, dens):
    """Principal value from the one-sided limit (sg = +1 exterior)."""
    if name == "D":
        return val - 0.5 * sg * dens
    if name in ("Gx", "Gy"):
        return val + 0.5 * sg * dens * g["nt"][:, 0 if name == "Gx" else 1, None]
    if name in ("Hx", "Hy"):
        q = case["q_tgt"]
        xt, wt = _gl(q)
        vand = np.polynomial.legendre.legvander(xt, q - 1)
        der = np.stack([np.polynomial.legendre.legval(xt, np.polynomial.legendre.legder(np.eye(q)[j])) for j in range(q)], 1)
        Dm = torch.as_tensor(der @ ((np.arange(q) + 0.5)[:, None] * (vand * wt[:, None]).T), device=dens.device)
        dd = torch.einsum("ji,mir->mjr", Dm.to(torch.complex128), dens.reshape(-1, q, dens.shape[1])).reshape(dens.shape)
        dd = dd / (g["wt"].reshape(-1, q) / torch.as_tensor(wt, device=dens.device)).reshape(-1, 1)
        tan = -g["nt"][:, 1] if name == "Hx" else g["nt"][:, 0]
        return val - 0.5 * sg * tan[:, None] * dd
    return val


def _apply(case, g, dens, names_of, chunk):
    """{name: [n_tgt, nrhs]} of the on-surface operators."""
    n = dens.shape[0]
    wd = _upsample(case, g, dens)
    sides = {"int": [0], "ext": [1], "two": [0, 1]}[case["side"]]
    total = {}
    for sd in sides:
        rows = {}
        for a in range(0, n, chunk):
            b = min(n, a + chunk)
            ker = _kernels(case, g, g["c"][sd * n + a:sd * n + b], g["xt"][a:b], names_of, case["eta"])
            for m, v in ker.items():
                rows.setdefault(m, []).append(v @ wd)
        for m, v in rows.items():
            v = torch.cat(v)
            if len(sides) == 1 and case["limit"] == "pv":
                v = _jumps(case, g, m, v, 1.0 if sd else -1.0, dens)
            total[m] = total.get(m, 0.0) + v / len(sides)
    return total


def _outputs(total, ops):
    return [torch.stack([total[o + "x"], total[o + "y"]], 1) if o in "GH" else total[o] for o in ops]


def exact(case, seed):
    dev, kind, ops, k = "cuda", case["kind"], case["ops"], _k(case)
    rng = np.random.default_rng(seed)
    M, qt, nrhs = case["M"], case["q_tgt"], case["nrhs"]
    rows = lambda c: max(16, int(3e6 // (c["M"] * c["q_src"])))
    with torch.no_grad():
        if kind == "batch":
            Ms, ks = _sizes(case, seed)
            outs = []
            for i, (m, kk) in enumerate(zip(Ms, ks)):
                c = dict(case, M=m, kre=kk)
                g = _geometry(c, _curve(case, rng), _edges(m, 0), dev)
                outs.append(_outputs(_apply(c, g, _dens(m * qt, nrhs, seed + 1009 * i), ops, rows(c)), ops))
            return outs
        cur, edges = _curve(case, rng), _edges(M, case["levels"])
        g = _geometry(case, cur, edges, dev)
        n = M * qt
        if kind == "apply":
            return _outputs(_apply(case, g, _dens(n, nrhs, seed), ops, rows(case)), ops)
        if kind == "cfie":
            t = _apply(case, g, _dens(n, nrhs, seed), "SD", rows(case))
            return [t["D"] - 1j * k * t["S"]]
        if kind == "solve":
            A = []
            for a in range(0, n, rows(case)):
                b = min(n, a + rows(case))
                v = 0.0
                for sd in (0, 1):
                    ker = _kernels(case, g, g["c"][sd * n + a:sd * n + b], g["xt"][a:b], "SD")
                    v = v + 0.5 * (ker["D"] - 1j * k * ker["S"])
                v = (v * g["ws"]).reshape(b - a, M, -1)
                A.append(torch.einsum("tmj,ji->tmi", v, g["P"].to(torch.complex128)).reshape(b - a, n))
            A = torch.cat(A) + 0.5 * torch.eye(n, dtype=torch.complex128, device=dev)
            x, y = g["xt"][:, 0], g["xt"][:, 1]
            f = _waves(x, y, complex(k), nrhs) + 0.05 * _dens(n, nrhs, seed)
            mu = torch.linalg.solve(A, f)
            w = g["wt"].sqrt()
            return [(A * w[:, None] / w[None, :]).T.contiguous(), mu, None]
        if kind == "field":
            wd = _upsample(case, g, _dens(n, nrhs, seed))
            o = n if case["side"] == "ext" else 0
            geo = {"ctr_x": g["c"][:, 0], "ctr_y": g["c"][:, 1], "ctr_r": g["r"]}
            far, near = _points(case, seed, geo, n)
            uf = torch.cat([_smooth(case, g, far[a:a + 500], ops)[ops] @ wd for a in range(0, far.shape[0], 500)])
            ctr, un = g["c"][o:o + n], []
            for a in range(0, n, rows(case)):
                x = near[a:a + rows(case)]
                ratio = torch.cdist(x, ctr, compute_mode="donot_use_mm_for_euclid_dist") / g["r"][o:o + n]
                un.append(_kernels(case, g, ctr[ratio.argmin(1)], x, ops)[ops] @ wd)
            return [uf, None, torch.cat(un)]
    # shape: reverse mode through the whole discretisation, row blocks of the value
    goal = _dens(n, nrhs, seed + 5)
    sam = [t.clone().requires_grad_() for t in _samples(case, cur, edges, dev)]
    dens = _dens(n, nrhs, seed).requires_grad_()
    leaves, u = [dens, *sam], []
    grads = [torch.zeros_like(t) for t in leaves]
    sd = 1 if case["side"] == "ext" else 0
    for a in range(0, n, 128):
        b = min(n, a + 128)
        g = _geometry(case, cur, edges, dev, sam)
        v = _kernels(case, g, g["c"][sd * n + a:sd * n + b], g["xt"][a:b], ops)[ops] @ _upsample(case, g, dens)
        if ops == "D" and case["limit"] == "pv":
            v = v - 0.5 * (1.0 if sd else -1.0) * dens[a:b]
        u.append(v.detach())
        for t, dt in zip(grads, torch.autograd.grad(v, leaves, 2.0 * (v.detach() - goal[a:b]))):
            t += dt
    u = torch.cat(u)
    return [(u - goal).abs().square().sum(), u, *grads]


def _samples(case, cur, edges, dev):
    mid, half = 0.5 * (edges[1:] + edges[:-1]), 0.5 * (edges[1:] - edges[:-1])
    nodes = lambda q: (mid[:, None] + half[:, None] * _gl(q)[0]).reshape(-1)
    return [torch.as_tensor(np.ascontiguousarray(a), device=dev) for a in (*cur(nodes(case["q_tgt"])), *cur(nodes(case["q_src"])))]
