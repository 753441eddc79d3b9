"""Distant sources through cluster moments against the same call pair by pair.

A plan whose workspace holds the partial sums but not the cluster arrays takes
every pair through the pair kernels, so the two routes of one call are compared
on the same inputs: the truncated sums are the same, only their order and the
cut of the clusters' series differ.  Bound: the cut leaves 5e-17 of a kernel
value, and each route rounds 10 to 100 units in the last place over its sums
(measured against 64-bit values: 3e-15 to 2e-14), so 1e-12 of the largest
output; where centres are inadmissible (closest source at less than 0.8 r) the
sums themselves amplify rounding by (r/rho)^p, so those sizes are kept out.
"""
import numpy as np
import pytest
import scipy.special as sp
import torch

import paper_1207_4461_gb300 as qbx
import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12


def pair_plan(g, qt, qs, nrhs, ncomp, nd=1, nsides=2):
    """A plan with room for the densities and two source splits only."""
    al = lambda b: (b + 255) // 256 * 256
    per = nsides * g.n_tgt * ncomp * nrhs * 16
    return qbx.Plan(qt, qs, workspace_bytes=nd * al(g.n_src * nrhs * 16) + 1024 + 2 * per)


def geometry(plan, curve, edges, scale=1.0):
    def scaled(t):
        a, b = curve(t)
        return scale * a, scale * b
    return qbx.qbx_geometry(plan, scaled, edges)


def check(got, ref, what):
    err = float((got - ref).abs().max() / ref.abs().max())
    assert np.isfinite(err) and err < TOL, (what, err)


CASES = [
    # M, q_tgt, q_src, k, p, ops, side, limit, nrhs, eta, scale
    (16, 16, 64, 5.0, 8, (0, 1), "int", 0, 1, None, 1.0),        # fewest panels that form clusters
    (17, 12, 40, 9.0, 10, (1,), "ext", 1, 3, None, 1.0),          # odd panel count, blocks across panels
    (33, 5, 21, 7.0, 6, (0, 1, 2), "two", 0, 1, None, 1.0),       # odd source count: whole-panel leaves
    (24, 16, 16, 6.0, 4, (2,), "two", 0, 2, None, 1.0),           # too few sources to halve a panel
    (29, 9, 128, 11.0, 9, (0, 2), "int", 1, 1, None, 1.0),        # most sources per panel
    (40, 16, 64, 8.0, 0, (0, 1, 2), "two", 0, 1, None, 1.0),      # orders at the bottom
    (40, 16, 64, 8.0, 1, (0, 1, 2), "ext", 1, 2, None, 1.0),
    (36, 16, 64, 6.0, 40, (0, 1, 2), "int", 0, 1, None, 1.0),     # and at the top
    (36, 16, 64, 3 + 0.4j, 30, (0, 1), "two", 0, 2, None, 1.0),
    (64, 16, 64, 20 + 1j, 12, (0, 1, 2), "two", 0, 1, None, 1.0),
    (48, 16, 64, 2 + 6j, 9, (1, 2), "ext", 1, 1, None, 1.0),      # strongly damped
    (48, 16, 64, 90.0, 12, (0, 1), "int", 0, 1, None, 1.0),       # k r above 5: no cluster is cut short
    (64, 16, 64, 250.0, 10, (0,), "two", 0, 1, None, 1.0),
    (40, 16, 64, 1e-3, 8, (0, 1, 2), "two", 0, 1, None, 1.0),     # Laplace-like
    (40, 16, 64, 5.0, 12, (0, 1), "two", 0, 1, None, 1e-4),       # a tiny curve
    (96, 16, 64, 14.0, 12, (0, 1, 2), "two", 0, 5, None, 1.0),
    (64, 16, 64, 12.0, 10, (0, 1, 2), "two", 0, 1, 6.0, 1.0),     # near-only: smooth rule beyond 6 r
    (64, 16, 64, 9 + 0.5j, 8, (0, 1), "int", 1, 3, 12.0, 1.0),
    (64, 16, 64, 9.0, 8, (2,), "ext", 1, 1, 1.5, 1.0),
]


@pytest.mark.parametrize("case", CASES)
def test_clusters_match_pairs(cuda, case):
    M, qt, qs, k, p, ops, side, limit, nrhs, eta, scale = case
    side = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}[side]
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=4, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M), scale)
    d = torch.as_tensor(W.complex_gaussian(M + p, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    got = qbx.qbx_apply_ops(plan, g, ops, side, limit, k / scale, p, d, eta=eta)
    qbx.qbx_sync_status(plan)
    pp = pair_plan(g, qt, qs, nrhs, sum(2 if o == 2 else 1 for o in ops))
    ref = qbx.qbx_apply_ops(pp, g, ops, side, limit, k / scale, p, d, eta=eta)
    for o in ops:
        check(got[o], ref[o], (case, o))


GROUP = [
    # M, q_tgt, q_src, k, p, ops ("cfie": the combined field), side, limit, nrhs, eta
    (16, 16, 64, 5.0, 8, (0,), "int", 0, 16, None),          # fewest panels and columns
    (19, 12, 40, 9.0, 10, (1,), "ext", 1, 17, None),         # blocks across panels, a ragged column group
    (37, 7, 33, 7.0, 6, (0, 1), "two", 0, 33, None),         # both sides averaged per pair, 66 columns: two passes
    (40, 16, 64, 6.0, 12, (0, 1, 2), "two", 0, 16, None),    # with grad S: sides kept apart
    (40, 16, 64, 3 + 0.5j, 9, (0, 1), "two", 0, 20, None),
    (36, 16, 64, 6.0, 40, (0, 1), "two", 0, 16, None),       # highest order
    (33, 16, 64, 8.0, 0, (0, 1), "two", 0, 16, None),        # lowest
    (64, 16, 64, 12.0, 10, (0, 1), "two", 0, 16, 6.0),       # near-only
    (64, 16, 64, 100.0, 10, (1,), "int", 0, 24, None),       # no cluster of more than a panel
    (48, 16, 64, 11.0, 14, "cfie", "two", 0, 1, None),       # one column
    (48, 16, 64, 11.0, 14, "cfie", "two", 0, 65, None),
    (48, 16, 64, 4 + 0.3j, 10, "cfie", "two", 0, 9, None),
]


@pytest.mark.parametrize("case", GROUP)
def test_many_columns_match_pairs(cuda, case):
    M, qt, qs, k, p, ops, side, limit, nrhs, eta = case
    side = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}[side]
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=4, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M + p, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    pp = pair_plan(g, qt, qs, nrhs, 1 if ops == "cfie" else sum(2 if o == 2 else 1 for o in ops))
    run = lambda pl: ([qbx.qbx_apply_cfie(pl, g, k, k - 0.5j, p, d)] if ops == "cfie" else
                      list(qbx.qbx_apply_ops(pl, g, ops, side, limit, k, p, d, eta=eta).values()))
    got = run(plan)
    qbx.qbx_sync_status(plan)
    for i, (a, b) in enumerate(zip(got, run(pp))):
        check(a, b, (case, i))


@pytest.mark.parametrize("case", [
    (64, 16, 64, 5.0, 8, (0,), "int", 0, 16, None),              # fewest leaves with super-blocks
    (131, 16, 64, 9.0, 10, (0, 1), "two", 0, 17, None),          # ragged at every level
    (150, 5, 21, 7.0, 6, (1,), "ext", 1, 16, None),              # several panels per block, whole-panel leaves
    (200, 16, 64, 40.0, 10, (0, 1), "int", 0, 16, None),         # k caps the nodes
    (160, 16, 64, 4 + 0.3j, 9, (0, 1), "ext", 0, 16, None),
    (160, 16, 64, 12.0, 10, (0, 1), "two", 0, 16, 6.0),          # near-only
    (128, 16, 64, 1e-3, 8, (0,), "two", 0, 16, None),
    (210, 16, 64, 11.0, 14, "cfie", "two", 0, 33, None),
    (130, 16, 64, 3 + 3j, 10, "cfie", "two", 0, 4, None)])
def test_super_blocks_match_pairs(cuda, case):
    """Nodes far from many blocks at once; panels of very different sizes too."""
    test_many_columns_match_pairs(cuda, case)
    M, qt, qs, k, p, ops, side, limit, nrhs, eta = case
    if qt != 16 or ops == "cfie" or eta:
        return
    edges = W.dyadic_edges(M, 6)
    cur, M = W.teardrop(), len(edges) - 1
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=4, nrhs=nrhs)
    g = geometry(plan, cur, edges)
    d = torch.as_tensor(W.complex_gaussian(M + p, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    got = qbx.qbx_apply_cfie(plan, g, k, 1.0, p, d)
    check(got, qbx.qbx_apply_cfie(pair_plan(g, qt, qs, nrhs, 1), g, k, 1.0, p, d), case)


@pytest.mark.parametrize("side,limit,ops,eta,ck", [("int", 1, (0, 1), 0.0, False), ("two", 0, (0, 1), 0.0, False),
                                                   ("ext", 0, (1,), 7.0, False), ("two", 0, (0,), 0.0, True)])
def test_batch_clusters_match_single_curves(cuda, side, limit, ops, eta, ck, Ms=(40, 9, 64, 16, 12, 33)):
    """A batch of curves with and without clusters (2 and 9 panels form none)
    against each curve alone, pair by pair; twice, for the kept counter."""
    side = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}[side]
    ks = [5.0, 9.0, 14.0, 3.0, 2.0, 7.0]
    if ck:
        ks = [v * (1 + 0.05j) if i % 2 else v for i, v in enumerate(ks)]
    nrhs, p = 12, 9
    plan = qbx.Plan(16, 64, n_src=64 * max(Ms), n_ctr=32 * max(Ms), ncoef=2, nrhs=nrhs)
    cur = W.starfish(0.15, 3)
    gs = [qbx.qbx_geometry(plan, cur, cur.edges(M)) for M in Ms]
    ds = [torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
          for M, g in zip(Ms, gs)]
    b = qbx.Batch(plan, gs, ks, p, ops, side, limit, ds)
    if eta:
        b.set_eta(eta)
    b.apply()
    out = b.apply()
    b.status()
    for g, k, d, o in zip(gs, ks, ds, out):
        ref = qbx.qbx_apply_ops(pair_plan(g, 16, 64, nrhs, len(ops)), g, ops, side, limit, k, p, d, eta=eta or None)
        for i in ops:
            check(o[i], ref[i], (g.M, i))


def test_batch_super_blocks_match_single_curves(cuda):
    """Curves with super-blocks of several levels beside curves with none."""
    test_batch_clusters_match_single_curves(cuda, "two", 0, (0, 1), 0.0, False, Ms=(130, 9, 64, 16, 90, 63))


@pytest.mark.parametrize("order", ["dyadic", "shuffled"])
def test_clusters_on_uneven_and_unordered_panels(cuda, order):
    """Panels refined towards a corner (lengths over a factor of 64), and panels
    listed in random order, where clusters overlap each other and their targets."""
    cur = W.teardrop() if order == "dyadic" else W.starfish()
    edges = W.dyadic_edges(24, 6) if order == "dyadic" else cur.edges(48)
    M, k, p = len(edges) - 1, 6.0, 10
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=4, nrhs=1)
    g = qbx.qbx_geometry(plan, cur, edges)
    if order == "shuffled":
        perm = torch.as_tensor(np.random.default_rng(3).permutation(M), device="cuda")
        for n in ("src_x", "src_y", "src_nx", "src_ny", "src_w"):
            g[n].copy_(g[n].reshape(M, 64)[perm].reshape(-1).clone())
        for n in ("tgt_x", "tgt_y", "tgt_nx", "tgt_ny", "tgt_w"):
            g[n].copy_(g[n].reshape(M, 16)[perm].reshape(-1).clone())
        for n in ("ctr_x", "ctr_y", "ctr_r"):
            g[n].copy_(g[n].reshape(2, M, 16)[:, perm].reshape(-1).clone())
    d = torch.as_tensor(W.complex_gaussian(5, g.n_tgt).reshape(-1, 1), device="cuda")
    got = qbx.qbx_apply_ops(plan, g, (0, 1, 2), qbx.SIDE_EXT, 0, k, p, d)
    ref = qbx.qbx_apply_ops(pair_plan(g, 16, 64, 1, 4), g, (0, 1, 2), qbx.SIDE_EXT, 0, k, p, d)
    for o in (0, 1, 2):
        check(got[o], ref[o], (order, o))


ADJ = [
    # M, q_tgt, q_src, k, p, side, limit, nrhs
    (16, 16, 64, 5.0, 8, "int", 0, 1),
    (19, 7, 33, 9.0, 10, "ext", 1, 3),
    (40, 16, 64, 8.0, 0, "two", 0, 1),
    (40, 16, 64, 6.0, 40, "two", 0, 1),
    (48, 12, 40, 4 + 0.5j, 9, "two", 1, 2),
    (64, 16, 64, 60.0, 12, "int", 0, 1),
    (96, 16, 64, 12.0, 10, "ext", 0, 8),
]


@pytest.mark.parametrize("case", ADJ)
@pytest.mark.parametrize("op", [qbx.OP_S, qbx.OP_D])
def test_adjoint_clusters_match_pairs(cuda, case, op):
    """The transposed sweep, and the shape gradients, with and without clusters
    of the centres' discs (and of the sources, second derivatives included)."""
    M, qt, qs, k, p, side, limit, nrhs = case
    side = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}[side]
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, workspace_bytes=qbx.qbx_shape_adjoint_workspace_bytes(M, qt, qs, p, nrhs))
    g = geometry(plan, cur, cur.edges(M))
    d, go = (torch.as_tensor(W.complex_gaussian(M + p + i, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
             for i in (0, 1))
    al = lambda b: (b + 255) // 256 * 256
    ck = 16 if isinstance(k, complex) else 8
    nc = g.n_tgt * (2 if side == qbx.SIDE_TWO else 1)
    # room for the fixed arrays and two splits of either sweep only
    small = (2 * al(g.n_src * nrhs * 16) + al(nc * nrhs * 16) + al(nc * 2 * (p + 2) * ck) + al(nc * 32) + al(g.n_tgt * 8)
             + al(M * 8) + 2 * 2 * nc * 4 * nrhs * 16 + 2 * g.n_src * 5 * nrhs * 16 + 2048)
    pp = qbx.Plan(qt, qs, workspace_bytes=small)
    check(qbx.qbx_apply_adjoint(plan, g, op, side, limit, k, p, go),
          qbx.qbx_apply_adjoint(pp, g, op, side, limit, k, p, go), (case, op))
    got = qbx.qbx_apply_shape_adjoint(plan, g, side, k, p, d, go, op=op)
    ref = qbx.qbx_apply_shape_adjoint(pp, g, side, k, p, d, go, op=op)
    for i, (a, b) in enumerate(zip(got, ref)):
        # gradients through r = h/2 and the normals: a derivative of the order-p sums more, p/r times their rounding
        err = float((a - b).abs().max() / b.abs().max())
        assert np.isfinite(err) and err < 1e-11, (case, op, i, err)


@pytest.mark.parametrize("case", [c for c in ADJ if c[4] >= 1])
def test_grad_d_clusters_match_pairs(cuda, case):
    M, qt, qs, k, p, side, limit, nrhs = case
    nrhs = min(nrhs, 3)
    side = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}[side]
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=4, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M + p, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    got = qbx.qbx_apply(plan, g, qbx.OP_GRAD_D, side, limit, k, p, d)
    qbx.qbx_sync_status(plan)
    pp = qbx.Plan(qt, qs, workspace_bytes=(g.n_src * nrhs + 2 * g.n_tgt * 2 * nrhs * 3) * 16 + 2048)
    check(got, qbx.qbx_apply(pp, g, qbx.OP_GRAD_D, side, limit, k, p, d), case)


@pytest.mark.parametrize("M,qt,qs,k,p,kind,side,nrhs", [
    (16, 16, 64, 5.0, 8, 0, "int", 1), (33, 7, 33, 9.0, 10, 1, "ext", 3), (40, 16, 64, 6.0, 40, 1, "two", 1),
    (40, 16, 64, 8.0, 0, 0, "two", 8), (48, 12, 40, 4 + 0.5j, 9, 1, "two", 2), (64, 16, 64, 70.0, 12, 0, "int", 1)])
def test_locals_clusters_match_pairs(cuda, M, qt, qs, k, p, kind, side, nrhs):
    """Stored coefficients, each order against its own largest value, and the
    expansions evaluated at half the radius."""
    side = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}[side]
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=2 * p + 1, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    w = torch.as_tensor(W.complex_gaussian(M + p, g.n_src * nrhs).reshape(g.n_src, nrhs), device="cuda")
    nc = g.n_tgt * (2 if side == qbx.SIDE_TWO else 1)
    pp = qbx.Plan(qt, qs, workspace_bytes=nc * (2 * p + 1) * nrhs * 16 * 2 + 1024)
    got, ref = (qbx.qbx_form_locals(pl, g, kind, side, k, p, w) for pl in (plan, pp))
    qbx.qbx_sync_status(plan)
    for l in range(2 * p + 1):
        check(got[:, l], ref[:, l], (M, p, l - p))
    e = torch.arange(0, nc, 3, device="cuda", dtype=torch.int32)
    o = g.n_tgt if side == qbx.SIDE_EXT else 0
    ex = (g["ctr_x"][o:o + nc] + 0.5 * g["ctr_r"][o:o + nc])[e.long()].contiguous()
    ey = g["ctr_y"][o:o + nc][e.long()].contiguous()
    ev = [qbx.qbx_eval_locals(plan, g, side, k, p, a, ex=ex, ey=ey, ectr=e) for a in (got, ref)]
    check(ev[0], ev[1], (M, p))


@pytest.mark.parametrize("op,k,nrhs", [(qbx.OP_S, 9.0, 1), (qbx.OP_D, 9.0, 3), (qbx.OP_GRAD_S, 20.0, 1),
                                       (qbx.OP_R, 5 + 0.5j, 5), (qbx.OP_GRAD_S, 3 + 0.2j, 8), (qbx.OP_S, 150.0, 2)])
def test_far_points_clusters_match_pairs(cuda, op, k, nrhs):
    """Points in random order, from 1e-3 off the curve to far away, and one on a
    cluster's centre, where no cluster of it may be used."""
    M = 64
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=4000, ncoef=2, nrhs=nrhs)
    cur = W.starfish(0.2, 3)
    g = geometry(plan, cur, cur.edges(M))
    rng = np.random.default_rng(4)
    t = rng.uniform(0, 2 * np.pi, 1999)
    xy = cur(t)[0] * (1.0 + 10.0 ** rng.uniform(-3, 1.5, t.size))[:, None]
    xy[0] = [float(g["src_x"][:64].mean()), float(g["src_y"][:64].mean())]
    x = torch.as_tensor(xy, device="cuda")
    w = torch.as_tensor(W.complex_gaussian(7, g.n_src * nrhs).reshape(g.n_src, nrhs), device="cuda")
    comp = 2 if op == qbx.OP_GRAD_S else 1
    got = qbx.qbx_far(plan, g, op, k, w, x)
    qbx.qbx_sync_status(plan)
    pp = qbx.Plan(16, 64, workspace_bytes=len(t) * comp * nrhs * 16 * 2 + 2048 + g.n_src * 16)
    check(got, qbx.qbx_far(pp, g, op, k, w, x), (op, k))


def test_on_surface_with_far_points_fills_one_workspace(cuda):
    """Far points of an on-surface call share its workspace with the clusters."""
    M, n = 40, 3000
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=n, ncoef=2, nrhs=1)
    cur = W.starfish()
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(2, g.n_tgt).reshape(-1, 1), device="cuda")
    th = torch.linspace(0, 6.28, n, dtype=torch.float64, device="cuda")
    x = torch.stack([2 * torch.cos(th), 2 * torch.sin(th)], 1)
    on, far = qbx.qbx_apply(plan, g, qbx.OP_GRAD_S, qbx.SIDE_TWO, 0, 7.0, 8, d, x_far=x)
    pp = pair_plan(g, 16, 64, 1, 2)
    check(on, qbx.qbx_apply(pp, g, qbx.OP_GRAD_S, qbx.SIDE_TWO, 0, 7.0, 8, d), "on")
    p2 = qbx.Plan(16, 64, workspace_bytes=n * 2 * 16 * 2 + 2048)
    check(far, qbx.qbx_far(p2, g, qbx.OP_GRAD_S, 7.0, qbx.qbx_upsample(plan, g, d), x), "far")


def test_ratio_and_assignment_on_refined_panels(cuda):
    """Nearest-source ratios and disc assignment against numpy over panels whose
    lengths differ by 2^10 (the FP32 screening must not lose the nearest)."""
    edges = W.dyadic_edges(10, 10)
    M = len(edges) - 1
    plan = qbx.Plan(16, 64, workspace_bytes=1 << 20)
    g = qbx.qbx_geometry(plan, W.teardrop(), edges)
    c = np.stack([g["ctr_x"].cpu().numpy(), g["ctr_y"].cpu().numpy()], 1)
    s = np.stack([g["src_x"].cpu().numpy(), g["src_y"].cpu().numpy()], 1)
    r = g["ctr_r"].cpu().numpy()
    ref = np.array([np.sqrt(((s - q) ** 2).sum(1).min()) for q in c]) / r
    assert np.abs(g["ctr_ratio"].cpu().numpy() / ref - 1).max() < 1e-14
    rng = np.random.default_rng(1)
    i = rng.integers(0, g.n_tgt, 700)
    xy = c[i] + r[i, None] * rng.uniform(-0.9, 0.9, (700, 2))
    got = qbx.qbx_assign_centres(plan, g, qbx.SIDE_INT, torch.as_tensor(xy, device="cuda")).cpu().numpy()
    q = np.hypot(xy[:, None, 0] - c[None, :g.n_tgt, 0], xy[:, None, 1] - c[None, :g.n_tgt, 1]) / r[None, :g.n_tgt]
    want = np.where(q.min(1) <= 1.0, q.argmin(1), -1)
    assert np.array_equal(got, want)


def test_clusters_separate_densities_and_streams(cuda):
    """One density per operator, and the call on a stream of its own followed
    by work on that stream (the pair sums run beside it and join it)."""
    cur, M, k, p = W.starfish(), 50, 9.0, 10
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=4, nrhs=1)
    g = qbx.qbx_geometry(plan, cur, cur.edges(M))
    d = {o: torch.as_tensor(W.complex_gaussian(70 + o, g.n_tgt).reshape(-1, 1), device="cuda") for o in (0, 1, 2)}
    ref = qbx.qbx_apply_ops(pair_plan(g, 16, 64, 1, 4, nd=3), g, (0, 1, 2), qbx.SIDE_TWO, 0, k, p, d)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        got = qbx.qbx_apply_ops(plan, g, (0, 1, 2), qbx.SIDE_TWO, 0, k, p, d)
        twice = {o: got[o] * 2 for o in got}
    s.synchronize()
    for o in (0, 1, 2):
        check(0.5 * twice[o], ref[o], o)


def test_clusters_under_graph_capture(cuda):
    cur, M, k, p = W.starfish(), 40, 9.0, 10
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=2, nrhs=1)
    g = qbx.qbx_geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(1, g.n_tgt).reshape(-1, 1), device="cuda")
    out = {o: torch.empty(g.n_tgt, 1, dtype=torch.complex128, device="cuda") for o in (0, 1)}
    ref = {o: v.clone() for o, v in qbx.qbx_apply_ops(plan, g, (0, 1), qbx.SIDE_INT, 0, k, p, d).items()}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        qbx.qbx_apply_ops(plan, g, (0, 1), qbx.SIDE_INT, 0, k, p, d, out=out)
    for o in out:
        out[o].zero_()
    graph.replay()
    torch.cuda.synchronize()
    for o in ref:
        assert torch.equal(out[o], ref[o])


def test_non_finite_inputs_are_reported(cuda):
    """A non-finite density reaches every target, near or through clusters; a
    non-finite node makes its clusters inadmissible.  Both set the status word."""
    cur, M = W.starfish(), 32
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=2, nrhs=1)
    g = qbx.qbx_geometry(plan, cur, cur.edges(M))
    d = torch.ones(g.n_tgt, 1, dtype=torch.complex128, device="cuda")
    d[3] = complex(float("nan"), 0.0)
    out = qbx.qbx_apply(plan, g, qbx.OP_S, qbx.SIDE_INT, 0, 5.0, 8, d)
    with pytest.raises(qbx.QBXError):
        qbx.qbx_sync_status(plan)
    assert not torch.isfinite(out.abs()).any()
    d[3] = 1.0
    g["src_x"][700] = float("inf")
    qbx.qbx_apply(plan, g, qbx.OP_S, qbx.SIDE_INT, 0, 5.0, 8, d)
    with pytest.raises(qbx.QBXError):
        qbx.qbx_sync_status(plan)


@pytest.mark.parametrize("M,qt,qs,k,p,scale", [
    (16, 16, 64, 5.0, 8, 1.0), (33, 16, 64, 9.0, 10, 1.0), (41, 5, 21, 7.0, 6, 1.0), (37, 9, 128, 4.0, 12, 1.0),
    (37, 9, 127, 4 + 0.3j, 12, 1.0), (40, 12, 40, 6 + 0.5j, 9, 1.0), (40, 16, 64, 60.0, 12, 1.0),
    (40, 16, 64, 1e-3, 1, 1.0), (40, 16, 16, 5.0, 20, 1e-4), (50, 16, 64, 5.0, 30, 1.0), (64, 1, 8, 3.0, 0, 1.0)])
def test_assembled_matrix_clusters_match_pairs(cuda, M, qt, qs, k, p, scale):
    """Every entry against the largest: the rows of a far panel are cut at 5e-17 of a kernel value."""
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=8, nrhs=qt)
    g = geometry(plan, cur, cur.edges(M), scale)
    got = qbx.qbx_assemble_cfie(plan, g, k / scale, (2.0 - 0.5j) / scale, p)
    ref = qbx.qbx_assemble_cfie(qbx.Plan(qt, qs, workspace_bytes=4096), g, k / scale, (2.0 - 0.5j) / scale, p)
    check(got, ref, "A")


@pytest.mark.parametrize("k", [2 + 6j, 0.1 + 9j, 30 + 30j])
def test_hankel_ray_at_strong_damping(cuda, k):
    """The amplitude table loses nothing to e^{2 Im z}: scipy's scaled Hankel
    functions along the ray up to Im z = 60, each value to the fit's 1e-15 and
    the phase's z eps (2e-14 at Re z = 60), with a margin of four."""
    plan = qbx.Plan(16, 64, workspace_bytes=1 << 12)
    rho = np.linspace(2.01, 60.0, 1500) / abs(k)
    z = k * rho
    h0, h1 = qbx.qbx_debug_hankel01_ray(plan, k, torch.as_tensor(rho, device="cuda"))
    for n, h in ((0, h0), (1, h1)):
        ref = sp.hankel1e(n, z) * np.exp(1j * z)
        assert np.all(np.abs(h.cpu().numpy() - ref) <= 8e-14 * np.abs(ref)), n


class Circles:
    """n unit circles in a row, 3 apart, one after another in the parameter."""

    def __init__(self, n):
        self.n = n

    def __call__(self, t):
        j = np.minimum(np.floor(t / (2 * np.pi)), self.n - 1)
        c, s = np.cos(t), np.sin(t)
        return np.stack([3.0 * j + c, s], -1), np.stack([-s, c], -1)

    def edges(self, M):
        return np.linspace(0.0, 2 * np.pi * self.n, M + 1)


def test_parent_node_smaller_than_its_children(cuda):
    """Circles of 8 panels, two sides, 16 columns: at k = 6.5 the node of a
    circle (k R = 6.5) is in the lists of distant blocks, the nodes of its
    halves, whose radius about the centre of their bounding box is 1.118, are
    beyond every list's limit (7.23).  A first call leaves NaN in every row."""
    M, nrhs, p, ops = 256, 16, 10, (0, 1)
    assert 2 * M * len(ops) * nrhs > 8192   # moments carried upward
    cur = Circles(32)
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=4, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(3, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    qbx.qbx_apply_ops(plan, g, ops, qbx.SIDE_TWO, 0, 1.0, p, torch.full_like(d, float("nan")))
    with pytest.raises(qbx.QBXError):
        qbx.qbx_sync_status(plan)
    got = qbx.qbx_apply_ops(plan, g, ops, qbx.SIDE_TWO, 0, 6.5, p, d)
    qbx.qbx_sync_status(plan)
    ref = qbx.qbx_apply_ops(pair_plan(g, 16, 64, nrhs, 2), g, ops, qbx.SIDE_TWO, 0, 6.5, p, d)
    b = qbx.Batch(plan, [g], [6.5], p, ops, qbx.SIDE_TWO, 0, [d])
    out = b.apply()[0]
    b.status()
    for o in ops:
        check(got[o], ref[o], ("apply", o))
        check(out[o], ref[o], ("batch", o))


@pytest.mark.parametrize("M,k,p,kind", [(40, 1e-3, 40, 0), (40, 1e-4, 24, 1), (40, 3e-4, 30, 0), (40, 1e-4, 30, 0),
                                        (130, 1e-3, 40, 1), (40, 1e-3 + 1e-3j, 40, 0)])
def test_locals_at_low_frequency_stay_finite(cuda, M, k, p, kind):
    """Every order l <= p from distant nodes, whose waves H_{om + l} reach 1e344
    where H_p of the pairs stays below 1e270."""
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=M * 16, ncoef=2 * p + 1, nrhs=1)
    g = geometry(plan, cur, cur.edges(M))
    w = torch.as_tensor(W.complex_gaussian(M + p, g.n_src).reshape(g.n_src, 1), device="cuda")
    pp = qbx.Plan(16, 64, workspace_bytes=g.n_tgt * (2 * p + 1) * 16 * 2 + 1024)
    got, ref = (qbx.qbx_form_locals(pl, g, kind, qbx.SIDE_INT, k, p, w) for pl in (plan, pp))
    qbx.qbx_sync_status(plan)
    for l in range(2 * p + 1):
        check(got[:, l], ref[:, l], (M, p, l - p))


@pytest.mark.parametrize("M", [8, 40])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_weighted_density_at_an_odd_8_byte_address(cuda, M, nrhs):
    """qbx_c64 asks for the alignment of a double only: the same bits from an
    array 8 bytes off, pair by pair and through clusters."""
    k, p = 6.0, 9
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=2 * p + 1, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    w = torch.as_tensor(W.complex_gaussian(M, g.n_src * nrhs).reshape(g.n_src, nrhs), device="cuda")
    flat = torch.zeros(2 * g.n_src * nrhs + 1, dtype=torch.float64, device="cuda")
    flat[1:] = torch.view_as_real(w).reshape(-1)
    ptr = flat.data_ptr() + 8
    assert ptr % 16 == 8
    for kind in (qbx.OP_S, qbx.OP_D):
        ref = qbx.qbx_form_locals(plan, g, kind, qbx.SIDE_INT, k, p, w)
        out = torch.empty_like(ref)
        stream = torch.cuda.current_stream().cuda_stream
        assert qbx.lib().qbx_form_locals(plan.handle, g.ref(), kind, qbx.SIDE_INT, qbx.c64(k, 0.0), p, ptr, nrhs,
                                         out.data_ptr(), stream) == 0
        assert torch.equal(out, ref)


@pytest.mark.parametrize("call", ["apply", "locals", "grad_d_stored"])
def test_captured_calls_at_complex_k_keep_their_k(cuda, call):
    """A graph replayed after a call at another k, and calls at that k after the
    replay, on one plan: each takes the amplitudes of its own k."""
    M, p, k1, k2 = 24, 8, 5 + 0.5j, 9 + 0.3j
    nrhs = 4 if call == "grad_d_stored" else 1
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=2 * p + 1, nrhs=nrhs)
    cur = W.starfish(0.2, 3)
    g = geometry(plan, cur, cur.edges(M))
    n = g.n_src if call == "locals" else g.n_tgt
    d = torch.as_tensor(W.complex_gaussian(4, n * nrhs).reshape(n, nrhs), device="cuda")

    def run(k):
        if call == "locals":
            return qbx.qbx_form_locals(plan, g, qbx.OP_D, qbx.SIDE_INT, k, p, d)
        return qbx.qbx_apply(plan, g, qbx.OP_S if call == "apply" else qbx.OP_GRAD_D, qbx.SIDE_INT, 0, k, p, d)

    r2, r1 = run(k2).clone(), run(k1).clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = run(k1)
    assert torch.equal(run(k1), r1)   # (the captured table fill has not run yet)
    assert torch.equal(run(k2), r2)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, r1)
    assert torch.equal(run(k2), r2)
    fresh = torch.cuda.CUDAGraph()
    k3 = 4 + 1j
    with torch.cuda.graph(fresh):
        out3 = run(k3)
    now = run(k3)   # (a new k, captured before it was ever made)
    fresh.replay()
    torch.cuda.synchronize()
    assert torch.equal(out3, now) and torch.isfinite(torch.view_as_real(now)).all()


@pytest.mark.parametrize("M,ops,nrhs", [(16, (0,), 1), (128, (0,), 1), (256, (1,), 1), (256, (0, 1), 1), (256, (2,), 1),
                                        (128, (0, 1), 3), (1024, (0,), 1), (1024, (0, 1, 2), 1), (256, (1,), 16),
                                        (96, (0, 1), 16)])
def test_documented_workspace_holds_the_clusters(cuda, M, ops, nrhs):
    """qbx_workspace_bytes for one side and the operators' components: distant
    sources through moments, with the bits of a plan of twice the room."""
    k, p = 0.05 * M, 8
    ncoef = sum(2 if o == 2 else 1 for o in ops)
    cur = W.starfish(0.2, 3)
    size = qbx.qbx_workspace_bytes(M * 64, M * 16, ncoef, nrhs)
    plan, big = (qbx.Plan(16, 64, workspace_bytes=b) for b in (size, 2 * size + (64 << 20)))
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    got = qbx.qbx_apply_ops(plan, g, ops, qbx.SIDE_INT, 0, k, p, d)
    assert qbx.qbx_debug_route(plan)[0] == 1
    ref = qbx.qbx_apply_ops(big, g, ops, qbx.SIDE_INT, 0, k, p, d)
    assert qbx.qbx_debug_route(plan) == qbx.qbx_debug_route(big)
    for o in ops:
        assert torch.equal(got[o], ref[o])


def test_documented_workspace_holds_separate_densities_and_grad_d(cuda):
    M, k, p = 256, 12.0, 8
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(16, 64, workspace_bytes=qbx.qbx_workspace_bytes(M * 64, M * 16, 4, 1))
    g = geometry(plan, cur, cur.edges(M))
    d = {o: torch.as_tensor(W.complex_gaussian(o, g.n_tgt).reshape(-1, 1), device="cuda") for o in (0, 1, 2)}
    qbx.qbx_apply_ops(plan, g, (0, 1, 2), qbx.SIDE_INT, 0, k, p, d)
    assert qbx.qbx_debug_route(plan)[0] == 1
    plan = qbx.Plan(16, 64, workspace_bytes=qbx.qbx_workspace_bytes(M * 64, M * 16, 2, 1))
    qbx.qbx_apply(plan, g, qbx.OP_GRAD_D, qbx.SIDE_INT, 0, k, p, d[0])
    assert qbx.qbx_debug_route(plan)[0] == 1
    plan = qbx.Plan(16, 64, workspace_bytes=qbx.qbx_workspace_bytes(M * 64, M * 16, 2 * p + 1, 1))
    qbx.qbx_form_locals(plan, g, qbx.OP_D, qbx.SIDE_INT, k, p, qbx.qbx_upsample(plan, g, d[0]))
    assert qbx.qbx_debug_route(plan)[0] == 1


ROUTES = [
    # M, q_tgt, q_src, ops, side, nrhs, eta, clusters: either side of the rules by pairs, columns and sources per leaf
    (32, 16, 64, (0, 1, 2), "two", 16, None, 0), (48, 16, 64, (0, 1, 2), "two", 16, None, 1),   # the far values anew for 2 rhs
    (48, 16, 64, (0, 1, 2), "int", 16, None, 1), (64, 16, 64, (0, 1, 2), "int", 32, None, 0),
    (96, 16, 64, (0, 1, 2), "int", 32, None, 1), (64, 16, 64, (0, 1, 2), "two", 32, None, 0),
    (24, 16, 64, "cfie", "two", 8, None, 1), (48, 8, 32, "cfie", "two", 8, None, 0),            # leaves of 16 sources
    (200, 4, 8, "cfie", "two", 1, None, 0), (220, 4, 8, "cfie", "two", 1, None, 1),             # of 8
    (32, 16, 64, "cfie", "two", 32, None, 1), (64, 8, 32, "cfie", "two", 32, None, 0),
    (20, 16, 64, (0, 1), "two", 16, None, 1), (40, 16, 16, (0, 1), "two", 16, None, 0),
    (150, 4, 8, (0, 1), "two", 16, None, 0), (200, 4, 8, (0,), "int", 16, None, 0),
    (96, 8, 32, (0, 1), "int", 32, None, 0), (48, 16, 64, (0, 1), "int", 32, None, 1),
    (32, 16, 64, (0, 1), "two", 16, 6.0, 0), (40, 16, 64, (0, 1), "two", 16, 6.0, 1),           # the pairs beyond eta r are cheap
    (24, 16, 64, (0, 1), "int", 16, 10.0, 0), (48, 16, 64, (0, 1), "int", 32, 10.0, 0), (64, 16, 64, (0, 1), "int", 32, 10.0, 1),
    (48, 16, 64, (0, 1, 2), "int", 16, 10.0, 0), (64, 16, 64, (0, 1, 2), "int", 16, 10.0, 1),
    (45, 12, 40, (2,), "int", 16, None, 0), (64, 16, 64, (2,), "int", 16, None, 1),
    (48, 16, 64, (2,), "two", 8, None, 0), (64, 16, 64, (2,), "two", 8, None, 1), (24, 16, 64, (2,), "two", 3, None, 1),
    (16, 16, 64, (0, 1, 2), "int", 1, None, 1), (15, 16, 64, (0, 1, 2), "int", 1, None, 0),     # few columns: by panels alone
]


@pytest.mark.parametrize("case", ROUTES)
def test_route_rules(cuda, case):
    """Which calls go through clusters, and that both routes agree there."""
    M, qt, qs, ops, side, nrhs, eta, want = case
    side = {"int": qbx.SIDE_INT, "two": qbx.SIDE_TWO}[side]
    k, p = M * qs / 64 * 0.15, 8
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=4, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M + nrhs, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    ncomp = 1 if ops == "cfie" else sum(2 if o == 2 else 1 for o in ops)
    pp = pair_plan(g, qt, qs, nrhs, ncomp)
    run = lambda pl: ([qbx.qbx_apply_cfie(pl, g, k, k - 0.5j, p, d)] if ops == "cfie" else
                      list(qbx.qbx_apply_ops(pl, g, ops, side, 0, k, p, d, eta=eta).values()))
    got = run(plan)
    assert qbx.qbx_debug_route(plan)[0] == want
    ref = run(pp)
    assert qbx.qbx_debug_route(pp) == (0, 0, 0)
    for i, (a, b) in enumerate(zip(got, ref)):
        check(a, b, (case, i))


@pytest.mark.parametrize("call,M,q_tgt,q_src,side,nrhs,want", [
    ("adjoint", 33, 16, 64, "int", 1, 0), ("adjoint", 35, 16, 64, "int", 1, 1), ("adjoint", 48, 16, 64, "int", 3, 1),
    ("adjoint", 32, 16, 64, "two", 3, 0), ("adjoint", 64, 16, 64, "int", 8, 0), ("adjoint", 72, 16, 64, "int", 8, 1),
    ("shape_s", 16, 16, 64, "int", 1, 1), ("shape_s", 32, 16, 64, "int", 3, 0), ("shape_s", 40, 16, 64, "int", 3, 1),
    ("shape_s", 38, 16, 64, "int", 8, 0), ("shape_s", 48, 16, 64, "int", 8, 1), ("shape_d", 20, 16, 64, "int", 8, 1),
    ("locals", 16, 16, 64, "int", 1, 1), ("locals", 200, 4, 8, "int", 1, 0), ("locals", 200, 4, 8, "two", 1, 1),
    ("assemble", 40, 16, 16, "two", 1, 0), ("assemble", 40, 16, 64, "two", 1, 1), ("assemble", 40, 8, 32, "two", 1, 1)])
def test_route_rules_of_adjoints_locals_and_the_matrix(cuda, call, M, q_tgt, q_src, side, nrhs, want):
    side = {"int": qbx.SIDE_INT, "two": qbx.SIDE_TWO}[side]
    k, p = M * q_src / 64 * 0.15, 8
    cur = W.starfish(0.2, 3)
    size = max(qbx.qbx_workspace_bytes(M * q_src, 2 * M * q_tgt, 2 * p + 1, nrhs),
               qbx.qbx_workspace_bytes(M * q_src, 2 * M * q_tgt, 4, max(nrhs, q_tgt)),
               qbx.qbx_shape_adjoint_workspace_bytes(M, q_tgt, q_src, p, nrhs))
    plan = qbx.Plan(q_tgt, q_src, workspace_bytes=size)
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    if call == "adjoint":
        qbx.qbx_apply_adjoint(plan, g, qbx.OP_S, side, 0, k, p, d)
    elif call == "locals":
        qbx.qbx_form_locals(plan, g, qbx.OP_S, side, k, p, qbx.qbx_upsample(plan, g, d))
    elif call == "assemble":
        qbx.qbx_assemble_cfie(plan, g, k, k, p)
    else:
        qbx.qbx_apply_shape_adjoint(plan, g, side, k, p, d, d, op=qbx.OP_S if call == "shape_s" else qbx.OP_D)
    assert qbx.qbx_debug_route(plan)[0] == want


@pytest.mark.parametrize("M,q_tgt,q_src,ops,nrhs", [(16, 16, 64, (0,), 32), (31, 12, 40, (0,), 4), (12, 16, 64, (0, 1), 32)])
def test_batch_of_one_small_curve_on_both_sides(cuda, M, q_tgt, q_src, ops, nrhs):
    """Both sides of a target are one item, twice as long per source: ranges down
    to 256 sources there, so that there are no fewer items than one side at a time has."""
    plan = qbx.Plan(q_tgt, q_src, n_src=M * q_src, n_ctr=2 * M * q_tgt, ncoef=2, nrhs=nrhs)
    cur = W.starfish(0.2, 3)
    g = qbx.qbx_geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    b = qbx.Batch(plan, [g], [3.0], 7, ops, qbx.SIDE_TWO, 0, [d])
    one = qbx.Batch(plan, [g], [3.0], 7, ops, qbx.SIDE_INT, 0, [d])
    assert b.info()[1] == one.info()[1] // 2 and b.info()[2] >= 2 * ((g.n_tgt + 31) // 32) * (g.n_src // 512)
    out = b.apply()[0]
    b.status()
    ref = qbx.qbx_apply_ops(pair_plan(g, q_tgt, q_src, nrhs, len(ops)), g, ops, qbx.SIDE_TWO, 0, 3.0, 7, d)
    for o in ops:
        check(out[o], ref[o], o)


@pytest.mark.parametrize("q_tgt,q_src,M,nrhs", [(10, 100, 40, 4), (4, 8, 100, 16), (5, 21, 9, 3), (3, 16, 7, 17)])
def test_group_blocks_across_the_sides(cuda, q_tgt, q_src, M, nrhs):
    """400, 400, 45 and 21 targets (no multiple of 32), S + D + grad S on both
    sides: pair by pair 32 centres to a block across the sides, in a batch and
    (from 16 rhs on) in one apply; against single right-hand sides."""
    plan = qbx.Plan(q_tgt, q_src, n_src=M * q_src, n_ctr=2 * M * q_tgt, ncoef=4, nrhs=nrhs)
    cur, k, p, ops = W.starfish(0.2, 3), 3.0, 7, (0, 1, 2)
    g = qbx.qbx_geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    b = qbx.Batch(plan, [g, g], [k, k], p, ops, qbx.SIDE_TWO, 0, [d, d])
    n = b.info()[2]
    assert n % (2 * ((2 * g.n_tgt + 31) // 32)) == 0   # items: blocks of both sides together, times equal ranges
    outs = b.apply()
    b.status()
    got = qbx.qbx_apply_ops(plan, g, ops, qbx.SIDE_TWO, 0, k, p, d)
    for r in range(0, nrhs, 3):
        pp = pair_plan(g, q_tgt, q_src, 1, 4)
        ref = qbx.qbx_apply_ops(pp, g, ops, qbx.SIDE_TWO, 0, k, p, d[:, r:r + 1].contiguous())
        for o in ops:
            check(got[o][..., r:r + 1], ref[o], ("apply", o, r))
            for out in outs:
                check(out[o][..., r:r + 1], ref[o], ("batch", o, r))


@pytest.mark.parametrize("Ms,q_tgt,q_src,side,ops,nrhs,eta,want", [
    ((31,), 16, 64, "int", (0, 1), 4, 0.0, 0), ((32,), 16, 64, "int", (0, 1), 4, 0.0, 1),
    ((47,), 16, 64, "int", (0, 1), 32, 0.0, 0), ((40, 30, 9), 16, 64, "int", (0, 1), 32, 0.0, 1),
    ((100,) * 12, 4, 8, "int", (0, 1), 32, 0.0, 0), ((150,) * 12, 4, 8, "int", (0, 1), 32, 0.0, 1),
    ((64,), 8, 32, "int", (0,), 16, 0.0, 0), ((32,), 16, 64, "two", (0,), 12, 8.0, 0), ((40,), 16, 64, "two", (0,), 12, 8.0, 1)])
def test_batch_route_rules(cuda, Ms, q_tgt, q_src, side, ops, nrhs, eta, want):
    side, k, p = {"int": qbx.SIDE_INT, "two": qbx.SIDE_TWO}[side], 4.0, 7
    cur = W.starfish(0.15, 3)
    plan = qbx.Plan(q_tgt, q_src, n_src=q_src * max(Ms), n_ctr=2 * q_tgt * max(Ms), ncoef=2, nrhs=nrhs)
    gs = [qbx.qbx_geometry(plan, cur, cur.edges(M)) for M in Ms]
    ds = [torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
          for M, g in zip(Ms, gs)]
    b = qbx.Batch(plan, gs, [k] * len(Ms), p, ops, side, 0, ds)
    if eta:
        b.set_eta(eta)
    assert b.debug_route() == want
    out = b.apply()
    b.status()
    ref = qbx.qbx_apply_ops(pair_plan(gs[0], q_tgt, q_src, nrhs, len(ops)), gs[0], ops, side, 0, k, p, ds[0], eta=eta or None)
    for o in ops:
        check(out[0][o], ref[o], o)


def test_batch_tuning_is_kept_apart_for_clusters_and_pairs(cuda):
    """Two batches whose pairs lie in one power-of-two bucket on either side of
    the clusters' threshold: tuning one leaves the other its own items."""
    nrhs, p, ops = 12, 7, (0,)
    cur = W.starfish(0.15, 3)
    plan = qbx.Plan(16, 64, n_src=64 * 32, n_ctr=32 * 32, ncoef=2, nrhs=nrhs)

    def batch(Ms):
        gs = [qbx.qbx_geometry(plan, cur, cur.edges(M)) for M in Ms]
        ds = [torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
              for M, g in zip(Ms, gs)]
        return qbx.Batch(plan, gs, [4.0, 3.0], p, ops, qbx.SIDE_INT, 0, ds)

    pairs, clusters = (30, 8), (30, 10)   # 0.99e6 and 1.02e6 pairs, between 2^19 and 2^20
    a, b = batch(pairs), batch(clusters)
    assert a.debug_route() == 0 and b.debug_route() == 1
    own = a.info()
    b.tune()
    assert batch(pairs).info() == own
    assert a.info() == own and own[1] >= 512


@pytest.mark.parametrize("M,q_tgt,q_src,nrhs", [(70, 4, 8, 1), (18, 16, 64, 33), (100, 4, 8, 16)])
def test_few_items_beyond_whole_rounds(cuda, M, q_tgt, q_src, nrhs):
    """9 x 17, 9 x 34 and 13 x 25 items over 152 SMs: a split or two fewer, and
    the sums as with two splits."""
    k, p = 2.0, 8
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(q_tgt, q_src, n_src=M * q_src, n_ctr=2 * M * q_tgt, ncoef=2, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    got = qbx.qbx_apply_cfie(plan, g, k, k, p, d)
    assert qbx.qbx_debug_route(plan)[0] == 0
    check(got, qbx.qbx_apply_cfie(pair_plan(g, q_tgt, q_src, nrhs, 1), g, k, k, p, d), M)


MANY = [
    # M, q_tgt, q_src, k, p, ops, side, limit, nrhs, eta, (carried upward, super-blocks)
    (32, 16, 64, 5.0, 8, (0,), "int", 0, 16, None, (0, 0)),            # smallest
    (75, 12, 40, 9.0, 10, (1,), "ext", 1, 17, None, (0, 0)),           # blocks across panels, a ragged column group
    (75, 7, 33, 7.0, 6, (0, 1), "two", 0, 33, None, (0, 0)),           # whole-panel leaves, 66 columns: two passes
    (131, 7, 33, 7.0, 6, (0, 1), "two", 0, 33, None, (1, 1)),
    (63, 16, 64, 9.0, 10, (0, 1), "two", 0, 33, None, (1, 0)),         # upward, a leaf short of super-blocks
    (64, 16, 64, 9.0, 10, (0, 1), "two", 0, 33, None, (1, 1)),         # fewest leaves with them
    (62, 16, 64, 9.0, 10, (0, 1), "two", 0, 33, None, (0, 0)),         # 8184 leaf columns
    (64, 16, 64, 6.0, 40, (0, 1), "int", 1, 33, None, (1, 1)),         # highest order
    (64, 16, 64, 6.0, 0, (0, 1), "two", 0, 33, None, (1, 1)),          # lowest
    (128, 16, 64, 9.0, 9, (0,), "int", 0, 16, None, (0, 1)),           # super-blocks by blocks, not upward
    (128, 16, 64, 9 + 0.5j, 9, (0,), "int", 0, 16, None, (0, 0)),      # (complex k: from 128 blocks on)
    (128, 16, 64, 1e-3, 8, (0,), "two", 0, 33, None, (1, 1)),          # Laplace-like
    (200, 5, 21, 7.0, 6, (1,), "ext", 1, 48, None, (1, 1)),            # several panels per block
    (96, 16, 64, 12.0, 10, (0, 1), "two", 0, 48, 6.0, (1, 1)),         # near-only
    (130, 16, 64, 3 + 3j, 10, "cfie", "two", 0, 40, None, (1, 1)),
    (131, 16, 64, 30.0, 12, "cfie", "two", 0, 65, None, (1, 1)),
]


@pytest.mark.parametrize("case", MANY)
def test_many_columns_by_route(cuda, case):
    """Sums at every level and moments carried upward, with and without
    super-blocks: the route that each size stands for, and the pairs' result."""
    M, qt, qs, k, p, ops, side, limit, nrhs, eta, (up, sup) = case
    side = {"int": qbx.SIDE_INT, "ext": qbx.SIDE_EXT, "two": qbx.SIDE_TWO}[side]
    cur = W.starfish(0.2, 3)
    plan = qbx.Plan(qt, qs, n_src=M * qs, n_ctr=2 * M * qt, ncoef=4, nrhs=nrhs)
    g = geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M + p, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    pp = pair_plan(g, qt, qs, nrhs, 1 if ops == "cfie" else len(ops))
    run = lambda pl: ([qbx.qbx_apply_cfie(pl, g, k, k - 0.5j, p, d)] if ops == "cfie" else
                      list(qbx.qbx_apply_ops(pl, g, ops, side, limit, k, p, d, eta=eta).values()))
    got = run(plan)
    qbx.qbx_sync_status(plan)
    r = qbx.qbx_debug_route(plan)
    assert r[:2] == (1, up) and (r[2] > 0) == bool(sup)
    ref = run(pp)
    assert qbx.qbx_debug_route(pp)[0] == 0
    for i, (a, b) in enumerate(zip(got, ref)):
        check(a, b, (case, i))


@pytest.mark.parametrize("M,q_tgt,q_src", [(16, 4, 8), (20, 16, 64), (100, 4, 8), (2, 5, 7)])
def test_batch_items_of_both_sides_are_as_many_as_of_one_each(cuda, M, q_tgt, q_src):
    """64, 320, 400 and 10 targets: as many items as both sides one by one have,
    also where a side's sources are a single range."""
    nrhs, k, p = 4, 2.0, 7
    plan = qbx.Plan(q_tgt, q_src, n_src=M * q_src, n_ctr=2 * M * q_tgt, ncoef=2, nrhs=nrhs)
    cur = W.starfish(0.2, 3)
    g = qbx.qbx_geometry(plan, cur, cur.edges(M))
    d = torch.as_tensor(W.complex_gaussian(M, g.n_tgt * nrhs).reshape(g.n_tgt, nrhs), device="cuda")
    one, b = (qbx.Batch(plan, [g], [k], p, (0,), s, 0, [d]) for s in (qbx.SIDE_INT, qbx.SIDE_TWO))
    assert one.debug_route() == b.debug_route() == 0
    if g.n_src >= 32:
        assert b.info()[2] >= 2 * one.info()[2]
    out = b.apply()[0]
    b.status()
    ref = qbx.qbx_apply_ops(pair_plan(g, q_tgt, q_src, nrhs, 1), g, (0,), qbx.SIDE_TWO, 0, k, p, d)
    check(out[0], ref[0], M)
