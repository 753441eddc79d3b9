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
