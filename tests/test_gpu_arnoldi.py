"""The solver's Arnoldi kernels where their splits can go wrong: one
right-hand side (all threads of a CTA on one column), counts that do not
divide a CTA, more than a CTA has threads (several passes), cycles from two
steps on, meshes of fewer target rows than CTAs and of several rows per CTA,
with the assembled matrix and matrix-free."""
import numpy as np
import pytest
import torch

import paper_1207_4461_gb300 as qbx
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("panels,nrhs,restart,assembled", [
    (8, 1, 30, True), (8, 300, 30, True), (8, 5, 2, True), (24, 16, 7, True), (24, 1, 60, True), (24, 33, 60, True),
    (24, 7, 60, False), (8, 1, 3, False)])
def test_solution_satisfies_the_dense_system(cuda, panels, nrhs, restart, assembled):
    """The true residual of every system, f - A mu in the sqrt-weight norm, is
    the estimate the solver stops at: <= 1e-10, with a tenth for the rounding
    of the two products (n eps = 1e-13 of the norm) and of the matrix-free
    operator against the assembled one (1e-12)."""
    edges = W.dyadic_edges(panels, 2)
    M = len(edges) - 1
    plan = qbx.Plan(16, 64, n_src=M * 64, n_ctr=2 * M * 16, ncoef=4, nrhs=nrhs)
    g = qbx.qbx_geometry(plan, W.teardrop(), edges)
    k, p, n = 3.0, 6, g.n_tgt
    A = qbx.qbx_assemble_cfie(plan, g, k, k, p)
    gen = torch.Generator(device="cuda").manual_seed(5)
    f = torch.randn(n, nrhs, dtype=torch.complex128, device="cuda", generator=gen)
    mu, its, res = qbx.qbx_solve_exterior_dirichlet(plan, g, k, k, p, f, tol=1e-10, restart=restart, maxiter=4000,
                                                     A=A if assembled else None)
    assert np.all(res <= 1e-10)
    sw = torch.sqrt(g["tgt_w"]).reshape(-1, 1)
    r = sw * f - A.T @ (sw * mu)
    rel = torch.linalg.norm(r, dim=0) / torch.linalg.norm(sw * f, dim=0)
    assert float(rel.max()) <= 1.1e-10
