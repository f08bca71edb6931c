"""Solutions returned by a low-precision solve: X, G and the reported residual belong together, also after the extra cycle
that columns get which only just meet the tolerance, and at tolerances near the floor of the residual, where that cycle
cannot improve every column."""
import numpy as np
import pytest

from oracle import bc, hbar
from oracle import sigma as sg

from gpu_util import inputs, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.mark.parametrize("prec", ["tf32", "bf16"])
@pytest.mark.parametrize("o,v,np_,nw,tol", [(4, 8, 4, 7, 1e-6), (7, 13, 7, 5, 1e-10), (5, 12, 5, 6, 3e-13), (4, 8, 12, 5, 2e-14)])
def test_solution_and_residual_belong_together(torch, prec, o, v, np_, nw, tol):
    from paper_1902_06016_gb300 import Context
    inp = inputs(o, v, 103)
    M = sg.dense_matrix(hbar.build(inp))
    porb, eta = list(range(np_)), 0.005
    ws = np.linspace(-1.0, -0.1, nw)
    B, C = bc.b_vectors(inp, porb), bc.c_vectors(inp, porb)
    ctx = Context(inp, tol=tol, precision=prec, residual_precision="fp64", max_restarts=25)
    r = ctx.solve_full(ws, eta, porb, want_A=False, want_X=True)
    plain = ctx.solve_full(ws, eta, porb, want_A=False)
    ctx.close()
    worst, slack = 0.0, 0.0
    for k, w in enumerate(ws):
        A, X = M + (w - 1j * eta) * np.eye(inp.dim), r["X"][k]
        bn = np.linalg.norm(B, axis=1)
        worst = max(worst, (np.linalg.norm(X @ A.T - B, axis=1) / bn).max())
        # the rounding of this product and of the library's own residual
        slack = max(slack, (8.0 * inp.dim * 2.0 ** -53 * np.linalg.norm(np.abs(X) @ np.abs(A).T, axis=1) / bn).max())
        # G = c^T X of the returned X, up to the rounding of the sums
        bound = 4.0 * inp.dim * 2.0 ** -53 * (np.abs(X) @ np.abs(C).T)
        assert np.all(np.abs(r["G"][k] - X @ C.T) <= bound)
    # the reported residual is the one of the solutions returned, and below the tolerance wherever the call says so
    assert abs(worst - r["stats"].max_rel_res) <= slack
    assert not r["converged"] or r["stats"].max_rel_res <= tol
    assert r["converged"] or tol <= slack     # only below the rounding of the residual itself may the cycles run out
    # X or not, the same tolerance holds
    assert plain["converged"] == r["converged"] or tol <= slack
