"""Arnoldi sweeps of the FP32 basis with delayed re-orthogonalisation, and the dot products, updates and norms of the
FP64 basis: batches of every block width (4, 8, 16 and 32 columns, full and ragged), bases beyond the 32 vectors of
one sweep, spaces smaller than the restart length (the basis breaks down) and a restart length of one."""
import numpy as np
import pytest

from oracle import bc, hbar
from oracle import sigma as sg

from gpu_util import inputs, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.mark.parametrize("prec", ["bf16", "tf32", "fp64", "fp64_tc"])
@pytest.mark.parametrize("o,v,np_,nw,restart,eta", [
    (2, 1, 1, 1, 30, 0.05), (2, 1, 2, 3, 40, 0.05),
    (4, 8, 1, 1, 40, 0.005), (4, 8, 3, 1, 70, 0.005), (4, 8, 1, 5, 33, 0.005), (4, 8, 3, 3, 32, 0.005),
    (4, 8, 1, 17, 31, 0.005), (4, 8, 3, 11, 100, 0.005), (7, 13, 20, 13, 65, 0.01), (3, 5, 8, 4, 1, 0.5)])
def test_sweeps_at_every_batch_width_and_basis_length(torch, prec, o, v, np_, nw, restart, eta):
    from paper_1902_06016_gb300 import Context
    inp = inputs(o, v, 103)
    M = sg.dense_matrix(hbar.build(inp))
    porb = list(range(np_))
    ws = np.linspace(-1.0, 0.0, nw)
    tol = 1e-10
    ctx = Context(inp, tol=tol, precision=prec, residual_precision="fp64", restart=restart, max_restarts=2000)
    r = ctx.solve_full(ws, eta, porb, want_X=True)
    assert r["converged"] and r["stats"].max_rel_res <= tol
    B = bc.b_vectors(inp, porb)
    for k, w in enumerate(ws):
        A = M + (w - 1j * eta) * np.eye(inp.dim)
        X = r["X"][k]
        res = np.linalg.norm(X @ A.T - B, axis=1) / np.linalg.norm(B, axis=1)
        # the FP64 residual that was tested against tol, up to its rounding and that of this product
        slack = 8.0 * inp.dim * 2.0 ** -53 * np.linalg.norm(np.abs(X) @ np.abs(A).T, axis=1) / np.linalg.norm(B, axis=1)
        assert np.all(res <= tol + slack)
    ctx.close()
