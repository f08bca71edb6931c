"""The FP64 sigma on both sides of the dimension up to which it runs on M as a dense matrix: forward and transposed,
against the oracle's matrix, on host arrays, on device buffers in place, with a leading dimension and onto itself."""
import numpy as np
import pytest

import synth
from oracle import hbar
from oracle import sigma as sg

from gpu_util import need_gpu, random_vectors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.mark.parametrize("o,v,nvec", [(2, 1, 1), (3, 4, 5), (4, 8, 700), (6, 16, 33), (6, 17, 33)])
@pytest.mark.parametrize("transpose", [False, True])
def test_sigma_across_the_dense_limit(torch, o, v, nvec, transpose):
    from paper_1902_06016_gb300 import Context
    inp = synth.make_inputs(o, v, 70 + o)
    M = sg.dense_matrix(hbar.build(inp))
    ctx = Context(inp)
    X = random_vectors(ctx.D, nvec, 3)
    ref = X @ M if transpose else X @ M.T
    # FP64 throughout: D rounding errors of 2^-53 of the sum of magnitudes, in M's elements and in the product
    bound = 4.0 * (ctx.D + o * v) * 2.0 ** -53 * (np.abs(X) @ np.abs(M if transpose else M.T)).max()
    assert np.abs(ctx.sigma(X, transpose=transpose) - ref).max() <= bound
    pad = torch.full((nvec, ctx.D + 3), 7.0, dtype=torch.complex128, device="cuda")
    pad[:, :ctx.D] = torch.from_numpy(X).cuda()
    out = torch.full_like(pad, 9.0)
    ctx.sigma(pad, transpose=transpose, out=out)
    assert np.abs(out[:, :ctx.D].cpu().numpy() - ref).max() <= bound
    ctx.sigma(pad, transpose=transpose, out=pad)   # onto its own input
    assert np.abs(pad[:, :ctx.D].cpu().numpy() - ref).max() <= bound
    ctx.close()
