"""Evaluation of a reduced model of order 64 in one batch of 2^21 columns: more rows of the products' right operand than
a grid of 32-row tiles has in its second dimension (65535). Any part of such a batch is what a short list of its
frequencies gives."""
import struct

import numpy as np
import pytest

import synth

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def test_order_64_at_131072_frequencies(torch, tmp_path):
    from paper_1902_06016_gb300 import Context
    inp = synth.make_inputs(6, 13, 46)
    orb, eta, nw = list(range(16)), 0.02, 131072
    ctx = Context(inp, tol=1e-9)
    ctx.mor_build(np.linspace(-1.4, -0.1, 4), eta, orb)
    assert ctx.mor_info()["m"] == 64
    ws = np.linspace(-1.5, 0.0, nw)
    G = torch.empty((nw, 16, 16), dtype=torch.complex128, device="cuda")
    r = ctx.mor_eval(ws, G=G, want_res=True)
    part = np.unique(np.concatenate([np.arange(0, nw, 4099), np.arange(nw - 40, nw)]))
    short = ctx.mor_eval(ws[part], want_res=True)
    path = str(tmp_path / "model.bin")
    ctx.mor_save(path)
    ctx.close()
    raw = open(path, "rb").read()
    D, m, npp, nq = struct.unpack_from("<7i", raw, 8)[2:6]
    ns, = struct.unpack_from("<i", raw, 44)
    pos = 48 + 8 * ns + 4 * npp + 4 * nq + 8 * npp + 2 * 16 * D * m
    H = np.frombuffer(raw, np.complex128, m * m, pos).reshape(m, m).T
    b = np.frombuffer(raw, np.complex128, m * npp, pos + 16 * m * m).reshape(npp, m).T
    c = np.frombuffer(raw, np.complex128, nq * m, pos + 16 * m * (m + npp)).reshape(m, nq).T
    # the solves of a frequency do not depend on the batch; the products differ by the rounding of m terms, each at most
    # 2^-53 (sums in FP64) or 2^-60 (digits) of |c_q| |y_p|
    for k, w in enumerate(ws[part]):
        y = np.linalg.solve(H + (w - 1j * eta) * np.eye(m), b)
        scale = np.linalg.norm(c, axis=1)[None, :] * np.linalg.norm(y, axis=0)[:, None]
        assert np.all(np.abs(G[int(part[k])].cpu().numpy() - short["G"][k]) <= 4 * m * 2.0 ** -53 * scale)
    # residuals relative to ||b_p||: the same rounding of sums whose terms are at most (|w| + ||H||) ||y_p||, about
    # 6 ||b_p|| / eta: 4 m 2^-53 6 / eta = 9e-12
    assert np.abs(r["maxres"][part] - short["maxres"]).max() <= 1e-11
