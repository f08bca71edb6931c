"""The shifted Hessenberg solves of the reduced-model evaluation against dense solves of the same reduced
matrices (read back from a saved model), at the edges of their 32-row tiles and right-hand-side groups."""
import struct

import numpy as np
import pytest

import synth

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def torch():
    return need_gpu()


def read_model(path):
    """(Hhat [m, m], bhat [m, np], chat [nq, m]) of a saved model."""
    raw = open(path, "rb").read()
    o, v, D, m, npp, nq, qn = struct.unpack_from("<7i", raw, 8)
    pos = 8 + 28 + 8
    ns, = struct.unpack_from("<i", raw, pos)
    pos += 4 + 8 * ns + 4 * npp + 4 * nq + 8 * npp + 2 * 16 * D * m   # frequencies, orbitals, norms, S, Z
    out = []
    for cols, rows in ((m, m), (npp, m), (m, nq)):
        a = np.frombuffer(raw, dtype=np.complex128, count=rows * cols, offset=pos)
        pos += 16 * rows * cols
        out.append(a.reshape(cols, rows).T)
    return out


# (o, v, orbitals, seeds): orders on both sides of one and two tiles; groups of 8 to 48 right-hand sides with
# and without padding, more than one group
@pytest.mark.parametrize("o,v,norb,ns", [(5, 11, 1, 3), (5, 11, 1, 31), (6, 13, 1, 32), (6, 13, 1, 33), (6, 13, 3, 21),
                                         (6, 13, 8, 8), (6, 13, 9, 4), (6, 14, 17, 4), (8, 18, 26, 3), (10, 24, 33, 2),
                                         (12, 32, 42, 2), (12, 40, 51, 2)])
def test_eval_matches_dense_reduced_solves(tmp_path, o, v, norb, ns):
    from paper_1902_06016_gb300 import Context
    inp = synth.make_inputs(o, v, 40 + o)
    eta = 0.02
    ctx = Context(inp, tol=1e-9)
    ctx.mor_build(np.linspace(-1.4, -0.1, ns), eta, list(range(norb)))
    path = str(tmp_path / "model.bin")
    ctx.mor_save(path)
    ws = np.linspace(-1.5, 0.0, 37)
    G = ctx.mor_eval(ws)["G"]
    ctx.close()
    H, b, c = read_model(path)
    m = len(H)
    ref = np.empty_like(G)
    cond = 0.0
    for k, w in enumerate(ws):
        A = H + (w - 1j * eta) * np.eye(m)
        cond = max(cond, np.linalg.cond(A))
        ref[k] = (c @ np.linalg.solve(A, b)).T
    err = np.linalg.norm(G - ref) / np.linalg.norm(ref)
    # U is kept to 2^-48 and the substitution adds about m rounding errors of that size; the Hessenberg form and
    # the final products are FP64-accurate
    assert err <= 8.0 * (m + 32) * 2.0 ** -48 * cond, (m, err, cond)


def test_eval_rows_longer_than_shared_memory():
    """A subspace that spans the whole space (order above 2560, so that the elimination's rows do not fit in
    shared memory): the reduced model is then the full system."""
    from paper_1902_06016_gb300 import Context
    inp = synth.make_inputs(14, 30, 5)
    ctx = Context(inp, tol=1e-10, precision="fp64_tc")
    orb = list(range(44))
    ctx.mor_build_krylov(64, 0.05, orb)
    m = ctx.mor_info()["m"]
    assert m + len(orb) > 2560
    ws = np.array([-0.7, -0.3])
    G = ctx.mor_eval(ws)["G"]
    ref = ctx.solve_full(ws, 0.05, orb, want_A=False)["G"]
    ctx.close()
    assert np.linalg.norm(G - ref) <= 1e-7 * np.linalg.norm(ref)
