"""Contractions of the operator build whose rows mix magnitudes: the elements that decide a result may be far smaller than
others of their row that meet zeros. FP64 sums keep all 53 bits of them."""
import numpy as np
import pytest

import synth
from oracle import hbar
from oracle import sigma as sg

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

SMALL = 2.0 ** -40


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def mixed_inputs(o, v, seed):
    """t_j0^0b of order one where every <m0||e0> it meets is zero, all other doubles of order 2^-40; no singles, and of
    the integrals only <mn||ef>, of order one."""
    rng = np.random.default_rng(seed)

    def anti(x):
        x = x - x.transpose(1, 0, 2, 3)
        return x - x.transpose(0, 1, 3, 2)

    inp = synth.make_inputs(o, v, seed)
    for name in ("oooo", "ooov", "ovov", "ovvv", "t1", "l1", "l2"):
        setattr(inp, name, np.zeros_like(getattr(inp, name)))
    t2 = SMALL * anti(rng.uniform(0.5, 1.0, (o, o, v, v)) * rng.choice([-1.0, 1.0], (o, o, v, v)))
    oovv = anti(rng.uniform(0.5, 1.0, (o, o, v, v)) * rng.choice([-1.0, 1.0], (o, o, v, v)))
    big = rng.uniform(0.5, 1.0, (o, v))
    for j in range(1, o):
        for b in range(1, v):
            t2[j, 0, 0, b] = t2[0, j, b, 0] = big[j, b]
            t2[0, j, 0, b] = t2[j, 0, b, 0] = -big[j, b]
            oovv[j, 0, b, 0] = oovv[0, j, 0, b] = oovv[0, j, b, 0] = oovv[j, 0, 0, b] = 0.0
    inp.t2, inp.oovv = t2, oovv
    return inp


# the ring contraction t_jn^fb <mn||ef> has (o v)^3 multiply-adds: 3.3e7, 8.7e7, 2.0e8
@pytest.mark.parametrize("o,v", [(8, 40), (13, 34), (14, 42)])
def test_small_elements_beside_large_ones(torch, o, v):
    from paper_1902_06016_gb300 import Context
    inp = mixed_inputs(o, v, 7)
    hb = hbar.build(inp)
    ctx = Context(inp)
    pair = lambda i, j: j * (j - 1) // 2 + i  # noqa: E731
    idx = lambda i, j, a: o + pair(i, j) * v + a  # noqa: E731
    # columns r_kl^e and rows (ij)^a with one index of the pairs in common, a != e, no index 0: one element of the ring
    # block W_mbej = -t_jn^fb <mn||ef> each, with terms of order 2^-40 only
    k, l, e = 1, 2, 3
    X = np.zeros((1, ctx.D), dtype=complex)
    X[0, idx(k, l, e)] = 1.0
    rows = [(idx(k, j, a)) for j in range(3, o) for a in range(1, v) if a != e]
    y = ctx.sigma(X)[0, rows].real
    ref = sg.sigma(hb, X.real)[0, rows]
    ctx.close()
    assert np.abs(ref).max() <= 64 * o * v * SMALL   # nothing of order one is in them
    # K = o v terms of order 2^-40 in FP64: K rounding errors of at most 2^-53 of the sum of their magnitudes (each
    # amplitude and integral below 4), in the contraction and in the few sums after it
    K = o * v
    assert np.abs(y - ref).max() <= 8.0 * K * 2.0 ** -53 * K * 16.0 * SMALL


def test_projection_of_columns_that_mix_magnitudes(torch, tmp_path):
    """Hhat = S^H Z of a reduced model (2.1e7 complex multiply-adds): the columns are unit vectors whose entries go from
    order one down to 10^-6."""
    import struct

    from paper_1902_06016_gb300 import Context
    inp = synth.make_inputs(12, 60, 31)
    ctx = Context(inp, tol=1e-9, precision="tf32")
    ctx.mor_build(np.linspace(-1.2, -0.2, 6), 0.02, list(range(12)))
    path = str(tmp_path / "model.bin")
    ctx.mor_save(path)
    ctx.close()
    raw = open(path, "rb").read()
    D, m, npp, nq = struct.unpack_from("<7i", raw, 8)[2:6]
    ns, = struct.unpack_from("<i", raw, 44)
    pos = 48 + 8 * ns + 4 * npp + 4 * nq + 8 * npp
    S, Z = (np.frombuffer(raw, np.complex128, D * m, pos + 16 * D * m * k).reshape(D, m).T for k in (0, 1))
    H = np.frombuffer(raw, np.complex128, m * m, pos + 32 * D * m).reshape(m, m).T
    assert m * m * D >= 1.6e7 and np.abs(S).min() < 2.0 ** -16 * np.abs(S).max()
    ref = np.conj(S) @ Z.T
    # sums in FP64 (here) lose at most 2 D 2^-53 of the sum of magnitudes; digits keep an element to 2^-62 of its
    # column's largest (here with the other factor's largest, for each of 4 D real terms and both factors)
    cols = lambda X: np.maximum(np.abs(X.real), np.abs(X.imag)).max(axis=1)  # noqa: E731
    bound = 2 * D * 2.0 ** -53 * (np.abs(S) @ np.abs(Z).T) + 16 * D * 2.0 ** -62 * np.outer(cols(S), cols(Z))
    assert np.all(np.abs(H - ref) <= bound)
