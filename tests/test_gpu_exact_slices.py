"""The exact-slice sigma at the limits of its integer arithmetic: digits of the largest magnitude in both operands
(every 256-product accumulation then reaches 2^24, the bound of exact FP32 sums), several K splits, column
chunks and ragged tiles, against the FP64 CUDA-core sigma."""
from types import SimpleNamespace

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def constant_inputs(o, v, x):
    """<ia||jb> = -x and <ij||kl> = x, everything else zero (no physics: the sigma is linear in whatever it is
    given): the ring block is x everywhere, the oooo block x everywhere, and no other product is left."""
    full = lambda y, *s: np.full(s, y)  # noqa: E731
    return SimpleNamespace(o=o, v=v, eps=np.zeros(o + v), oooo=full(x, o, o, o, o), ooov=full(0.0, o, o, o, v),
                           oovv=full(0.0, o, o, v, v), ovov=full(-x, o, v, o, v), ovvv=full(0.0, o, v, v, v),
                           t1=np.zeros((o, v)), t2=full(0.0, o, o, v, v), l1=np.zeros((o, v)), l2=full(0.0, o, o, v, v))


@pytest.mark.parametrize("o,v,nvec,x", [(3, 5, 1, 0.999999), (6, 60, 3, 0.999999), (4, 131, 2, 1.0 - 2.0 ** -44),
                                        (13, 37, 65, 0.50001), (20, 400, 40, 0.999999)])
def test_exact_sigma_with_extreme_digits(torch, o, v, nvec, x):
    from paper_1902_06016_gb300 import Context
    ctx = Context(constant_inputs(o, v, x))
    P = o * (o - 1) // 2
    rng = np.random.default_rng(o * v)
    X = np.full((nvec, ctx.D), x * (1.0 + 1.0j))
    X[1:] *= rng.choice([-1.0, 1.0], (nvec - 1, ctx.D))   # the first vector: every term of a product alike
    ref = ctx.sigma(X, precision="fp64")
    got = ctx.sigma(X, precision="fp64_tc")
    ctx.close()
    # |x| < 1: an element is kept to 2^-45, the dropped digit pairs weigh at most 4 2^-45 (and their tail as much
    # again at most), so a product's term is exact to 12 2^-45; two ring products of (o - 1) v terms, one oooo
    # product of P terms and the rounding of the FP64 sums (2^-53 of the same magnitude a step)
    terms = 2 * (o - 1) * v + P
    assert np.abs(got - ref).max() <= terms * (12.0 * 2.0 ** -45 + terms * 2.0 ** -53)
