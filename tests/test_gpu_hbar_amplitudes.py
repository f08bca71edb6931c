"""The operator build with doubles t_ij^ab = t_ji^ba that are not antisymmetric in i, j or in a, b alone: its expressions
are evaluated with the array as given, as the oracle evaluates them."""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import ea, hbar
from oracle import sigma as sg

from gpu_util import inputs, need_gpu, random_vectors, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.mark.parametrize("sector", ["ip", "ea"])
@pytest.mark.parametrize("o,v,seed", [(2, 1, 9), (2, 2, 9), (3, 5, 11), (5, 4, 12), (7, 13, 103), (4, 24, 13), (3, 37, 14)])
def test_sigma_with_any_doubles(torch, sector, o, v, seed):
    from paper_1902_06016_gb300 import Context
    if sector == "ea" and v < 2:
        pytest.skip("the attachment space needs two virtuals")
    inp = synth.random_amplitudes(inputs(o, v, seed), seed)
    rng = np.random.default_rng(seed)
    t2 = 0.1 * rng.standard_normal(inp.t2.shape)
    inp = dataclasses.replace(inp, t2=t2 + t2.transpose(1, 0, 3, 2))
    hb = ea.build(inp) if sector == "ea" else hbar.build(inp)
    ctx = Context(inp, sector=sector)
    X = random_vectors(ctx.D, 3, seed)
    # FP64 sums of at most o v v terms of order one throughout, as elsewhere in these tests
    assert rel_err(ctx.sigma(X), sg.sigma(hb, X)) <= 1e-12
    ctx.close()
