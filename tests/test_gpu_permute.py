"""Axis permutations of the operator build, dst = alpha P(src) + beta dst, in every order: axes that collapse, unit axes,
rows, tiles with ragged edges, short axes left to the element-wise form, and one axis."""
import ctypes as C
import itertools

import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


# (source dimensions): on both sides of the 32-long rows and tiles, of the 8-long tile edges and of the 2048 rows
@pytest.mark.parametrize("dims", [(1,), (77,), (1, 1, 1), (5, 1), (31, 33), (32, 64), (8, 7), (8, 8), (65, 1, 40), (2047, 33),
                                  (2048, 32), (3, 700, 33), (700, 3, 31), (9, 1, 34, 8), (33, 2, 7, 40), (4, 5, 6, 7),
                                  (2, 3, 1, 33, 9), (64, 3, 2, 1, 65), (2, 1, 3, 8, 1, 35), (3, 2, 4, 2, 5, 3)])
def test_every_order(torch, dims):
    from paper_1902_06016_gb300 import load
    f = load()["_ZN4gfcc7permuteEPKdPKiiS3_PdddP11CUstream_st"]   # gfcc::permute of csrc/tensor.cu
    f.restype = None
    f.argtypes = [C.c_void_p, C.POINTER(C.c_int), C.c_int, C.POINTER(C.c_int), C.c_void_p, C.c_double, C.c_double,
                  C.c_void_p]
    n = len(dims)
    g = torch.Generator(device="cuda").manual_seed(n)
    src = torch.randn(dims, dtype=torch.float64, device="cuda", generator=g)
    orders = list(itertools.permutations(range(n)))
    if len(orders) > 120:   # every seventh of the 720
        orders = orders[::7] + orders[-1:]
    for perm in orders:
        want = src.permute(perm).contiguous()
        for alpha, beta in ((1.0, 0.0), (-0.25, 0.0), (1.0, 1.0), (-1.5, 0.3)):
            old = torch.randn(want.shape, dtype=torch.float64, device="cuda", generator=g)
            # one spare element on each side shows a write outside; with beta = 0 the old values must not be read
            buf = torch.full((want.numel() + 2,), float("nan"), dtype=torch.float64, device="cuda")
            if beta != 0.0:
                buf[1:-1] = old.reshape(-1)
            torch.cuda.synchronize()
            f(src.data_ptr(), (C.c_int * n)(*dims), n, (C.c_int * n)(*perm), buf[1:].data_ptr(), alpha, beta, None)
            torch.cuda.synchronize()
            got = buf[1:-1].reshape(want.shape)
            assert torch.isnan(buf[0]) and torch.isnan(buf[-1])
            if beta == 0.0:
                assert torch.equal(got, alpha * want), (perm, alpha)
            else:   # two roundings of the two terms at most
                bound = 2.0 ** -52 * ((alpha * want).abs() + (beta * old).abs())
                assert torch.all((got - (alpha * want + beta * old)).abs() <= bound), (perm, alpha, beta)
