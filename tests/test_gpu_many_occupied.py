"""The operator build with more than 255 occupied spin-orbitals: their pairs (i, j) are more than a grid has blocks in its
second dimension."""
from types import SimpleNamespace

import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def test_256_occupied(torch):
    from paper_1902_06016_gb300 import Context, gfcc
    gfcc.release_cached_memory()
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 220 << 30:
        pytest.skip("needs 220 GB of device memory")
    o, v = 256, 1

    def zeros(*shape):
        return torch.zeros(shape, dtype=torch.float64, device="cuda")

    eps = torch.linspace(-1.5, 1.0, o + v, dtype=torch.float64, device="cuda")
    inp = SimpleNamespace(o=o, v=v, eps=eps, oooo=zeros(o, o, o, o), ooov=zeros(o, o, o, v), oovv=zeros(o, o, v, v),
                          ovov=zeros(o, v, o, v), ovvv=zeros(o, v, v, v), t1=zeros(o, v) + 0.01, t2=zeros(o, o, v, v),
                          l1=zeros(o, v), l2=zeros(o, o, v, v))
    ctx = Context(inp)
    inp.oooo = None
    X = torch.zeros((1, ctx.D), dtype=torch.complex128, device="cuda")
    idx = [0, 5, o - 1, o, o + 7, ctx.D - 1]
    X[0, idx] = 1.0
    Y = ctx.sigma(X)[0]
    ctx.close()
    gfcc.release_cached_memory()
    # without integrals M is diagonal: -eps_i, and eps_a - eps_i - eps_j for the pairs (0, 1), (1, 4), (o - 2, o - 1)
    e = eps.cpu()
    want = [-e[0], -e[5], -e[o - 1], e[o] - e[0] - e[1], e[o] - e[1] - e[4], e[o] - e[o - 2] - e[o - 1]]
    assert torch.allclose(Y[idx].real.cpu(), torch.stack([torch.as_tensor(x) for x in want]), rtol=1e-14, atol=0.0)
    Y[idx] = 0.0
    assert torch.count_nonzero(Y).item() == 0
