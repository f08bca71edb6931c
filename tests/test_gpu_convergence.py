"""Arnoldi steps of the FP32 basis with delayed re-orthogonalisation against those of the FP64 basis with two full
passes, at frequencies inside the 2h1p spectrum, where every cycle runs through its whole restart length (33 to 120
vectors, more than one sweep takes): wrong Hessenberg entries, or parts of the basis left out, cost steps."""
import numpy as np
import pytest

from gpu_util import inputs, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.mark.parametrize("o,v,np_,nw,restart,eta", [
    (7, 13, 20, 5, 100, 0.02), (7, 13, 3, 5, 64, 0.01), (9, 30, 3, 3, 100, 0.02), (12, 40, 2, 2, 120, 0.02),
    (9, 30, 30, 2, 33, 0.05)])
def test_steps_of_long_cycles(torch, o, v, np_, nw, restart, eta):
    from paper_1902_06016_gb300 import Context
    inp = inputs(o, v, 103)
    ws = np.linspace(-3.2, -2.0, nw)
    steps = {}
    for prec in ("fp64", "tf32", "bf16"):
        ctx = Context(inp, tol=1e-10, precision=prec, residual_precision="fp64", restart=restart)
        st = ctx.solve_full(ws, eta, list(range(np_)), want_A=False)["stats"]
        ctx.close()
        assert st.not_converged == 0
        steps[prec] = st.gmres_iters
    assert steps["fp64"] > 3 * restart
    # the inner action's rounding lets a cycle gain at most about three digits; that is more than these cycles gain, so
    # it may cost a cycle at the end and a few steps of the last one, but no more
    for prec, cycles in (("tf32", 1), ("bf16", 2)):
        assert steps[prec] <= 1.05 * steps["fp64"] + cycles * restart, steps
