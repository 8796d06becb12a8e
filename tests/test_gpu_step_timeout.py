"""A launch of several steps that gives up on one of its blocks (GPU only): the
waits are bounded, the status says so, and the control block is left as it was
found, so that later steps are right.  No step is made to fail: the self-test
launches the ends of steps alone, one block late."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Q.qp_init_tables(W.LAMBDA_M, 0)
    yield c
    torch.cuda.synchronize()
    Q.qp_destroy(c)


def _run(ctx, precision):
    sim = Simulation(W.plane_wave_collision(n=3000), precision=precision, ctx=ctx)
    sim.run(61)  # several steps a launch
    torch.cuda.synchronize()
    out = {nm: sp.host() for nm, sp in sim.species.items()}
    d = sim.diagnostics("electron")
    return out, d.status, d.n_emit


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_time_out_between_steps_leaves_the_context_usable(ctx, precision):
    want, status, n_emit = _run(ctx, precision)
    assert status >= 0 and n_emit > 0
    for _ in range(2):
        assert Q.qp_selftest_step_timeout(ctx, 2000) == Q.QP_ERR_TIMEOUT
        got, after, n = _run(ctx, precision)
        assert after == status and n == n_emit
        for name in want:
            for k in want[name]:
                np.testing.assert_array_equal(got[name][k], want[name][k], err_msg=name + k)
