"""Grid nodes that are no ordinary numbers (GPU): an infinite or NaN node
shows in the particles beside it and nowhere else; denormal nodes count."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation

pytestmark = pytest.mark.gpu

DT = 0.05
NEAR, FAR = (3.25, 3.75), (10.5, 10.5)  # electrons at rest, cells of size 1


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Q.qp_init_tables(W.LAMBDA_M, 0)
    yield c
    torch.cuda.synchronize()
    Q.qp_destroy(c)


def step(ctx, comps, precision):
    pos = np.array([NEAR, FAR])
    zero = np.zeros(2)
    w = {"dims": 2, "capacity": {"electron": 2, "positron": 1, "photon": 16},
         "field": {"kind": "yee2d", "dx": 1.0, "dy": 1.0, "comps": comps},
         "params": {"dt": DT, "seed": 1, "chi_th": 0.0, "pairs": True},
         "electrons": {"x": pos[:, 0], "y": pos[:, 1], "ux": zero, "uy": zero, "uz": zero,
                       "tau": np.full(2, 5.0), "w": np.ones(2)}}
    sim = Simulation(w, precision=precision, ctx=ctx, init_tau=False)
    sim.run(1)
    torch.cuda.synchronize()
    return sim.species["electron"].host()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_a_node_that_is_not_finite_shows(ctx, precision, value):
    comps = [np.zeros((16, 16), np.float32) for _ in range(6)]
    comps[1][3, 3] = value  # E_y at (3, 3.5): a corner of NEAR's cell
    got = step(ctx, comps, precision)
    assert not np.isfinite(got["uy"][0])
    assert [got[k][1] for k in ("x", "y", "ux", "uy", "uz", "tau")] == [*FAR, 0.0, 0.0, 0.0, 5.0]


def test_denormal_nodes_count(ctx):
    comps = [np.zeros((16, 16), np.float32) for _ in range(6)]
    comps[1][:] = np.float32(1e-40)
    got = step(ctx, comps, "fp64")
    # u_y = -dt E_y: interpolation and push round a dozen times, 2^-53 each
    np.testing.assert_allclose(got["uy"], -DT * float(np.float32(1e-40)), rtol=1e-14)
