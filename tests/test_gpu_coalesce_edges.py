"""Photons on the edges of the coalescence's direction bins (GPU): the groups
are the oracle's, bit for bit, where a component is an exact fraction of the
dominant one and the last bit of its reciprocal decides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import DeviceSpecies

pytestmark = pytest.mark.gpu

KEYS = ("x", "y", "z", "ux", "uy", "uz", "w")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Q.qp_init_tables(W.LAMBDA_M, 0)
    yield c
    torch.cuda.synchronize()
    Q.qp_destroy(c)


@pytest.mark.parametrize("axis,fractions", [(0, (-0.75, 0.0)), (1, (-0.75, 0.25)),
                                            (2, (-1.0, -0.75)), (0, (-1.0, -1.0))])
def test_groups_on_bin_edges_are_the_oracles(ctx, axis, fractions):
    n = 1_000_003
    rng = np.random.default_rng(axis + 10 * int(4 * fractions[1] + 8))
    u = np.empty((3, n))
    # mantissas above 4/3, where a reciprocal's last bit reaches the product's,
    # all ones among them; one energy octave of each, so groups are large
    d = rng.uniform(1.34, 2.0, n) * 2.0 ** rng.integers(2, 5, n)
    d[:64] = np.ldexp(2.0 - 2.0 ** -52, rng.integers(1, 4, 64))
    u[axis] = d * rng.choice((-1.0, 1.0), n)
    u[(axis + 1) % 3], u[(axis + 2) % 3] = fractions[0] * d, fractions[1] * d
    arr = {"x": rng.uniform(0, 8, n), "y": rng.uniform(0, 8, n), "z": rng.uniform(0, 8, n),
           "ux": u[0], "uy": u[1], "uz": u[2], "w": rng.uniform(0.5, 2.0, n),
           "tau": rng.exponential(size=n)}
    box, cells = (0.0, 0.0, 0.0, 8.0, 8.0, 8.0), (1, 1, 1)
    g = DeviceSpecies(ctx, Q.QP_PHOTON, n, 3, track_chi=False)
    g.load(arr, n)
    o = O.Species.from_arrays(arr, n, 3)
    o.tau[:n] = arr["tau"]
    st = Q.qp_coalesce_photons(ctx, g.handle, Q.coalesce_params(box, cells, 1, 8, 3, seed=3, step=1))
    so = O.coalesce(o, O.coalesce_params(box, cells, 1, 8, 3, dims=3, seed=3, step=1))
    assert st["groups_merged"] == so["groups_merged"] and st["n_after"] == so["n_after"]
    h = g.host()
    for k in KEYS:
        np.testing.assert_array_equal(h[k], getattr(o, k)[:so["n_after"]], err_msg=k)
    Q.qp_destroy_species(ctx, g.handle)
