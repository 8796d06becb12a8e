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


def _check(ctx, rng, d, axis, fractions):
    n = len(d)
    u = np.empty((3, n))
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


@pytest.mark.parametrize("axis,fractions", [(0, (-0.75, 0.0)), (1, (-0.75, 0.25)),
                                            (2, (-1.0, -0.75)), (0, (-1.0, -1.0))])
def test_groups_on_bin_edges_are_the_oracles(ctx, axis, fractions):
    n = 1_000_003
    rng = np.random.default_rng(axis + 10 * int(4 * fractions[1] + 8))
    # mantissas above 4/3, where a reciprocal's last bit reaches the product's,
    # all ones among them; one energy octave of each, so groups are large
    d = rng.uniform(1.34, 2.0, n) * 2.0 ** rng.integers(2, 5, n)
    d[:64] = np.ldexp(2.0 - 2.0 ** -52, rng.integers(1, 4, 64))
    _check(ctx, rng, d, axis, fractions)


# Mantissas whose reciprocals lie within 2^-25 of the last place of a tie (found
# by a search over 1.2e9 odd ones), and one whose product with a reciprocal that
# is one unit high passes 1.
NEAR_TIES = (
    "0x1.5ce00aae5b6c5p+0 0x1.66d684ffcb221p+0 0x1.678c946716b27p+0 0x1.69a0601f27ae7p+0 "
    "0x1.6a9e3e996322fp+0 0x1.6f65947e87e8bp+0 0x1.70beb0fbc9157p+0 0x1.722547cf1e317p+0 "
    "0x1.7239f51244989p+0 0x1.741932d48aa03p+0 0x1.7514d722f2199p+0 0x1.77fee98584025p+0 "
    "0x1.78fd16f84d1c7p+0 0x1.79559b8a4851fp+0 0x1.7be64684640d3p+0 0x1.7e63dd212d8fdp+0 "
    "0x1.7f9060accb149p+0 0x1.815a88bc9ec6fp+0 0x1.822143f134079p+0 0x1.847b2f155fd73p+0 "
    "0x1.84fa0787932c3p+0 0x1.868cc89708907p+0 0x1.870d85d72be55p+0 0x1.8e35e11961ba7p+0 "
    "0x1.8ff4c32fe961fp+0 0x1.909147e2016d9p+0 0x1.94d503b30cd43p+0 0x1.95932200144edp+0 "
    "0x1.9a9a84edba171p+0 0x1.a0d4d04a2861dp+0 0x1.a3d8dd9495917p+0 0x1.a4551f230dcbbp+0 "
    "0x1.a7a103fb29743p+0 0x1.a829a52423c5bp+0 0x1.ae4f3a37c74e3p+0 0x1.b0084473cb80fp+0 "
    "0x1.b19354fd378a3p+0 0x1.b2edfd1f83637p+0 0x1.b57bbe325604dp+0 0x1.b8b3c007578c1p+0 "
    "0x1.b909d96d7e74dp+0 0x1.ba78007dd91d1p+0 0x1.bc5690541f929p+0 0x1.be85063399173p+0 "
    "0x1.c09bb84b109c1p+0 0x1.c0bf939531c33p+0 0x1.c1a060a04a583p+0 0x1.c1beb7534476bp+0 "
    "0x1.c37c043a78aadp+0 0x1.c47b839619351p+0 0x1.c6a56dd9ed1ebp+0 0x1.c76265428f07bp+0 "
    "0x1.c87a362b20939p+0 0x1.c8f8727e4646fp+0 0x1.ca9fa21cf33d1p+0 0x1.cce9f69b8b151p+0 "
    "0x1.d05c66248766dp+0 0x1.d093801259d63p+0 0x1.d1772366f29f7p+0 0x1.d25196220b60fp+0 "
    "0x1.d2e5eacf348b3p+0 0x1.d380f8b6fb88bp+0 0x1.d519aa428cee5p+0 0x1.d93d7b6973d41p+0 "
    "0x1.d947a102a3c37p+0 0x1.dd339897cdb4fp+0 0x1.df057e1485089p+0 0x1.e21c616edffcfp+0 "
    "0x1.e355e1761c575p+0 0x1.e49e64a6ae7e7p+0 0x1.e75080bdefe7bp+0 0x1.e94cd3fd75627p+0 "
    "0x1.fffffafccdd98p+0").split()


@pytest.mark.parametrize("axis,fractions", [(0, (-0.75, 0.0)), (1, (-0.75, -0.5)),
                                            (2, (-1.0, -0.75))])
def test_reciprocals_nearest_to_a_tie(ctx, axis, fractions):
    rng = np.random.default_rng(axis)
    m = np.array([float.fromhex(t) for t in NEAR_TIES])
    n = 40 * len(m)
    d = np.repeat(m, 40)[rng.permutation(n)] * 2.0 ** rng.integers(2, 5, n)
    _check(ctx, rng, d, axis, fractions)
