"""qp_diagnostics against host sums (GPU only): sizes around a tile of 256
slots and around 512 blocks of one tile, energies on both sides of the
spectrum's bin edges closer than FP32 resolves, decayed photons left out,
weights that are all in one bin.

Tolerances: the device sums at most n/131072 + 1 values a thread, then trees
of fewer than 64 adds, and each value has fewer than 8 roundings, so a sum is
within 80 x 2^-53 = 9e-15 of the exact one relative to the sum of the absolute
values; the host sum (fsum) is exact.  1e-14 is asserted.  The bins must agree
exactly: energies stand 1e-9 off an edge, log10 is good to 1e-15."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import DeviceSpecies

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Q.qp_init_tables(W.LAMBDA_M, 0)
    yield c
    torch.cuda.synchronize()
    Q.qp_destroy(c)


@pytest.mark.parametrize("kind", [Q.QP_PHOTON, Q.QP_ELECTRON])
@pytest.mark.parametrize("n,one_bin", [(0, False), (1, False), (255, False), (256, True),
                                       (257, False), (131_072, False), (131_073, True),
                                       (300_001, False)])
def test_sums_and_spectrum(ctx, kind, n, one_bin):
    rng = np.random.default_rng(n + kind)
    photon = kind == Q.QP_PHOTON
    edges = 10.0 ** (-1.0 + 6.0 / 64.0 * np.arange(64))
    g = edges[rng.integers(11, 64, n)] * np.where(rng.uniform(size=n) < 0.5, 1 - 1e-9, 1 + 1e-9)
    far = rng.uniform(size=n) < 0.5
    g = np.where(far, 10.0 ** rng.uniform(0.01, 5.3, n), g)  # some above the last bin
    if photon:
        g = np.where(rng.uniform(size=n) < 0.1, 10.0 ** rng.uniform(-3.0, 0.0, n), g)
    if one_bin:
        g = np.full(n, 50.0)
    p = g if photon else np.sqrt((g - 1.0) * (g + 1.0))
    axis = rng.integers(0, 3, n)
    sign = np.where(rng.uniform(size=n) < 0.5, -1.0, 1.0)
    u = np.zeros((3, n))
    u[axis, np.arange(n)] = sign * p
    arr = {"x": np.zeros(n), "y": np.zeros(n), "z": np.zeros(n), "ux": u[0], "uy": u[1],
           "uz": u[2], "w": rng.uniform(0.5, 2.0, n),
           "tau": np.where(rng.uniform(size=n) < 0.2, -1.0, 1.0)}
    sp = DeviceSpecies(ctx, kind, n + 7, 3)
    sp.load(arr, n)
    d = Q.qp_diagnostics(ctx, sp.handle)
    assert d.n_live == n
    live = arr["tau"] >= 0 if photon else np.ones(n, bool)
    w, u = arr["w"][live], u[:, live]
    e = np.sqrt((u * u).sum(0) + (0.0 if photon else 1.0))
    assert d.n_alive == int(live.sum())
    for got, v in ((d.weight, w), (d.energy, w * e), (d.px, w * u[0]), (d.py, w * u[1]),
                   (d.pz, w * u[2])):
        assert abs(got - math.fsum(v)) <= 1e-14 * math.fsum(np.abs(v))
    b = np.clip((np.log10(e) + 1.0) * (64.0 / 6.0), 0, 63).astype(int)
    for k in range(64):
        v = w[b == k]
        assert abs(d.hist[k] - math.fsum(v)) <= 1e-14 * math.fsum(v), k
    again = Q.qp_diagnostics(ctx, sp.handle)
    assert list(again.hist) == list(d.hist) and again.energy == d.energy and again.px == d.px
    Q.qp_destroy_species(ctx, sp.handle)
