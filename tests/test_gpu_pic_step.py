"""qp_pic_step against the calls that make up a cycle (GPU only).

Weights of 0 give no current, so no float atomics: several cycles must then
agree bit for bit.  With weights, one cycle: fields B and particles bit for
bit (B does not see the cycle's current), the current within the rounding of
its float sums in any order.  A node gets at most m terms, so two orders
differ by at most 2 m 2^-24 of the sum of the terms' magnitudes; with m < 500
(4 particles a cell, 4 cells, both species, and the foil's random crowding)
that is below 6e-5, taken of the sum of magnitudes at the fullest node, which
is at least the largest current and below 20 times it for currents of
alternating sign: 1.2e-3 of the largest current is asserted, and E within dt
of that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation

pytestmark = pytest.mark.gpu


def _run(nx, ny, positrons, weight, cycles, whole):
    w = W.laser_on_foil(nx=nx, ny=ny, ppc=4, foil_cells=8, seed=5)
    w["field"]["pic"] = {"a0": 200.0, "w0": W.length(3 * W.LAMBDA_M),
                         "tau_fwhm": W.duration(30e-15),
                         "x_focus": (nx // 2) * w["field"]["dx"], "t_focus": 0.0,
                         "y_axis": 0.5 * ny * w["field"]["dy"]}
    n = len(w["electrons"]["x"])
    w["electrons"]["w"] = np.asarray(w["electrons"]["w"]) * weight
    w["capacity"] = {"electron": n + 1000, "positron": n if positrons else 0, "photon": 4 * n}
    if not positrons:
        w["params"]["pairs"] = False
    sim = Simulation(w, precision="mixed")
    if positrons:
        src = {k: np.asarray(v)[: n // 3].copy() for k, v in w["electrons"].items()}
        src["ux"] = src["ux"] + 3.0
        src["tau"] = np.full(n // 3, 0.5)
        sim.species["positron"].load(src, n // 3)
    sim.J.fill_(7.0)  # what an earlier cycle left
    if whole:
        sim.run(cycles)
    else:
        j = [sim.J[k].data_ptr() for k in range(3)]
        dt, ctx = sim.params.dt, sim.ctx
        for k in range(cycles):
            Q.qp_yee_advance_b(ctx, sim.field, 0.5 * dt)
            sim.params.step, sim.params.n_steps = sim.step_index + k, 1
            Q.qp_step(ctx, sim.params)
            torch.cuda.synchronize()
            sim.J.zero_()
            torch.cuda.synchronize()
            for name in ("electron", "positron"):
                if sim.species[name].cap:
                    Q.qp_deposit_current(ctx, sim.species[name].handle, sim.field, *j, dt)
            Q.qp_yee_advance_b(ctx, sim.field, 0.5 * dt)
            Q.qp_yee_advance_e(ctx, sim.field, *j, dt)
    torch.cuda.synchronize()
    out = {"dt": sim.params.dt, "J": sim.J.cpu().numpy(),
           "grid": [c.cpu().numpy() for c in sim._keep],
           "species": {nm: sp.host() for nm, sp in sim.species.items() if sp.cap}}
    sim.close()
    return out


@pytest.mark.parametrize("nx,ny", [(256, 40), (253, 31)])
@pytest.mark.parametrize("positrons", [True, False])
@pytest.mark.parametrize("weight,cycles", [(0.0, 3), (1.0, 1)])
def test_cycles_match_their_calls(nx, ny, positrons, weight, cycles):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a = _run(nx, ny, positrons, weight, cycles, True)
    b = _run(nx, ny, positrons, weight, cycles, False)
    for nm in a["species"]:
        for k in a["species"][nm]:
            np.testing.assert_array_equal(a["species"][nm][k], b["species"][nm][k], err_msg=nm + k)
    exact = range(6) if weight == 0.0 else range(3, 6)
    for k in exact:
        np.testing.assert_array_equal(a["grid"][k], b["grid"][k], err_msg=str(k))
    if weight == 0.0:
        assert not a["J"].any() and not b["J"].any()
        return
    top = np.abs(b["J"]).max()
    assert top > 0.0
    assert np.abs(a["J"] - b["J"]).max() <= 1.2e-3 * top
    for k in range(3):
        scale = np.abs(b["grid"][k]).max()
        assert np.abs(a["grid"][k] - b["grid"][k]).max() <= 1.2e-3 * top * a["dt"] + 2.0 ** -23 * scale
