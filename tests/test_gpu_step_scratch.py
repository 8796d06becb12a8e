"""The append scratch of qp_step where long tiles' larger one is not there
(GPU only): a step captured in a graph whose warm-up was of another field kind
keeps to short tiles and gives the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation, stream_handle

pytestmark = pytest.mark.gpu


def _simulation():
    # capacities above the line of long tiles (4.4e6 slots on 152 SMs), few
    # particles
    w = W.plane_wave_collision(n=3000)
    w["capacity"] = {"electron": 3000, "positron": 0, "photon": 6_000_000}
    return Simulation(w, precision="mixed", track_chi=False)


def _state(sim):
    torch.cuda.synchronize()
    d = sim.diagnostics("electron")
    out = {nm: sp.host() for nm, sp in sim.species.items() if sp.cap}
    sim.close()
    return out, d.status, d.n_emit


def test_a_captured_step_needs_no_larger_scratch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sim = _simulation()
    sim.run(24)
    want, status, n_emit = _state(sim)
    assert n_emit > 0

    sim = _simulation()
    # a warm-up on a grid without field, counts at 0: the species' chains, the
    # short tiles' scratch
    grid = [torch.zeros((8, 8), device="cuda") for _ in range(6)]
    warm = Q.qp_step_params.from_buffer_copy(sim.params)
    warm.field.kind, warm.field.nx, warm.field.ny = Q.QP_FIELD_YEE2D, 8, 8
    warm.field.dx = warm.field.dy = 1.0
    for k, c in enumerate(grid):
        warm.field.yee[k] = c.data_ptr()
    warm.step, warm.n_steps = 0, 1
    counts = sim.counts.clone()
    sim.counts.zero_()
    Q.qp_step(sim.ctx, warm, stream_handle(None))
    sim.counts.copy_(counts)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        sim.run(24, stream)
    graph.replay()
    got, after, n = _state(sim)
    assert after == status and n == n_emit
    for name in want:
        for k in want[name]:
            np.testing.assert_array_equal(got[name][k], want[name][k], err_msg=name + k)
