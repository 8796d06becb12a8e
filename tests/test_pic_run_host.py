"""Simulation.run on a PIC workload keeps its step index with the grid when a
cycle fails (host only: the library's call is replaced)."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300.sim import Simulation


def test_step_index_follows_the_cycles_taken(monkeypatch):
    taken = []

    def pic_step(ctx, params, jx, jy, jz, stream=None):
        for k in range(params.n_steps):
            if len(taken) == 3:
                raise Q.QPError("qp_pic_step", Q.QP_ERR_CUDA)
            taken.append(params.step + k)
        return 0

    monkeypatch.setattr(Q, "qp_pic_step", pic_step)
    sim = Simulation.__new__(Simulation)
    sim.ctx, sim.pulse, sim.pic_pulse, sim.step_index = None, None, object(), 7
    sim.J = torch.zeros((3, 2, 2))
    sim.params = Q.qp_step_params()
    stream = types.SimpleNamespace(cuda_stream=0)
    with pytest.raises(Q.QPError):
        sim.run(5, stream)
    assert taken == [7, 8, 9] and sim.step_index == 10
