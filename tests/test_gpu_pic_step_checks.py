"""qp_pic_step rejects what qp_step rejects before it touches the grid, the
current or the particles (GPU only)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.laser_on_foil(nx=64, ny=40, ppc=2, foil_cells=4, seed=5)
    w["field"]["pic"] = {"a0": 200.0, "w0": W.length(3 * W.LAMBDA_M),
                         "tau_fwhm": W.duration(30e-15), "x_focus": 32 * w["field"]["dx"],
                         "t_focus": 0.0, "y_axis": 20 * w["field"]["dy"]}
    s = Simulation(w, precision="mixed")
    yield s
    s.close()


@pytest.mark.parametrize("name,value", [("precision", 7), ("max_emissions", 0),
                                        ("chi_threshold", -1.0), ("photon_min_gamma", -1.0),
                                        ("dt", 0.0), ("dt", -0.1), ("step", -1), ("n_steps", -1),
                                        ("electron", "photon"), ("photon", "positron"),
                                        ("photon", 99)])
def test_a_rejected_call_changes_nothing(sim, name, value):
    sim.J.fill_(7.0)
    torch.cuda.synchronize()
    grid = [c.cpu().numpy() for c in sim._keep]
    rows = sim.species["electron"].block.cpu().numpy()
    params = Q.qp_step_params.from_buffer_copy(sim.params)
    params.n_steps = 2
    setattr(params, name, sim.species[value].handle if isinstance(value, str) else value)
    j = [sim.J[k].data_ptr() for k in range(3)]
    with pytest.raises(Q.QPError):
        Q.qp_pic_step(sim.ctx, params, *j)
    torch.cuda.synchronize()
    for k in range(6):
        np.testing.assert_array_equal(sim._keep[k].cpu().numpy(), grid[k], err_msg=str(k))
    assert bool((sim.J == 7.0).all())
    np.testing.assert_array_equal(sim.species["electron"].block.cpu().numpy(), rows)
