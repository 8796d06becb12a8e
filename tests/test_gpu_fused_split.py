"""Fused windows whose tiles are split into warps of fewer lanes (GPU only):
electrons and positrons of ragged numbers, from one lepton (one lane a warp)
over each halving of the lanes to whole tiles, against single steps, bit for
bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation

pytestmark = pytest.mark.gpu


def _run(n, n_p, precision, fused):
    w = W.plane_wave_collision(n=n + n_p, n_steps=12)
    src = {k: np.asarray(v) for k, v in w["electrons"].items()}
    w["electrons"] = {k: v[:n] for k, v in src.items()}
    w["capacity"] = {"electron": n + 3, "positron": n_p + 1, "photon": 8 * (n + n_p) + 64}
    w["params"] = dict(w["params"], pairs=False, step=1000)  # inside the wave
    sim = Simulation(w, precision=precision)
    if n_p:
        pos = {k: v[n:].copy() for k, v in src.items()}
        pos["tau"] = np.full(n_p, 0.05)
        sim.species["positron"].load(pos, n_p)
    if fused:
        sim.run_fused(12, 12)
    else:
        sim.run(12)
    torch.cuda.synchronize()
    out = {nm: sp.host() for nm, sp in sim.species.items()}
    emitted = sum(sim.diagnostics(nm).n_emit for nm in ("electron", "positron"))
    sim.close()
    return out, emitted


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,n_p", [(1, 0), (1, 1), (33, 31), (700, 0), (1200, 45), (2431, 1),
                                   (4865, 100), (9700, 700), (19_500, 33), (38_000, 2000)])
def test_split_tiles_give_the_bits_of_single_steps(n, n_p, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a, ea = _run(n, n_p, precision, True)
    b, eb = _run(n, n_p, precision, False)
    assert ea == eb and (ea > 0 or n < 100)
    for nm in b:
        for k, v in b[nm].items():
            if v is not None:
                np.testing.assert_array_equal(a[nm][k], v, err_msg=f"{nm} {k}")
