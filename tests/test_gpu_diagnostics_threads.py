"""qp_diagnostics from two host threads (GPU only): each call returns its own
species' figures, on one stream and on two."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import DeviceSpecies, stream_handle

pytestmark = pytest.mark.gpu

CALLS = 4000


@pytest.mark.parametrize("streams", [1, 2])
def test_threads_get_their_own_figures(streams):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = Q.qp_init_tables(W.LAMBDA_M, 0)
    species = []
    for k, n in enumerate((300, 70_000)):
        rng = np.random.default_rng(k)
        arr = {c: rng.normal(size=n) for c in ("x", "y", "z", "ux", "uy", "uz")}
        arr.update(w=np.full(n, 1.0 + k), tau=np.ones(n))
        s = DeviceSpecies(ctx, Q.QP_ELECTRON, n, 3, track_chi=False)
        s.load(arr, n)
        species.append(s)
    torch.cuda.synchronize()
    made = [torch.cuda.Stream() for _ in range(streams)]
    handles = [stream_handle(made[k % streams]) for k in range(2)]

    def figures(k):
        d = Q.qp_diagnostics(ctx, species[k].handle, handles[k])
        return d.n_live, d.n_alive, d.weight, d.energy, tuple(d.hist)

    want = [figures(k) for k in range(2)]
    assert [w[0] for w in want] == [300, 70_000]
    wrong = [0, 0]

    def work(k):
        for _ in range(CALLS):
            wrong[k] += figures(k) != want[k]

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    Q.qp_destroy(ctx)
    assert wrong == [0, 0]
