"""A batch's append scratch follows its problems (GPU only): small ones need
little, and a graph captured before a large one was set steps it with the same
bits as qp_step."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation, stream_handle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Q.qp_init_tables(W.LAMBDA_M, 0)
    yield c
    torch.cuda.synchronize()
    Q.qp_destroy(c)


def _simulation(ctx, n, cap):
    w = W.plane_wave_collision(n=1)
    w["capacity"] = {"electron": n, "positron": 0, "photon": cap}
    sim = Simulation(w, precision="mixed", ctx=ctx, track_chi=False, load=False)
    g = torch.Generator(device="cuda").manual_seed(n)
    t = sim.species["electron"].t
    for nm in ("x", "uy", "uz"):
        t[nm][:n] = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    t["ux"][:n] = -2000.0 * (1.0 + 0.1 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    t["tau"][:n] = -torch.log1p(-torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    t["w"][:n] = 1.0
    sim.species["electron"].n_live.fill_(n)
    return sim


def test_small_problems_take_little_memory(ctx):
    Q.qp_batch_destroy(Q.qp_batch_create(ctx, 4, Q.QP_MIXED, Q.QP_FIELD_PLANE))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    batch = Q.qp_batch_create(ctx, 4, Q.QP_MIXED, Q.QP_FIELD_PLANE)
    used = before - torch.cuda.mem_get_info()[0]
    Q.qp_batch_destroy(batch)
    # short tiles: 17 words a slot, 4 tiles of 128 slots a block, 7 blocks an SM
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    short = 8 * 17 * 4 * 128 * 7 * sms
    assert used <= short + (32 << 20), (used, short)


def test_a_graph_from_before_a_large_problem_steps_it(ctx):
    steps, n = 3, 4_700_000  # above the line of long tiles
    want = _simulation(ctx, n, n // 2)
    want.run(steps)
    torch.cuda.synchronize()
    ref = {nm: sp.host() for nm, sp in want.species.items() if sp.cap}
    del want

    batch = Q.qp_batch_create(ctx, 2, Q.QP_MIXED, Q.QP_FIELD_PLANE)
    stream = torch.cuda.Stream()
    sh = stream_handle(stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        Q.qp_batch_step(batch, 1, sh)
    scratch = []
    sims = [_simulation(ctx, 1000, 4000), _simulation(ctx, n, n // 2)]
    torch.cuda.synchronize()
    for k, sim in enumerate(sims):
        p = Q.qp_step_params.from_buffer_copy(sim.params)
        p.step, p.n_steps = 0, steps
        words = Q.qp_batch_scratch_words(ctx, p)
        scratch.append(torch.zeros(words, dtype=torch.int64, device="cuda"))
        torch.cuda.synchronize()
        Q.qp_batch_set(batch, k, p, scratch[-1].data_ptr(), words, sh)
        if k == 0:  # a launch with the small problem alone
            with torch.cuda.stream(stream):
                graph.replay()
    with torch.cuda.stream(stream):
        for _ in range(steps):
            graph.replay()
    torch.cuda.synchronize()
    got = {nm: sp.host() for nm, sp in sims[1].species.items() if sp.cap}
    Q.qp_batch_destroy(batch)
    assert len(got["photon"]["x"]) > 100_000
    for name in ref:
        for k in ref[name]:
            np.testing.assert_array_equal(got[name][k], ref[name][k], err_msg=name + k)
