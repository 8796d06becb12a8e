"""The step kernel's two kinds of tile and its launches of several steps (GPU
only).  A population large enough for long tiles is stepped whole and as parts
small enough for short ones, every particle with its own id: the primaries
and what they append must agree bit for bit, and the parts' event counts
add up.  n steps in one call must equal n calls of one step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.sim import Simulation

pytestmark = pytest.mark.gpu

ROWS = ("x", "y", "z", "ux", "uy", "uz", "tau", "w")
COUNTS = ("n_emit", "n_photon", "n_subthreshold", "n_pair", "n_saturated", "n_clamped",
          "n_continuous")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Q.qp_init_tables(W.LAMBDA_M, 0)
    yield c
    torch.cuda.synchronize()
    Q.qp_destroy(c)


def _beam(n, u_lo, u_hi, g):
    """n particles around the pulse peak, moving mostly along -x."""
    r = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    h = lambda: torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    x, y, z = W.length(2e-6) * r(3, n)
    u = u_lo * (u_hi / u_lo) ** h()
    ty, tz = 0.05 * r(2, n)
    norm = torch.sqrt(1.0 + ty * ty + tz * tz)
    return torch.stack([x, y, z, -u / norm, u * ty / norm, u * tz / norm,
                        -torch.log1p(-h()), 0.5 + h()])


def _step(ctx, w, precision, parts, first, steps=1, calls=1):
    """Steps the given blocks (electron, positron, photon); first: the ids of
    their first slots.  Returns the species' live rows and the counters."""
    names = ("electron", "positron", "photon")
    n = [p.shape[1] for p in parts]
    w = dict(w, capacity={"electron": n[0] + n[2] + 64, "positron": n[1] + n[2] + 64,
                          "photon": n[2] + 4 * (n[0] + n[1]) + 64})
    sim = Simulation(w, precision=precision, ctx=ctx, track_chi=False, load=False,
                     ids={k: (f, 0, 0) for k, f in zip(names, first)})
    for k, p in zip(names, parts):
        sp = sim.species[k]
        sp.block[:, :p.shape[1]].copy_(p)
        sp.n_live.fill_(p.shape[1])
        Q.qp_reset_counters(ctx, sp.handle)
    sim.step_index = 990
    for _ in range(calls):
        sim.run(steps)
    live = sim.live_counts()
    rows = [sim.species[k].block[:, :live[k]].clone() for k in names]
    diag = [sim.diagnostics(k) for k in names]
    assert all(d.status >= 0 and d.n_photon_drop == 0 and d.n_pair_drop == 0 for d in diag)
    for sp in sim.species.values():
        Q.qp_destroy_species(ctx, sp.handle)
    return rows, np.array([[getattr(d, c) for c in COUNTS] for d in diag])


# slots past the line at which long tiles begin (4.36e6 slots on 152 SMs, mixed
# path; 2.49e6 FP64), with ragged last sub-tiles, parts and tiles
@pytest.mark.parametrize("precision,n_e,n_p,n_g", [
    ("mixed", 3_000_001, 0, 1_500_003),
    ("mixed", 0, 2_600_031, 1_900_097),
    ("mixed", 255, 1, 4_600_000),
    ("mixed", 4_500_000, 33, 0),
    ("fp64", 1_700_003, 0, 900_001),
    ("fp64", 31, 2_600_001, 257),
])
def test_long_tiles_equal_short_ones(ctx, precision, n_e, n_p, n_g):
    g = torch.Generator(device="cuda").manual_seed(5)
    w = W.beam_collision(n=1, buffer=1)
    blocks = [_beam(n_e, 2000.0, 6000.0, g), _beam(n_p, 300.0, 6000.0, g),
              _beam(n_g, 1.0, 3000.0, g)]
    blocks[2][6][::7] = -1.0  # decayed ones among the photons
    whole, counts = _step(ctx, w, precision, blocks, (0, 0, 0))
    cuts = [np.linspace(0, b.shape[1], 5).astype(int) for b in blocks]
    parts, total = [], 0
    for k in range(4):
        own = [b[:, c[k]:c[k + 1]] for b, c in zip(blocks, cuts)]
        rows, cnt = _step(ctx, w, precision, own, [int(c[k]) for c in cuts])
        parts.append((own, rows))
        total = total + cnt
    assert np.array_equal(counts, total)
    assert counts[:2, 0].sum() > 0 or n_e + n_p < 1000
    for s, n in enumerate((n_e, n_p, n_g)):
        prim = torch.cat([rows[s][:, :own[s].shape[1]] for own, rows in parts], dim=1)
        made = torch.cat([rows[s][:, own[s].shape[1]:] for own, rows in parts], dim=1)
        assert torch.equal(whole[s][:, :n], prim), s
        # appended in the order of their parents (one lepton species emits)
        if s != 2 or n_e == 0 or n_p < 100:
            got = whole[s][:, n:]
            assert got.shape == made.shape
            # a few parents of the other lepton species come last in the whole
            m = got.shape[1] if s != 2 or n_p == 0 or n_e == 0 else 0
            assert torch.equal(got[:, :m], made[:, :m]), s


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n_e,n_p,n_g", [(1, 0, 0), (130, 33, 1000), (40_000, 20_001, 90_000)])
def test_steps_in_one_call_equal_single_steps(ctx, precision, n_e, n_p, n_g):
    g = torch.Generator(device="cuda").manual_seed(6)
    w = W.beam_collision(n=1, buffer=1)
    blocks = [_beam(n_e, 2000.0, 6000.0, g), _beam(n_p, 300.0, 6000.0, g),
              _beam(n_g, 1.0, 3000.0, g)]
    one, c1 = _step(ctx, w, precision, blocks, (0, 0, 0), steps=1, calls=11)
    many, c2 = _step(ctx, w, precision, blocks, (0, 0, 0), steps=11, calls=1)
    assert np.array_equal(c1, c2)
    for a, b in zip(one, many):
        assert torch.equal(a, b)
