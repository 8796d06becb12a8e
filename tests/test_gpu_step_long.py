"""Launches of several steps on long tiles, and launches whose kind of tile
changes between two steps (GPU only): n steps in one call must equal n calls of
one step, bit for bit, with all counters.  Where both lepton species emit, long
tiles append what short ones do, the electrons' photons before the positrons'."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from tests.test_gpu_step_tiles import COUNTS, _beam, _step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Q.qp_init_tables(W.LAMBDA_M, 0)
    yield c
    torch.cuda.synchronize()
    Q.qp_destroy(c)


def _line(precision):
    """Sub-tiles of 32 slots from which a launch takes long tiles: 128 for each
    of the 7 (FP64: 4) resident blocks of an SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 128 * sms * (7 if precision == "mixed" else 4)


def _subs(counts):
    return sum((int(n) + 31) // 32 for n in counts)


def _compare(ctx, precision, blocks, steps):
    w = W.beam_collision(n=1, buffer=1)
    one, c1 = _step(ctx, w, precision, blocks, (0, 0, 0), steps=1, calls=steps)
    many, c2 = _step(ctx, w, precision, blocks, (0, 0, 0), steps=steps, calls=1)
    assert np.array_equal(c1, c2)
    for a, b in zip(one, many):
        assert torch.equal(a, b)
    return [b.shape[1] for b in many]


@pytest.mark.parametrize("precision,n_e,n_p,n_g", [("mixed", 3_000_001, 40_007, 1_500_003),
                                                   ("mixed", 900_001, 31, 3_800_003),
                                                   ("fp64", 1_700_003, 20_001, 900_001)])
def test_several_steps_on_long_tiles(ctx, precision, n_e, n_p, n_g):
    g = torch.Generator(device="cuda").manual_seed(7)
    blocks = [_beam(n_e, 2000.0, 6000.0, g), _beam(n_p, 300.0, 6000.0, g),
              _beam(n_g, 1.0, 3000.0, g)]
    assert _subs((n_e, n_p, n_g)) >= _line(precision)
    _compare(ctx, precision, blocks, 4)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("short_by", [1, 3000])
def test_a_launch_that_crosses_to_long_tiles(ctx, precision, short_by):
    # the electrons' photons take the launch over the line after one step
    # (short_by 1) or a few
    g = torch.Generator(device="cuda").manual_seed(8)
    line = _line(precision)
    n_p, n_g = 1001, 60_007
    n_e = 32 * (line - short_by - _subs((0, n_p, n_g)))
    blocks = [_beam(n_e, 2000.0, 6000.0, g), _beam(n_p, 300.0, 6000.0, g),
              _beam(n_g, 1.0, 3000.0, g)]
    assert _subs((n_e, n_p, n_g)) == line - short_by
    after = _compare(ctx, precision, blocks, 6)
    assert _subs(after) >= line


@pytest.mark.parametrize("n_e,n_p", [(4_500_000, 33), (2_300_001, 2_200_003)])
def test_both_lepton_species_append_in_order(ctx, n_e, n_p):
    g = torch.Generator(device="cuda").manual_seed(9)
    w = W.beam_collision(n=1, buffer=1)
    blocks = [_beam(n_e, 2000.0, 6000.0, g), _beam(n_p, 2000.0, 6000.0, g), _beam(0, 1.0, 2.0, g)]
    whole, counts = _step(ctx, w, "mixed", blocks, (0, 0, 0))
    cuts = [np.linspace(0, b.shape[1], 5).astype(int) for b in blocks]
    by = [[], []]  # photons of the electrons, of the positrons
    photon = COUNTS.index("n_photon")
    for k in range(4):
        own = [b[:, c[k]:c[k + 1]] for b, c in zip(blocks, cuts)]
        rows, cnt = _step(ctx, w, "mixed", own, [int(c[k]) for c in cuts])
        m = int(cnt[0, photon])
        by[0].append(rows[2][:, :m])
        by[1].append(rows[2][:, m:])
    made = torch.cat([torch.cat(b, dim=1) for b in by], dim=1)
    assert made.shape[1] == counts[:2, photon].sum() > 0
    assert torch.equal(whole[2], made)
