"""The split-step push of many particles with many events in a call: the rounds after the steps'
own run on lists of most of the population, and have to evaluate a point in about the time that
the rounds over all particles take, with the same results."""
import numpy as np
import pytest

from paper_2403_06706_gb300 import synth
from test_gpu_neural_small import WIND, _network

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")


def _context(counts, lam):
    c = gcpush.Context(seed=11)
    c.field_load(synth.wind_grid(WIND, dtype=np.float32), WIND.r_min_au, WIND.r_max_au)
    c.siren_set(_network(), omega0=30.0, r_max_au=WIND.r_max_au, B_scale=WIND.B1, E_scale=WIND.B1 * WIND.u_sw)
    c.field_select(gcpush.FIELD_SIREN)
    c.inject([synth.EnsembleSpec(n, lam_au=k, r_out_au=2.0) for n, k in zip(counts, lam)])
    c.tally_arm(cadence=2, n_mu=8, n_E=8, n_r=16)
    return c


def test_long_lists_take_the_large_tiles():
    """200 000 particles, 8 steps of 3e-4 AU at most (0.5 s at 0.5 c, 81 keV) with a free path
    of 2e-4 AU: half of all evaluations or so are on lists. With the tiles of the rounds over
    all particles (21 waves) a point costs the same there but for the last, short lists, some
    20 rounds of one wave each: 5 % of the time. Tiles of 16 points take several times as long
    a point. The line is drawn at 1.25."""
    per = {}
    for lam in (100.0, 2e-4):
        with _context([200_000], (lam,)) as c:
            c.advance(0.5, 8)
            best = 1e9
            for _ in range(3):
                a = c.stats()
                c.advance(0.5, 8)
                b = c.stats()
                best = min(best, (b["field_ms"] - a["field_ms"]) / (b["field_evals"] - a["field_evals"]))
            events = b["collisions"] + b["rebirths"] - a["collisions"] - a["rebirths"]
            per[lam] = (best * 1e6, events)
    print(per)  # ns per evaluated point, events of the last call
    assert per[2e-4][1] > 2 * 200_000
    assert per[2e-4][0] < 1.25 * per[100.0][0]


@pytest.mark.parametrize("n", [1, 300, 2400])
def test_lists_of_any_length_give_the_same_results(n):
    """The same particles beside 30 000 others without events (lists of at most n, tiles of 16
    points) and beside 30 000 with many (lists of most of them, tiles of 64, then of 16 as they
    shorten): a point's sums are the same in either tile, so states and tallies are equal bit
    for bit."""
    out = []
    for lam in (100.0, 5e-4):
        with _context([n, 30_000], (5e-4, lam)) as c:
            c.advance(0.5, 20)
            s = c.get_state()
            out.append(({k: v[..., :n] for k, v in s.items()}, {k: v[0] for k, v in c.tally_read().items() if k != "n_seen"},
                        int(s["ncoll"][n:].sum())))
    (a, ta, ca), (b, tb, cb) = out
    assert ca < 3000 and cb > 30_000 and (n < 100 or int(a["ncoll"].sum()) > n)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    for k in ta:
        assert np.array_equal(ta[k], tb[k]), k
