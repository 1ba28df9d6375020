"""The FP64 push of few particles (four lanes each) against one thread per particle: both take
the same roundings, so states, tallies and counters have to be equal bit for bit. A single
particle, the edges of a warp's eight, the largest population it takes and the first that it
does not; every E_par mode, collision form and drift option; events, replays of a graph, and
particles on the polar axis and beyond the grid."""
import numpy as np
import pytest

from paper_2403_06706_gb300 import synth

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")

WIND = synth.WindSpec(32, 16, 32, eps=0.1, n_modes=4, phi1_v=200.0)


def _run(n, ideal, opts, outside, **shape):
    ens = [synth.EnsembleSpec(n - n // 3, lam_au=0.02, r_in_au=0.9, r_out_au=1.1)]
    if n // 3:
        ens.append(synth.EnsembleSpec(n // 3, r0_au=0.5, lat_deg=-40.0, lam_au=0.5, r_in_au=0.2, r_out_au=0.52))
    graph = shape.pop("graph", False)
    with gcpush.Context(precision=0, seed=5, **opts) as c:
        c.field_load(synth.wind_grid(WIND, dtype=np.float64), WIND.r_min_au, WIND.r_max_au, ideal=ideal)
        c.inject(ens)
        if outside:
            s = c.get_state()
            s["x"][:2] = s["y"][:2] = 0.0
            s["x"][2:4] *= 100.0
            c.set_state(s)
        c.tally_arm(cadence=7, n_mu=8, n_E=8, n_r=16)
        c.set_launch(steps_per_launch=40, **shape)
        c.set_graph(graph)
        for dt, steps in ((0.5, 1), (0.5, 90), (0.5, 90), (0.3, 5)):
            try:
                c.advance(dt, steps)
            except gcpush.GcError:
                assert outside  # particles flagged on the axis or off the grid
        return c.get_state(), c.tally_read(), c.stats()


@pytest.mark.parametrize("n,ideal,opts,shape", [
    (1, True, {}, {}),
    (7, 2, {}, {}),
    (8, False, {}, {}),
    (9, True, {"wind_u": 4e5}, {"graph": True}),
    (33, True, {"collision_form": 1}, {}),
    (1000, 2, {"drift_mask": 1}, {}),
    (1000, False, {"drift_mask": 1, "no_scatter": True}, {}),
    (1000, True, {"no_rebirth": True}, {}),
    (152 * 48, False, {}, {}),
    (152 * 48, 2, {"collision_form": 1}, {"graph": True}),
    (152 * 48 + 1, True, {}, {}),
])
def test_four_lanes_equal_one_thread_per_particle(n, ideal, opts, shape):
    outside = n == 1000
    a, ta, sa = _run(n, ideal, opts, outside, **dict(shape))
    b, tb, sb = _run(n, ideal, opts, outside, grid_waves=0, block=32)
    for k in a:
        assert np.array_equal(a[k], b[k], equal_nan=a[k].dtype.kind == "f"), k
    for k in ta:
        assert np.array_equal(ta[k], tb[k]), k
    for k in ("collisions", "rebirths", "flags_or", "particle_steps"):
        assert sa[k] == sb[k], k
