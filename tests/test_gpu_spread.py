"""The push's default launch (one block per SM; the last, partial round spread over all SMs)
against one thread per particle: every particle is advanced once, whatever its place, so
states and tallies have to be equal bit for bit. A single particle, a ragged group, just below
and above one and two rounds of the FP32, time-dependent and FP64 kernels, small blocks, and
graph replay over several launches (of the same steps in both runs: a launch boundary passes
position and gamma v_par through doubles, which is exact for the pair of floats a value is
kept in except while it passes through zero)."""
import numpy as np
import pytest

from paper_2403_06706_gb300 import synth

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")

WIND = synth.WindSpec(32, 16, 32, eps=0.1, n_modes=4)


def _run(prec, nodes, n, mode, **shape):
    r_out = synth.r_out_default(WIND)
    ens = [synth.EnsembleSpec(n // 3, lam_au=0.02, r_out_au=r_out, r_in_au=0.25),
           synth.EnsembleSpec(n - n // 3, r0_au=0.5, lat_deg=-40.0, lam_au=0.5, r_out_au=0.52)]
    graph = shape.pop("graph", False)
    with gcpush.Context(precision=prec, seed=5) as c:
        c.field_load(nodes, WIND.r_min_au, WIND.r_max_au)
        if mode == "time":
            c.field_load_next(nodes * nodes.dtype.type(1.1), 0.0, 60.0)
        c.inject(ens)
        c.tally_arm(cadence=3, n_mu=8, n_E=8, n_r=16)
        c.set_launch(**shape)
        c.set_graph(graph)
        c.advance(0.5, 7)
        c.advance(0.5, 7)
        return c.get_state(), c.tally_read(), c.stats()


@pytest.mark.parametrize("prec,n,mode,shape", [
    (1, 1, "steady", {}),
    (1, 4097, "steady", {}),
    (1, 152 * 512 - 1, "steady", {}),
    (1, 152 * 512 + 129, "steady", {"steps_per_launch": 3, "graph": True}),
    (1, 2 * 152 * 512 + 152 * 128 + 33, "steady", {"block": 128}),
    (1, 60_001, "steady", {"block": 64}),
    (1, 152 * 384 + 385, "time", {}),
    (0, 4096, "steady", {}),
    (0, 152 * 256 + 31, "steady", {"block": 96}),
    (0, 2 * 152 * 256 + 4000, "steady", {}),
])
def test_spread_round_equals_one_thread_per_particle(prec, n, mode, shape):
    nodes = synth.wind_grid(WIND, dtype=np.float64 if prec == 0 else np.float32)
    a, ta, sa = _run(prec, nodes, n, mode, **dict(shape))
    b, tb, sb = _run(prec, nodes, n, mode, grid_waves=0, block=32, steps_per_launch=shape.get("steps_per_launch", 0))
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    for k in ta:
        assert np.array_equal(ta[k], tb[k]), k
    for k in ("collisions", "rebirths", "flags_or", "particle_steps"):
        assert sa[k] == sb[k], k
