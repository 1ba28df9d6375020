"""The push of few particles beside the network's evaluation (one launch, tiles of 16 particles)
against the rounds that larger populations take. A second ensemble lifts the same particles (same
ids, streams and sites) over the limit; the first one's state and tallies then have to agree:
integers exactly, the rest to 1e-13 (both run the same FP32 arithmetic; mu_B is kept between
rounds as the 53-bit value it was injected with and here as the FP32 push's pair of floats,
48 bits). Sizes at the edges of tiles, of one tile per SM, and of the limit; a stretch of steps
cut into launches; a free path short enough for events in every tile."""
import numpy as np
import pytest

from paper_2403_06706_gb300 import synth

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")

WIND = synth.WindSpec(32, 16, 32)
LIMIT = 2 * 16 * 152


def _network():
    """A field of nearly constant direction falling as 1 / r^2, with a tenth of the seeded
    network's structure on it."""
    p = synth.siren_init(7).copy()
    p[198400:200448] *= 0.1
    p[200448:] = [0.8, 0.5, 0.3, 0.05, -0.1, 0.08, 1.0, 0.0]
    return p


def _run(n, extra, steps, per_launch):
    ens = [synth.EnsembleSpec(n, lam_au=0.004, r_out_au=0.5, scatter_law=1),
           synth.EnsembleSpec(extra, lam_au=0.5, r_out_au=2.0)][:2 if extra else 1]
    with gcpush.Context(seed=11, wind_u=4.0e5) as c:
        c.field_load(synth.wind_grid(WIND, dtype=np.float32), WIND.r_min_au, WIND.r_max_au)
        c.siren_set(_network(), omega0=30.0, r_max_au=WIND.r_max_au, B_scale=WIND.B1, E_scale=WIND.B1 * WIND.u_sw)
        c.field_select(gcpush.FIELD_SIREN)
        c.inject(ens)
        c.tally_arm(cadence=4, n_mu=8, n_E=8, n_r=16)
        c.set_launch(steps_per_launch=per_launch)
        c.advance(0.5, steps)
        c.advance(0.5, 3)
        st = {k: v[..., :n] for k, v in c.get_state().items()}
        ta = {k: v[0] for k, v in c.tally_read().items() if k != "n_seen"}
        return st, ta, c.stats()


@pytest.mark.parametrize("n,steps,per_launch", [(1, 40, 2000), (17, 40, 7), (152 * 16 + 1, 30, 2000),
                                                (LIMIT - 3, 25, 2000), (LIMIT, 25, 10)])
def test_small_population_equals_rounds(n, steps, per_launch):
    a, ta, sa = _run(n, 0, steps, per_launch)
    b, tb, sb = _run(n, LIMIT + 1, steps, per_launch)
    assert sa["kernel_launches"] < 40 + 2 * steps // min(per_launch, steps) and sb["kernel_launches"] > 4 * steps
    for k in gcpush.U32_STATE:
        assert np.array_equal(a[k], b[k]), k
    for k in gcpush.F64_STATE + ("F0", "F1"):
        scale = np.abs(b[k]).max() + 1e-300
        assert np.abs(a[k] - b[k]).max() <= 1e-13 * scale, k
    for k in ta:
        assert np.array_equal(ta[k], tb[k]), k
    if n > 1000:
        assert sa["collisions"] > n // 4 and sa["rebirths"] > 0
