"""A tally cadence near 2^31 steps: the sample after one taken lies beyond an int, and the step
loops have to end all the same, with that one sample. The FP32 push, FP64 with four lanes and
with one per particle, and the rounds of the split-step push."""
import numpy as np
import pytest

from paper_2403_06706_gb300 import synth

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")

WIND = synth.WindSpec(32, 16, 32)


@pytest.mark.parametrize("prec,n,source", [(1, 100, 0), (0, 100, 0), (0, 152 * 48 + 1, 0), (1, 100, 2)])
@pytest.mark.parametrize("cadence", [2**31 - 1, 2**31 - 12])
def test_one_sample_and_no_other(prec, n, source, cadence):
    with gcpush.Context(precision=prec, seed=1) as c:
        c.field_load(synth.wind_grid(WIND, dtype=np.float64 if prec == 0 else np.float32), WIND.r_min_au, WIND.r_max_au)
        c.inject([synth.EnsembleSpec(n, lam_au=0.1, r_out_au=1.9)])
        if source:
            c.field_select(gcpush.FIELD_GRID_SAMPLED)
        c.tally_arm(cadence=cadence, n_mu=4, n_E=4, n_r=4)
        c.set_clock(0.0, cadence - 6)
        for _ in range(2):
            c.advance(0.5, 20)
        assert int(c.tally_read()["n_seen"][0]) == n
        assert c.stats()["step"] == cadence + 34
