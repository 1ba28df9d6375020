"""Points on the polar axis or within the smallest floats of it: flagged as on the axis and as
nothing else, and advanced as a point a little further out at the same longitude is."""
import numpy as np
import pytest

from paper_2403_06706_gb300 import synth

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")

WIND = synth.WindSpec(32, 16, 32)
AXIS = 2  # GC_FLAG_AXIS
# directions whose products with the scales below have subnormal floats, zeros, or both
DIRS = np.array([[1, 2], [2, -1], [-3, 0.5], [-1, -1], [0, 1], [1, 0], [-1, 0], [0, -2], [300, 1], [-1, 300]])


def _advance(prec, scale):
    n = len(DIRS)
    with gcpush.Context(precision=prec, seed=2, no_scatter=True) as c:
        c.field_load(synth.wind_grid(WIND, dtype=np.float64 if prec == 0 else np.float32), WIND.r_min_au, WIND.r_max_au)
        c.inject([synth.EnsembleSpec(n, r0_au=0.5, lat_deg=30.0, r_in_au=0.2, r_out_au=1.9)])
        s = c.get_state()
        s["z"][:] = np.hypot(np.hypot(s["x"], s["y"]), s["z"]) * np.where(np.arange(n) % 2, -1.0, 1.0)
        s["x"][:], s["y"][:] = (DIRS * scale).T
        s["F0"][:] = s["F1"][:] = 0.0  # the predictor point is the particle's own
        c.set_state(s)
        with pytest.raises(gcpush.GcError):
            c.advance(0.5, 1)
        return c.get_state()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("scale", [1e-40, 3e-39, 1e-45])
def test_next_to_the_axis(prec, scale):
    """At 1e-20 m, where no float is subnormal, the radius that the axis is cut off at is in
    force as well (1e-15 m): the same field is read there and the two advance alike, to the
    rounding of their longitude (at 1e-45 m floats are whole multiples of 1.4e-45: only the
    flags are compared)."""
    a, b = _advance(prec, scale), _advance(prec, 1e-20)
    assert (a["flags"] == AXIS).all() and (b["flags"] == AXIS).all()
    if scale > 1e-44:
        for k in ("z", "u", "mub", "F0", "vpar"):
            assert np.allclose(a[k], b[k], rtol=1e-5 if prec else 1e-9, atol=1e-5 * np.abs(b[k]).max()), k
    assert all(np.isfinite(v).all() for v in a.values())
