"""The FP32 sine and cosine of gc_f32x2.cuh on the CPU: the polynomials with the header's own
literals, replayed with correctly rounded multiply-adds, stay within the 1.55 ulp that its
comment states, over the whole range that the fast reduction takes and next to every multiple
of pi/2 in it, where the reduction cancels."""
import os
import re
import sys

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_06706_gb300", "csrc")
f4 = np.float32


def _replay():
    sys.path.insert(0, CSRC)
    try:
        import sincos_coeffs
    finally:
        sys.path.remove(CSRC)
    text = open(os.path.join(CSRC, "gc_f32x2.cuh")).read()
    body = text[text.index("void sincos2("):]
    lit = [f4(v) for v in re.findall(r"p2_bcast\((-?[0-9.e+-]+)f\)", body)]
    inv, magic, magic2, m0, m1, m2, s2, s1, s0, c2, c1, c0, half, one = lit
    assert inv == f4(2 / np.pi) and magic == magic2 == f4(1.5 * 2**23) and half == f4(-0.5) and one == f4(1.0)
    parts = [-m0, -m1, -m2]
    assert parts == sincos_coeffs.split_pi_2()
    most = float(re.search(r"kSincosMax = ([0-9.]+)f;", text).group(1))
    stated = float(re.search(r"At most ([0-9.]+) ulp", text).group(1))
    return (lambda z: sincos_coeffs.sincos(z, (s0, s1, s2), (c0, c1, c2), parts)), most, stated


def test_sine_and_cosine_within_the_stated_bound():
    sincos, most, stated = _replay()
    rng = np.random.default_rng(2)
    z = [rng.uniform(-lim, lim, 1_000_000) for lim in (1e-3, 1.0, 30.0, 400.0, most)]
    near = (np.arange(-int(most / (np.pi / 2)), int(most / (np.pi / 2)) + 1) * (np.pi / 2)).astype(f4)
    for away in range(4):  # the nearest floats on either side
        z += [near.copy(), -near]
        near = np.nextafter(near, f4(np.inf), dtype=f4)
    z = np.concatenate([v.astype(f4) for v in z])
    z = z[(z != 0) & (np.abs(z) <= most)]
    for got, want in zip(sincos(z), (np.sin(z.astype(np.float64)), np.cos(z.astype(np.float64)))):
        ulp = np.abs(got - want) / np.spacing(np.abs(want).astype(f4))
        assert ulp.max() <= stated, (ulp.max(), z[ulp.argmax()])
