"""Coefficients of the FP32 sine and cosine of gc_f32x2.cuh.

On |r| <= pi/4: sin r = r + r^3 S(r^2) with S of degree 2, cos r = 1 - r^2/2 + r^4 C(r^2) with C
of degree 2, each fitted in FP64 by Lawson's iteratively reweighted least squares (minimal
maximum error of the result), plus the three-part split of pi/2 for Cody and Waite's reduction
r = z - q pi/2 (Software Manual for the Elementary Functions, 1980). Prints the literals and
the errors of the FP32 evaluation, replayed with correctly rounded multiply-adds. (Reducing to
pi/2 with one more term each would drop the exchange of sine and cosine, at an rms error of
2.1e-8 and 2.9e-8 instead of 1.7e-8.)"""
import numpy as np

f4 = np.float32


def fit(f, basis, deg, n=4001):
    x = np.cos(np.linspace(0.0, np.pi, n)) * (np.pi / 4)
    x = x[x > 1e-4]
    A = np.stack([basis(x) * x ** (2 * k) for k in range(deg + 1)], 1)
    w = np.ones_like(x)
    for _ in range(200):
        c = np.linalg.lstsq(A * np.sqrt(w)[:, None], f(x) * np.sqrt(w), rcond=None)[0]
        e = np.abs(A @ c - f(x))
        w *= e + 1e-30
        w /= w.sum()
    return c.astype(f4), e.max()


def split_pi_2():
    p, parts = np.longdouble("1.57079632679489661923132169163975144"), []
    for _ in range(3):
        parts.append(f4(p))
        p -= np.longdouble(parts[-1])
    return parts


def fma(a, b, c):
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(f4)


def sincos(z, s, c, parts):
    t = fma(z, f4(2 / np.pi), f4(12582912.0))
    q, k, r = (t - f4(12582912.0)).astype(f4), t.view(np.int32), z
    for p in parts:
        r = fma(q, -p, r)
    r2 = (r * r).astype(f4)
    ps, pc = fma(fma(s[2], r2, s[1]), r2, s[0]), fma(fma(c[2], r2, c[1]), r2, c[0])
    sn, cs = fma((r * r2).astype(f4), ps, r), fma(fma(pc, r2, f4(-0.5)), r2, f4(1.0))
    a, b = np.where(k & 1, cs, sn), np.where(k & 1, sn, cs)
    return np.where(k & 2, -a, a), np.where((k + 1) & 2, -b, b)


if __name__ == "__main__":
    s, es = fit(lambda x: np.sin(x) - x, lambda x: x**3, 2)
    c, ec = fit(lambda x: np.cos(x) - 1 + x * x / 2, lambda x: x**4, 2)
    parts = split_pi_2()
    print("sin:", " ".join("%.9ef" % v for v in s), "max error %.2g" % es)
    print("cos:", " ".join("%.9ef" % v for v in c), "max error %.2g" % ec)
    print("pi/2:", " ".join("%.9ef" % v for v in parts), " 2/pi: %.9ef" % f4(2 / np.pi))
    for lim in (1.0, 30.0, 3e4):
        z = np.random.default_rng(1).uniform(-lim, lim, 1000000).astype(f4)
        for got, want in zip(sincos(z, s, c, parts), (np.sin(z.astype(np.float64)), np.cos(z.astype(np.float64)))):
            e = np.abs(got - want)
            print("|z| <= %g: max %.2f ulp, rms %.2g" % (lim, (e / np.spacing(np.abs(want).astype(f4))).max(), np.sqrt((e * e).mean())))
