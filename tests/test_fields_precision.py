"""The mixed path's output velocity v = u + F/(2 rho) is a correctly rounded FP64 quotient
up to one unit in the last place, although it is computed in triple-float arithmetic.

  * CPU: the three-digit division restated in rounded FP32 operations, against exact
    rationals;
  * GPU: populations whose sums are exact and whose density is uniform (so F = 0), against
    FP64 division on the host.
"""
from fractions import Fraction

import numpy as np
import pytest

f4 = np.float32


def rnd(x):
    """A rational rounded to FP32 (through FP64: the double rounding costs under 2^-52)."""
    return f4(float(x))


def two_sum(a, b):
    s = f4(a + b)
    return s, rnd(Fraction(float(a)) + Fraction(float(b)) - Fraction(float(s)))


def fma(a, b, c):
    return rnd(Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c)))


def tf_sum(xs):
    a, b, c = f4(xs[0]), f4(0), f4(0)
    for x in xs[1:]:
        a, e = two_sum(a, f4(x))
        b, e = two_sum(b, e)
        c = f4(c + e)
    return a, b, c


def tf_div(n, hi, lo):
    inv = f4(f4(1) / hi)
    s, sl = two_sum(n[0], n[1])
    q0 = f4(s * inv)
    p, t = f4(q0 * hi), f4(q0 * lo)
    low = f4(n[2] - fma(q0, lo, -t))
    m, e = two_sum(f4(s - p), -fma(q0, hi, -p))
    low = f4(low + e)
    for x in (sl, -t):
        m, e = two_sum(m, x)
        low = f4(low + e)
    q1 = f4(f4(m + low) * inv)
    p1 = f4(q1 * hi)
    rem = f4(f4(m - p1) - fma(q1, hi, -p1))
    rem = f4(rem + fma(-q1, lo, low))
    return float(q0) + (float(q1) + float(f4(rem * inv)))


def test_triple_float_quotient_is_fp64():
    rng = np.random.default_rng(3)
    worst = 0.0
    for i in range(400):
        scale = 10.0 ** rng.uniform(-9, 0)
        g = (rng.uniform(0.5, 1.5, 7) * scale * rng.choice([1.0, 1e-3], 7)).astype(f4)
        g[1::2] *= f4(-1)
        if i % 4 == 0:
            g[1] = -np.nextafter(g[0], f4(2))  # cancelling pair
        r = rng.uniform(1, 9) * scale
        hi = f4(r)
        lo = f4(r - float(hi))
        exact = sum(Fraction(float(x)) for x in g) / (Fraction(float(hi)) + Fraction(float(lo)))
        got = tf_div(tf_sum(g), hi, lo)
        # one FP64 unit of the quotient, or 2^-66 of the terms where they cancel
        tol = max(abs(float(exact)) * 2.0**-52, float(np.abs(g).max()) / r * 2.0**-66)
        worst = max(worst, abs(float(Fraction(got) - exact)) / tol)
    assert worst <= 1.0, worst


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(8, 8), (37, 29), (260, 130)])
def test_mixed_velocity_is_fp64(cuda, nx, ny):
    from paper_1906_09530_gb300 import Simulation
    rng = np.random.default_rng(nx)
    # multiples of 2^-12, antisymmetric in each opposite pair: every sum is exact
    f = np.full((9, ny, nx), 0.0625)
    f[0] = 0.3125 - 5 * 2.0**-14
    for i, j in ((1, 3), (2, 4), (5, 7), (6, 8)):
        d = rng.integers(-200, 201, (ny, nx)) * 2.0**-12
        f[i] += d
        f[j] -= d
    sim = Simulation(nx, ny, 0.6, 0.1, 1.0, 0.5, precision="mixed")
    sim.set_populations(f)
    rho, vx, vy, mu = sim.fields()
    mass, vmax, rmin, rmax = sim.diag()
    sim.close()
    r = f.sum(axis=0)
    wx = ((f[1] + f[5] + f[8]) - (f[3] + f[6] + f[7])) / r
    wy = ((f[2] + f[5] + f[6]) - (f[4] + f[7] + f[8])) / r
    assert np.array_equal(rho, r)
    for v, w in ((vx, wx), (vy, wy)):
        assert np.all(np.abs(v - w) <= np.spacing(np.abs(w)))
    assert abs(vmax - np.sqrt(wx**2 + wy**2).max()) <= 4 * np.spacing(vmax)
    assert rmin == rmax == r[0, 0] and abs(mass - r.sum()) <= 1e-12 * mass
    assert np.all(mu == mu[0, 0])
