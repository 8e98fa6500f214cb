"""Writes the FP64 heatbath deviate's table (erfcinv_f64_table.inc, run by the build).

The deviate is erfc^-1(u) / sqrt(3) for u = m 2^-32, m odd in [1, 2^32).  The
range of m is cut into segments, each with the Taylor polynomial of the
function about a node of its own:

  u < 1/2   31 octaves of u (lz = number of leading zeros of m, 1 .. 31) x 32
            segments of n = m << lz, node at the segment's middle,
            argument r = (n mod 2^26) - 2^25
  u > 1/2   64 segments of m' = 2^32 - m (x = 1 - u = m' 2^-32 < 1/2), node at
            the middle and r = (m' mod 2^25) - 2^24, but x = 0 and r = m' for
            the first one, so that the deviate keeps its relative accuracy
            where it goes to 0

Node values come from Newton's method on the power series of erf in 60-digit
decimals; the higher coefficients from the differential equation
y' = -(sqrt(pi) / 2) exp(y^2), y'' = 2 y y'^2 (dy/du), term by term.  The
argument r is an integer, so the powers of two of the segment's width are
folded into the coefficients exactly.  COEFS terms leave a truncation error
below 2^-59 of the value (8 would leave 2^-52.8); nothing is fitted.
"""
from decimal import Decimal as D, getcontext
from statistics import NormalDist
import math
import sys

getcontext().prec = 60
OCTAVES, PER_OCTAVE, CENTRE = 31, 32, 64
COEFS, ROW = 9, 10  # terms, and the row's length with its padding (80 bytes)
PI = D("3.14159265358979323846264338327950288419716939937510582097494459")
HALF_SQRT_PI = PI.sqrt() / 2


def erf(y):
    """2/sqrt(pi) sum_n (-1)^n y^(2n+1) / (n! (2n+1))"""
    t, s, n, y2 = y, y, 0, y * y
    while abs(t) > D(10) ** -58:
        n += 1
        t = -t * y2 / n
        s += t / (2 * n + 1)
    return s / HALF_SQRT_PI


def node(u):
    """erfc^-1(u) for 0 < u <= 1"""
    if u == 1:
        return D(0)
    y = D(-NormalDist().inv_cdf(float(u) / 2) / math.sqrt(2.0))
    for _ in range(2):  # 16 -> 32 -> 60 digits
        f = 1 - erf(y) - u
        y += f * HALF_SQRT_PI * (y * y).exp() * (1 + f * HALF_SQRT_PI * (y * y).exp() * y)
    return y


def taylor(u, step):
    """Coefficients of erfc^-1(u + step r) / sqrt(3) in r"""
    y = [node(u)]
    p = [-HALF_SQRT_PI * (y[0] * y[0]).exp()]
    for n in range(COEFS - 1):
        y.append(p[n] / (n + 1))
        pp = [sum(p[i] * p[k - i] for i in range(k + 1)) for k in range(n + 1)]
        p.append(2 * sum(y[k] * pp[n - k] for k in range(n + 1)) / (n + 1))
    r3 = D(3).sqrt()
    return [float(c * step ** k / r3) for k, c in enumerate(y)]


def segments():
    """(u of the node, du per unit of r) in table order"""
    for o in range(OCTAVES):
        e = D(2) ** (-32 - (o + 1))
        for j in range(PER_OCTAVE):
            yield ((PER_OCTAVE + j) * 2 ** 26 + 2 ** 25) * e, e
    for j in range(CENTRE):
        e = D(2) ** -32
        yield 1 - (j * 2 ** 25 + (2 ** 24 if j else 0)) * e, -e


def main(path):
    rows = [taylor(u, e) for u, e in segments()]
    with open(path, "w") as f:
        f.write("// written by gen_erfcinv_f64.py\n")
        for r in rows:
            f.write("{" + ", ".join(c.hex() for c in r + [0.0] * (ROW - COEFS)) + "},\n")


if __name__ == "__main__":
    main(sys.argv[1])
