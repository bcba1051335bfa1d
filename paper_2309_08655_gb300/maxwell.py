"""Table for the inverse distribution of the Maxwellian speed (csrc/rt_maxwell.cuh).

The speed x = |k| / k0 has the density f(x) = 4/sqrt(pi) x^2 exp(-x^2).  Its
inverse distribution is tabulated cell by cell over [1/32, 4): 128 cells per
octave below 2 and 256 in [2, 4), so that a cell is the leading bits of a float.
Around the centre x0 of a cell, with t the change of the distribution divided by
f(x0),

    x = x0 + t + c2 t^2 + ... + c9 t^9,

the reversed Taylor series of the distribution (the ratio f(x0 + d) / f(x0) is
(1 + d/x0)^2 exp(-2 x0 d - d^2)).  The half-width of a cell keeps the first term
left out below 2^-53 x.  Cells below the median hold the distribution itself and
1/f(x0), cells above it the complement and -1/f(x0): v = u or 1 - u is then never
a small difference.

A cell is ten doubles: the distribution (or complement) at x0, +-1/f(x0), c2 .. c9.
"""
from __future__ import annotations

import decimal
import math

DEGREE = 9
X_LO, X_MID, X_HI = 2.0 ** -5, 2.0, 4.0
LOW_BITS, HIGH_BITS = 7, 8            # cells per octave (log2) below and above X_MID
LOW_CELLS = 6 << LOW_BITS
CELLS = LOW_CELLS + (1 << HIGH_BITS)
MEDIAN = 1.0876520317
_CTX = decimal.Context(prec=45)


def centre(cell: int) -> float:
    """The middle of a cell (exact in binary)."""
    if cell < LOW_CELLS:
        octave, k = divmod(cell, 1 << LOW_BITS)
        return X_LO * 2.0 ** octave * (1.0 + (k + 0.5) / (1 << LOW_BITS))
    return X_MID * (1.0 + (cell - LOW_CELLS + 0.5) / (1 << HIGH_BITS))


def _pi() -> decimal.Decimal:
    """Machin's formula."""
    def arctan_inv(n: int) -> decimal.Decimal:
        total = term = _CTX.divide(decimal.Decimal(1), decimal.Decimal(n))
        k, n2 = 1, n * n
        while abs(term) > decimal.Decimal(10) ** -44:
            term = -_CTX.divide(term, decimal.Decimal(n2))
            k += 2
            total = _CTX.add(total, _CTX.divide(term, decimal.Decimal(k)))
        return total

    return _CTX.subtract(16 * arctan_inv(5), 4 * arctan_inv(239))


def distribution(x: float, sqrt_pi: decimal.Decimal) -> tuple[decimal.Decimal, decimal.Decimal]:
    """The distribution and the density at x: x^3 exp(-x^2) times a series of
    positive terms (no cancellation)."""
    with decimal.localcontext(_CTX):
        X = decimal.Decimal(x)
        y = X * X
        e = (-y).exp()
        term = total = decimal.Decimal(1) / 3
        k = 0
        while term > total * decimal.Decimal(10) ** -40:
            k += 1
            term = term * 2 * y / (2 * k + 3)
            total += term
        return 4 * X * y * e * total / sqrt_pi, 4 * y * e / sqrt_pi


def _reversed_series(x0: float) -> list[float]:
    """c1 = 1, c2 .. c_DEGREE."""
    n = DEGREE
    # Taylor coefficients of (1 + d/x0)^2 exp(-2 x0 d - d^2)
    ex = [1.0]
    for k in range(1, n):
        ex.append((-2.0 * x0 * ex[k - 1] - (2.0 * ex[k - 2] if k > 1 else 0.0)) / k)
    q = [1.0, 2.0 / x0, 1.0 / (x0 * x0)]
    r = [sum(q[j] * ex[k - j] for j in range(min(k, 2) + 1)) for k in range(n)]
    a = [0.0] + [r[k] / (k + 1) for k in range(n)]       # t = d + a2 d^2 + ...
    c = [0.0, 1.0]
    for m in range(2, n + 1):
        # the coefficient of t^m in sum_k a_k d(t)^k without c_m
        d = c + [0.0] * (n + 1 - len(c))
        power, total = d[:], 0.0
        for k in range(2, m + 1):
            power = [sum(power[i] * d[j - i] for i in range(j + 1)) for j in range(n + 1)]
            total += a[k] * power[m]
        c.append(-total)
    return c[1:]


def table() -> list[list[float]]:
    sqrt_pi = _CTX.sqrt(_pi())
    rows = []
    for cell in range(CELLS):
        x0 = centre(cell)
        F, f = distribution(x0, sqrt_pi)
        c = _reversed_series(x0)
        if x0 < MEDIAN:
            rows.append([float(F), float(_CTX.divide(decimal.Decimal(1), f))] + c[1:])
        else:
            rows.append([float(_CTX.subtract(decimal.Decimal(1), F)),
                         -float(_CTX.divide(decimal.Decimal(1), f))] + c[1:])
    return rows


def first_upper_cell() -> int:
    return next(i for i in range(CELLS) if centre(i) >= MEDIAN)


def write(path: str) -> None:
    """The table as a C array initialiser."""
    rows = table()
    assert all(math.isfinite(v) for r in rows for v in r)
    with open(path, "w") as f:
        f.write("// Written by maxwell.py: cells of the inverse Maxwellian distribution.\n")
        f.write("constexpr int MAXWELL_CELLS = %d, MAXWELL_LOW_CELLS = %d;\n" % (CELLS, LOW_CELLS))
        f.write("constexpr int MAXWELL_FIRST_UPPER = %d;\n" % first_upper_cell())
        f.write("__device__ __align__(16) const double maxwell_table[MAXWELL_CELLS][%d] = {\n" % (DEGREE + 1))
        for r in rows:
            f.write("{" + ",".join(v.hex() for v in r) + "},\n")
        f.write("};\n")
