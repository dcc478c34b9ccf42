"""Writes the table of the fixed-point tanh (csrc/fixed.cuh) as a C++ include.

Row j holds the degree-6 polynomial of tanh on [j/64, (j+1)/64) in the variable
r = 128 (s - (j + 1/2)/64) in [-1, 1): the Taylor polynomial of degree 20 about the
interval's middle, from the recurrence of T' = 1 - T^2, lowered to degree 6 by
subtracting the leading multiples of Chebyshev polynomials (economisation,
Lanczos 1938); the dropped terms are below 2^-58.  Coefficients are integers in
units of 2^-61.  The last row is the constant 1 - 2^-61, for s >= 22 where
1 - tanh(s) < 2^-62.

A row is three 16-byte words: (c0, c1), (c2, c3) in 64 bits each, then c4, c5, c6.
"""
from __future__ import annotations

import decimal
import os

ROWS_PER_UNIT = 64
LIMIT = 22
DEGREE = 6
BITS = 61
TAYLOR = 20


def row(j: int):
    """The seven integer coefficients of interval j."""
    D = decimal.Decimal
    s0 = D(2 * j + 1) / (2 * ROWS_PER_UNIT)
    e = (-2 * s0).exp()
    h = D(1) / (2 * ROWS_PER_UNIT)
    a = [(1 - e) / (1 + e)]
    for k in range(TAYLOR):   # (k + 1) a_{k+1} = [k = 0] - sum_i a_i a_{k-i}
        a.append(((1 if k == 0 else 0) - sum(a[i] * a[k - i] for i in range(k + 1))) / (k + 1))
    c = [a[k] * h ** k for k in range(TAYLOR + 1)]
    cheb = [[1], [0, 1]]      # T_n as integer monomial coefficients
    for n in range(2, TAYLOR + 1):
        p = [0] + [2 * v for v in cheb[n - 1]]
        for i, v in enumerate(cheb[n - 2]):
            p[i] -= v
        cheb.append(p)
    for n in range(TAYLOR, DEGREE, -1):
        t = c[n] / cheb[n][n]
        for i, v in enumerate(cheb[n]):
            c[i] -= t * v
    return [int((v * 2 ** BITS).to_integral_value()) for v in c[:DEGREE + 1]]


def words(c):
    """A row as twelve 32-bit words."""
    def split(v):
        return [v & 0xFFFFFFFF, (v >> 32) & 0xFFFFFFFF]
    assert all(-2 ** 31 <= v < 2 ** 31 for v in c[4:])
    w = split(c[0]) + split(c[1]) + split(c[2]) + split(c[3])
    w += [v & 0xFFFFFFFF for v in c[4:]] + [0]
    return w


def write(path: str) -> None:
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        rows = [row(j) for j in range(ROWS_PER_UNIT * LIMIT)]
    rows.append([2 ** BITS - 1] + [0] * DEGREE)
    with open(path + ".tmp", "w") as f:
        f.write("// written by tanh_table.py\n")
        for c in rows:
            w = [v - 2 ** 32 if v >= 2 ** 31 else v for v in words(c)]
            for q in range(0, 12, 4):
                # the smallest int has no literal of its own
                f.write("{%s}, " % ", ".join("(-2147483647 - 1)" if v == -2 ** 31 else str(v)
                                             for v in w[q:q + 4]))
            f.write("\n")
    os.replace(path + ".tmp", path)
