"""The table of |z| Phi(-|z|) that the float64 split-digit value function reads
(csrc/gelu_table.inc), against integer arithmetic of 200 bits (CPU).

A row holds one interval of width 2^-7: the quintic in tau = 256 (|z| - centre),
coefficients c0 (62 fraction bits), c1 (71), c2 (80; the low 16 bits hold c5),
c3 (57), c4 (58), c5 (59).  The largest error stated beside the table is 2^-56.9,
the root mean square 2^-59.2."""
import math
import os
import re

import paper_2601_01903_gb300 as fsi

FRAC = 200
ONE = 1 << FRAC
TABLE = os.path.join(os.path.dirname(fsi.__file__), "csrc", "gelu_table.inc")


def _rows():
    with open(TABLE) as f:
        return [[int(w, 16) for w in re.findall(r"0x([0-9a-fA-F]+)ull", line)] for line in f if "ull" in line]


def _signed(v, bits):
    return v - (1 << bits) if v >> (bits - 1) else v


def _pi():
    """Machin's formula."""
    def arctan_inverse(n):
        s = t = (ONE << 20) // n
        k, sign = 1, -1
        while t:
            t //= n * n
            s += sign * (t // (2 * k + 1))
            k, sign = k + 1, -sign
        return s
    return (16 * arctan_inverse(5) - 4 * arctan_inverse(239)) >> 20


def _exp_neg(x):
    """exp(-x), x >= 0, by halving the argument 12 times and Taylor's series."""
    x >>= 12
    s = t = ONE
    k = 1
    while t:
        t = -(t * x >> FRAC) // k if t > 0 else (-t * x >> FRAC) // k
        s += t
        k += 1
        if abs(t) <= 1:
            break
    for _ in range(12):
        s = s * s >> FRAC
    return s


INV_SQRT_2PI = math.isqrt((ONE ** 3) // (2 * _pi()))  # 1 / sqrt(2 pi)


def _tail(z):
    """z Phi(-z) for z >= 0 (FRAC fraction bits): z (1/2 - phi(z) sum z^(2n+1) / (2n+1)!!)."""
    z2 = z * z >> FRAC
    s, t, n = 0, z, 0
    while t:
        s += t
        n += 1
        t = (t * z2 >> FRAC) // (2 * n + 1)
    phi = INV_SQRT_2PI * _exp_neg(z2 >> 1) >> FRAC
    return z * ((ONE >> 1) - (phi * s >> FRAC)) >> FRAC


def _quintic(row, tau_num, tau_den):
    """The row's polynomial at tau = tau_num / tau_den, FRAC fraction bits."""
    w0, w1, w2, w3 = row
    c5 = _signed(w2 & 0xffff, 16)
    coef = [(_signed(w0, 64), 62), (_signed(w1, 64), 71), (_signed(w2, 64), 80),
            (_signed(w3 & 0xffffffff, 32), 57), (_signed(w3 >> 32, 32), 58), (c5, 59)]
    acc = 0
    for c, f in reversed(coef):
        acc = acc * tau_num // tau_den + (c << (FRAC - f))
    return acc


def test_every_interval_stays_within_the_stated_error():
    """The stated bounds to their last digit: the largest error at the ends,
    where a truncated polynomial is worst, and between; the root mean square
    over points spread evenly over every interval."""
    rows = _rows()
    assert len(rows) == 1121 and all(len(r) == 4 for r in rows)

    def error(i, tau16):  # at tau = tau16 / 16
        z = (2 * i + 1) * ONE // 256 + tau16 * ONE // 4096
        return abs(_quintic(rows[i], tau16, 16) - _tail(z))

    even = [[error(i, t) for t in range(-15, 16, 2)] for i in range(1120)]
    assert max(max(error(i, -16), error(i, 16), max(even[i])) for i in range(1120)) <= ONE / 2 ** 56.85
    assert math.sqrt(sum((e / ONE) ** 2 for r in even for e in r) / (16 * 1120)) <= 2 ** -59.15


def test_beyond_the_table_the_result_is_zero():
    assert _rows()[1120] == [0, 0, 0, 0]
    assert _tail(1120 * ONE // 128) < ONE / 2 ** 56
