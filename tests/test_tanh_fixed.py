"""The integer tanh of the FP64 digit kernels (csrc/digits.cuh tanh_fixed), restated in Python integers, against
30-digit arithmetic: every interval of its table, 40 to 56 fraction bits of the argument, and the clamp at 20 (CPU).

Bar: the table's leading coefficients have 62 fraction bits and the result 54 (2^-55 of rounding); what is left is
the quadratic coefficient times the 32-bit cubic one's rounding, d^3 2^-32 with |d| <= 2^-7: 2^-53, and the FP32
tail, d^4 2^-24 / 6: 2^-54.6.  Together below 2^-52."""
import math
import random
from decimal import Decimal, getcontext

import numpy as np

getcontext().prec = 36
N = 1281


def _tanh(x):
    e = (2 * x).exp()
    return (e - 1) / (e + 1)


def _node(k):
    """c0 .. c6 at k / 64: Taylor coefficients, the degree-7 one economised over |d| <= 2^-7."""
    t = _tanh(Decimal(k) / 64)
    q = [None, [Decimal(1)]]
    for n in range(2, 8):
        p = [Decimal(0)] * (len(q[n - 1]) + 2)
        for j, c in enumerate(q[n - 1]):
            p[j] += c
            p[j + 2] -= c
        q.append([p[j] * j for j in range(1, len(p))])
    c = [t]
    for n in range(1, 8):
        s = Decimal(0)
        for v in reversed(q[n]):
            s = s * t + v
        c.append((1 - t * t) * s / math.factorial(n))
    h = Decimal(1) / 128
    c[5] += c[7] * h ** 2 * 112 / 64
    c[3] -= c[7] * h ** 4 * 56 / 64
    c[1] += c[7] * h ** 6 * 7 / 64

    def fix(v, bits):
        return int((v * 2 ** bits).to_integral_value())

    return fix(c[0], 62), fix(c[1], 62), fix(c[2], 62), fix(c[3], 32), [np.float32(float(v)) for v in c[4:7]]


def _tanh_fixed(z, zs, node):
    lim = 32 << zs
    z = max(-lim, min(lim, z))
    a = abs(z)
    k = (a + (1 << (zs - 7))) >> (zs - 6)
    d = a - (k << (zs - 6))
    if k >= N - 1:
        k, d = N - 1, 0
    D = d << (70 - zs)
    assert -2 ** 63 <= D < 2 ** 63
    Dh = D >> 32
    c0, c1, c2, c3, (c4, c5, c6) = node(k)
    f = np.float32
    df = f(Dh) * f(2.0 ** -38)
    F = f(np.float64(df) * f(np.float64(df) * c6 + c5) + c4)
    u3 = c3 + int(np.rint(f(df * F) * f(2.0 ** 32)))
    u2 = c2 + ((Dh * u3) >> 8)
    u1 = c1 + (((D * u2) >> 64) >> 6)
    t = c0 + (((D * u1) >> 64) >> 6)
    assert abs(t) < 2 ** 63
    t = (t + 128) >> 8
    return -t if z < 0 else t


def test_error_over_all_intervals():
    rng = random.Random(5)
    cache = {}

    def node(k):
        if k not in cache:
            cache[k] = _node(k)
        return cache[k]

    worst = rms = 0.0
    args = [k + o for k in range(N + 40) for o in (-0.5, rng.uniform(-0.5, 0.5), 0.0, rng.uniform(-0.5, 0.5))]
    for n, a in enumerate(args):
        zs = 40 + n % 17
        z = int(math.floor(a / 64.0 * 2.0 ** zs)) * (1 if rng.random() < 0.5 else -1)
        t = Decimal(_tanh_fixed(z, zs, node)) / 2 ** 54
        e = float(t - _tanh(Decimal(z) / 2 ** zs))
        worst, rms = max(worst, abs(e)), rms + e * e
    rms = math.sqrt(rms / len(args))
    assert worst <= 2.0 ** -52, math.log2(worst)
    assert rms <= 2.0 ** -54, math.log2(rms)
    print(f"rms 2^{math.log2(rms):.1f}, at most 2^{math.log2(worst):.1f}")


def test_clamp_and_limits():
    for zs in (40, 52, 56):
        for z in (20 << zs, (32 << zs) + 5, 2 ** 63 - 1, -2 ** 63):
            t = _tanh_fixed(z, zs, _node)
            assert t == (2 ** 54 if z > 0 else -2 ** 54)
        assert _tanh_fixed(0, zs, _node) == 0
