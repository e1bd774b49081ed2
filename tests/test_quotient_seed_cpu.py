"""The FP64 quotient of the force of infection as the kernels evaluate it: a float reciprocal of the
divisor's leading 24 bits (truncated, not rounded), off by up to two float ulps, one
Newton-Raphson step and Markstein's remainder correction (each a fused multiply-add), with exact
rational arithmetic for every FMA.  After the Newton step the reciprocal's relative error is at most
(2^-21)^2 = 2^-42, after the correction 2^-84 plus the last rounding: the correctly rounded quotient
unless it lies within 2^-31 ulps of a tie, so all but a vanishing share of the draws must equal it
and none may be off by more than one ulp."""
from fractions import Fraction

import numpy as np


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def _quotient(num, d, ulps):
    bits = np.array([d]).view(np.uint64)[0]
    f = np.array([np.uint64(bits) & ~np.uint64((1 << 29) - 1)]).view(np.float64)[0]  # 23 fraction bits kept
    f32 = np.float32(f)
    assert float(f32) == f
    r32 = np.float32(1.0) / f32
    r = float((np.array([r32]).view(np.int32) + np.int32(ulps)).view(np.float32)[0])
    r = _fma(r, _fma(-d, r, 1.0), r)
    q = num * r
    return _fma(r, _fma(-d, q, num), q)


def test_one_newton_step_and_the_correction_round_correctly():
    g = np.random.Generator(np.random.PCG64(19789))
    n = 3000
    d = 2.0 ** g.uniform(-99, 99, n)
    d[: n // 3] = g.uniform(0.05, 2.0, n // 3)       # densities of the workloads
    d[n // 3: n // 2] = g.uniform(100.0, 130.0, n // 2 - n // 3)  # the paper's, per square kilometre
    num = d * g.uniform(0.0, 1.0, n) * 10.0 ** g.uniform(-8, 0, n)
    for ulps in (-2, -1, 0, 1, 2):
        for a, b in zip(num[::5 if ulps else 1], d[::5 if ulps else 1]):
            want = float(Fraction(float(a)) / Fraction(float(b)))
            assert _quotient(float(a), float(b), ulps) == want, (a, b, ulps)
