"""Host-side checks of the arithmetic identities the CUDA quantizer's division-free arithmetic
relies on, against the plain definition (Appendix A.3: SINT4, fp16 scale, RTN)."""
from fractions import Fraction

import numpy as np
import pytest

from oracle import lq_oracle as O


def test_scale_by_reciprocal_equals_division_for_every_fp16_maximum():
    """The kernel forms the group scale as fp16(a * fl32(1/7)); the definition is fp16(a /fl32 7).
    Every finite non-negative fp16 value can be a group maximum: check them all through the
    oracle's quantizer (a one-element group has maximum a)."""
    a16 = np.arange(0, 0x7C00, dtype=np.uint16).view(np.float16)
    _, s_def = O.qgrp(a16.astype(np.float32)[:, None], group=64)
    s_fast = (a16.astype(np.float32) * np.float32(1.0 / 7.0)).astype(np.float16)
    s_fast = np.maximum(s_fast, O.SCALE_FLOOR)
    assert np.array_equal(s_def[:, 0].view(np.uint16), s_fast.view(np.uint16))


def _rn32(v: Fraction) -> Fraction:
    """v rounded to the nearest binary32 number, ties to even (normal range), in exact rational arithmetic."""
    if v == 0:
        return Fraction(0)
    sign, a = (-1 if v < 0 else 1), abs(v)
    e = a.numerator.bit_length() - a.denominator.bit_length() - 23
    while a / Fraction(2) ** e >= 2 ** 24:
        e += 1
    while a / Fraction(2) ** e < 2 ** 23:
        e -= 1
    t = a / Fraction(2) ** e
    n = t.numerator // t.denominator
    rem = t - n
    if rem > Fraction(1, 2) or (rem == Fraction(1, 2) and n % 2 == 1):
        n += 1
    return sign * n * Fraction(2) ** e


def test_fma_corrected_quotient_is_the_correctly_rounded_division():
    """The kernel never divides: with y = fl32(1/b) it forms q0 = fl32(a y), r = a - b q0 (exact in an FMA) and
    q1 = fl32(q0 + r y).  q1 must be fl32(a / b), the definition's quotient (Appendix A.3: RTN of the scaled value),
    for fp16 numerators over fp16 scales (main branch) and over fp32 per-token scales (low-rank branch), including
    quotients that sit exactly on k + 1/2.  Everything here is exact rational arithmetic."""
    rng = np.random.default_rng(0)
    cases = []
    x16 = rng.standard_normal(6000).astype(np.float16)
    s16 = (np.abs(rng.standard_normal(6000)) * 0.3 + 2.0 ** -10).astype(np.float16)
    cases += [(Fraction(float(a)), Fraction(float(b))) for a, b in zip(x16, s16)]
    for k in range(0, 8):                                    # exact ties x = (k + 1/2) s
        for b in s16[:60]:
            a = np.float16((k + 0.5) * float(b))
            cases.append((Fraction(float(a)), Fraction(float(b))))
    xb = (rng.standard_normal(6000) * 3).astype(np.float16)
    rowmax = np.abs(xb).max()
    for qm in (127.0, 31.0, 7.0):
        sb = np.float32(np.float32(rowmax) / np.float32(qm))
        cases += [(Fraction(float(a)), Fraction(float(sb))) for a in xb[:2000]]
    ties = 0
    for a, b in cases:
        y = _rn32(1 / b)
        q0 = _rn32(a * y)
        r = a - b * q0
        assert _rn32(r) == r, "the remainder must be a binary32 number (exact FMA)"
        q1 = _rn32(q0 + r * y)
        assert q1 == _rn32(a / b), (float(a), float(b))
        ties += (2 * a / b).denominator == 1 and (a / b).denominator == 2
    assert ties > 100


@pytest.mark.parametrize("qm", [127, 31])
def test_row_scale_without_a_division(qm):
    """sb = fl32(max / qm) of every finite fp16 maximum from the product with fl32(1 / qm) and one correction step.  (The last FMA is rounded from a sum in 64 bits: a
    quotient is never nearer than 2^-33 to the middle between two binary32 numbers.)"""
    rm = np.arange(1, 0x7C00, dtype=np.uint16).view(np.float16).astype(np.float32)
    rqm = np.float64(np.float32(1) / np.float32(qm))
    q0 = (rm * rqm).astype(np.float32).astype(np.float64)
    rest = rm.astype(np.float64) - q0 * qm
    assert np.array_equal(rest, rest.astype(np.float32))
    assert np.array_equal((q0 + rest * rqm).astype(np.float32), rm / np.float32(qm))


@pytest.mark.parametrize("qm", [127, 31])
def test_one_fma_with_a_chosen_reciprocal_gives_the_codes_of_the_quotient(qm):
    """Branch codes by x -> rint(x inv) (one FMA with 1.5 * 2^23: the product is not rounded before) for every finite fp16 row
    maximum and, of the values up to it, the two next to every tie (k + 1/2) max / qm and the tie itself: the codes of the definition,
    rint(fl32(x / sb)).  Values away from ties cannot differ if these do not.  Rows whose maximum's significand is a multiple of qm
    go another way and are left out."""
    bits = np.arange(1, 0x7C00, dtype=np.uint32)
    significand = (bits & 0x3FF) | np.where(bits < 0x400, 0, 0x400)
    rm = bits[significand % qm != 0].astype(np.uint16).view(np.float16).astype(np.float32)
    sb = rm / np.float32(qm)
    exact = (1.0 / sb.astype(np.float64)).astype(np.float32)
    near = {127: 2.0 ** -19, 31: 2.0 ** -21}[qm]                                         # half an ulp of qm / 2
    up = 0.5 * rm.astype(np.float64) - sb.astype(np.float64) * (0.5 * qm) >= -near * sb  # exact: 31 bits
    assert np.array_equal(up, np.rint((np.float32(0.5) * rm) / sb) == (qm + 1) // 2)
    codes = []                                                       # of reciprocals up to an ulp and a half off
    for off in (-1, 0, 1):
        rcp = (exact.view(np.int32) + off).astype(np.int32).view(np.float32)
        above = 0.5 * rm.astype(np.float64) * rcp.astype(np.float64) - 0.5 * qm >= 0      # exact: 35 bits
        codes.append(np.where(above == up, rcp.view(np.int32), rcp.view(np.int32) + np.where(up, 4, -4)).astype(np.int32).view(np.float32))
        assert (above != up).sum() > 1000
    ties = 0
    for k in range(qm):
        t = (k + 0.5) * rm.astype(np.float64) / qm
        mid = t.astype(np.float16)
        for step in (-1, 0, 1):
            x = (mid.view(np.int16) + step).astype(np.int16).view(np.float16).astype(np.float64)
            x = np.where((x >= 0) & (x <= rm), x, 0.0)
            code = np.rint((x.astype(np.float32) / sb).astype(np.float64))
            for inv in codes:
                assert np.array_equal(np.rint(x * inv.astype(np.float64)), code), k
            ties += (x * 2 * qm == (2 * k + 1) * rm.astype(np.float64)).sum()
    assert ties > 10000
