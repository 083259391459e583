"""The FP64 exp of the KLE kernels as they evaluate it (field.cu, kle_exp):
from t = x 64 / ln 2, with the nearest integer by the 1.5 2^52 shift, the
Taylor polynomial in t - N and the power of two added to the exponent field.
Simulated in exact rational arithmetic with the source's constants, it stays
within 1.5 ulp of 2^(t/64) (half an ulp of its last FMA, one of the table's
entry and the polynomial) over the range it is used in, and the index and
exponent it takes from the low word are those of the nearest integer."""
import math
import random
import re
import struct
from decimal import Decimal, getcontext
from fractions import Fraction
from pathlib import Path

import pytest

SRC = (Path(__file__).resolve().parents[1] / "paper_2111_11788_gb300" / "csrc" / "field.cu").read_text()


def const(name):
    tok = re.search(r"constexpr double %s = ([^;]+);" % name, SRC).group(1).strip()
    return float.fromhex(tok) if tok.startswith("0x") else float(tok)


INV = const("kInvLn2x64")
R = const("kR")
ROUND = const("kRound")
BIG = int(re.search(r"constexpr int kBig = (0x[0-9a-f]+);", SRC).group(1), 16)
C = [R, R * R / 2.0, R * R * R / 6.0, R * R * R * R / 24.0, R * R * R * R * R / 120.0]
getcontext().prec = 60
TAB = [float((Decimal(2).ln() * j / 64).exp()) for j in range(64)]


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def words(x):
    lo, hi = struct.unpack("<II", struct.pack("<d", x))
    return hi, lo


def kle_exp(t):
    y = t + ROUND
    N = struct.unpack("<i", struct.pack("<I", words(y)[1]))[0]
    f = t - (y - ROUND)
    assert N == round(t) and Fraction(f) == Fraction(t) - N
    q = fma(f, C[4], C[3])
    for c in (C[2], C[1], C[0]):
        q = fma(f, q, c)
    T = TAB[N & 63]
    hi, lo = words(fma(T, f * q, T))
    return struct.unpack("<d", struct.pack("<II", lo, hi + ((N >> 6) << 20)))[0]


def test_constants_are_the_nearest_doubles():
    ln2 = Fraction(6931471805599453094172321214581765680755, 10 ** 40)
    assert abs(Fraction(R) - ln2 / 64) <= Fraction(math.ulp(R)) / 2
    assert abs(Fraction(INV) - 64 / ln2) <= Fraction(math.ulp(INV)) / 2


@pytest.mark.parametrize("scale", [1e-3, 1.0, 60.0, 700.0, 30000.0, 63480.0])
def test_within_an_ulp_and_a_half(scale):
    rng = random.Random(int(scale * 7))
    for k in range(400):
        t = rng.uniform(-scale, scale) if k > 4 else (0.0, -0.0, 0.5, -0.5, scale)[k]
        ref = (Decimal(2).ln() * Decimal(t) / 64).exp()
        got = kle_exp(t)
        assert abs(Decimal(got) - ref) <= Decimal(1.5) * Decimal(math.ulp(float(ref))), (t, got)


def test_the_fast_path_ends_before_the_exponent_does():
    t = struct.unpack("<d", struct.pack("<II", 0xFFFFFFFF, BIG - 1))[0]   # the largest t below the threshold
    assert 0.0 < kle_exp(-t) and kle_exp(t) < math.inf
    assert abs(kle_exp(-t) * kle_exp(t) - 1.0) < 1e-13
    for bad in (math.inf, -math.inf, math.nan):
        assert words(bad)[0] & 0x7FFFFFFF >= BIG
