"""The two FP64 forms that the kernels use in place of the library's division and
exponential, in exact arithmetic on the host (an FMA is the exact sum rounded
once): the corrected quotient of the power tables equals the correctly rounded
one, also where the quotient lies beside a midpoint of two doubles and where
the divisor's mantissa is all ones; the table-driven exponential of the 1-D
path is within 1.02 ulp of 40-digit values on its whole range, with the table
read from its source (half an ulp each of the table and of the last rounding,
0.01 of r and of the polynomial)."""
import decimal
import math
import os
import random
import re
from fractions import Fraction as F

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_11246_gb300", "csrc")


def fma(a, b, c):
    return float(F(a) * F(b) + F(c))


def quotient(a, s):  # vup_grid.cu: div_scale
    inv = 1.0 / s
    q = a * inv
    return fma(fma(-q, s, a), inv, q)


def test_corrected_quotient_is_correctly_rounded():
    rng = random.Random(3)
    mant = lambda: math.ldexp(rng.getrandbits(52) | (1 << 52), -52)
    for _ in range(20000):
        a, s = rng.choice((1, -1)) * mant() * 2.0 ** rng.randint(-300, 300), mant() * 2.0 ** rng.randint(-200, 200)
        assert quotient(a, s) == a / s, (a.hex(), s.hex())
    for _ in range(20000):
        u = rng.random()
        s = mant() if u > 0.4 else (2.0 - rng.randint(1, 40) * 2.0 ** -52 if u > 0.1 else 1.0 + rng.randint(0, 40) * 2.0 ** -52)
        m = rng.choice((rng.getrandbits(52) | (1 << 52), (1 << 52) + rng.randint(0, 999), (1 << 53) - 1 - rng.randint(0, 999)))
        a = float(F(s) * F(2 * m + 1, 1 << 53)) * 2.0 ** rng.randint(-100, 100)  # the quotient beside a midpoint
        for x in (a, math.nextafter(a, 0.0), math.nextafter(a, math.inf)):
            assert quotient(x, s) == x / s, (x.hex(), s.hex())


def _table():
    src = open(os.path.join(SRC, "vup_1d.cu")).read()
    body = src[src.index("kExpTab[64] = {"):]
    return [float.fromhex(h) for h in re.findall(r"0x1\.[0-9a-f]+p\+0", body[:body.index("};")])]


def exp_neg(x, tab):  # vup_1d.cu: exp_neg
    magic = 6755399441055744.0
    t = fma(x, float.fromhex("0x1.71547652b82fep+6"), magic)
    kd = t - magic
    k = int(kd)
    r = fma(kd, -float.fromhex("0x1.62e42fee00000p-7"), x)
    r = fma(kd, -float.fromhex("0x1.a39ef35793c76p-39"), r)
    q = fma(r, 1.0 / 720.0, 1.0 / 120.0)
    q = fma(q, r, 1.0 / 24.0)
    q = fma(q, r, 1.0 / 6.0)
    q = fma(q, r, 0.5)
    q = fma(q, r * r, r)
    s = tab[k & 63]
    return math.ldexp(fma(s, q, s), k >> 6)


def test_table_driven_exponential():
    tab = _table()
    assert len(tab) == 64
    decimal.getcontext().prec = 40
    ln2 = decimal.Decimal(2).ln()
    for j, v in enumerate(tab):
        assert v == float((ln2 * j / 64).exp())
    rng = random.Random(4)
    xs = [-rng.uniform(0.0, 700.0) for _ in range(4000)] + [-10.0 ** rng.uniform(-18.0, 0.0) for _ in range(2000)]
    xs += [-(j + d) * math.log(2.0) / 64 for j in range(0, 64000, 61) for d in (0.5, 0.499999)] + [0.0, -699.999]
    worst = 0.0
    for x in xs:
        if x <= -700.0:
            continue
        want = decimal.Decimal(x).exp()
        got = exp_neg(x, tab)
        worst = max(worst, float(abs(decimal.Decimal(got) - want) / decimal.Decimal(math.ulp(float(want)))))
    assert worst <= 1.02, worst
