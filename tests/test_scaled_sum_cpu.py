"""The integer sums of the batched rates' scaled form, compiled for the host: rounding
against exact rationals, and the recurrence they serve against the weighted one."""
import ctypes as C
import os
import random
import subprocess
from fractions import Fraction
from math import comb, frexp, ldexp

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2311_01492_gb300", "csrc")


@pytest.fixture(scope="module")
def sum4(tmp_path_factory):
    d = tmp_path_factory.mktemp("scaled_sum")
    src, lib = str(d / "s.cpp"), str(d / "s.so")
    with open(src, "w") as f:
        f.write('#include "%s/scaled_sum.cuh"\n'
                'extern "C" double sum4(double a, double b, double c, double d) {\n'
                "  return asora::round_sum(a + b, asora::pair_sum(c, d));\n}\n" % CSRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", src,
                    "-o", lib], check=True)
    fn = C.CDLL(lib).sum4
    fn.restype, fn.argtypes = C.c_double, [C.c_double] * 4
    return fn


@pytest.mark.parametrize("spread", [0, 1, 3, 12, 54, 80])
def test_rounds_like_the_exact_sum(sum4, spread):
    """a + b in double, then the sum with c + d: within half a unit in the last place of
    the sum (for a + b) plus half a unit and the three cuts at the ninth guard bit."""
    rng = random.Random(spread)
    for _ in range(4000):
        e = rng.randrange(-300, 300)
        v = [0.0 if rng.random() < 0.1 else
             ldexp(1 + rng.getrandbits(52) / 2 ** 52, e + rng.randint(-spread, spread))
             for _ in range(4)]
        exact = sum(map(Fraction, v))
        if exact == 0:
            continue
        got = sum4(*v)
        ulp = Fraction(2) ** (frexp(float(exact))[1] - 53)
        half_ab = Fraction(v[0] + v[1]) - Fraction(v[0]) - Fraction(v[1])
        assert abs(Fraction(got) - exact - half_ab) <= ulp * (Fraction(1, 2) + Fraction(3, 256))


def test_zero_and_exact_cases(sum4):
    assert sum4(0.0, 0.0, 0.0, 0.0) <= ldexp(1, -1020)
    assert sum4(1.0, 0.0, 0.0, 0.0) == 1.0
    assert sum4(0.0, 0.0, 0.0, 3.5) == 3.5
    assert sum4(1.0, 1.0, 1.0, 1.0) == 4.0
    big = ldexp(1, 900)
    assert sum4(big, 1.0, big, 1.0) == 2 * big


@pytest.mark.parametrize("m", [2, 3, 17, 50])
def test_scaled_recurrence_equals_the_weighted_one(sum4, m):
    """One layer step: kappa tau_in from four slots of layer m - 1, for every cell of
    layer m, against the bilinear weights in exact arithmetic (zero outside layer m - 1)."""
    rng = random.Random(m)
    tau = {(i, j): rng.uniform(0, 1e4) * 10.0 ** rng.randint(-6, 0)
           for i in range(m) for j in range(m)}
    S = {k: float(Fraction(v) * comb(m - 1, k[0]) * comb(m - 1, k[1])) for k, v in tau.items()}
    for a1 in range(m + 1):
        for a2 in range(m + 1):
            got = sum4(*(S.get((a1 - p, a2 - q), 0.0) for q in (0, 1) for p in (0, 1)))
            x, y = Fraction(a1, m), Fraction(a2, m)
            want = sum(wx * wy * Fraction(tau[(i, j)])
                       for wx, i in ((1 - x, a1), (x, a1 - 1)) if wx
                       for wy, j in ((1 - y, a2), (y, a2 - 1)) if wy)
            kappa = comb(m, a1) * comb(m, a2)
            # four rounded slots, one rounded bracket and the rounded sum: each at most half
            # a unit in the last place of a part of the whole
            assert abs(Fraction(got) / kappa - want) <= want * Fraction(2) ** -51
