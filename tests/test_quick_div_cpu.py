"""Quotients formed mostly on the FP32 and integer units (quick_div.cuh), compiled for the
host with seeds as far off as the hardware's may be, against exact rationals."""
import ctypes as C
import os
import random
import subprocess
from fractions import Fraction
from math import frexp, inf, isnan, ldexp, nan

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2311_01492_gb300", "csrc")


@pytest.fixture(scope="module", params=[-1, 0, 1])  # units in the last place of the seed
def lib(request, tmp_path_factory):
    d = tmp_path_factory.mktemp("quick_div")
    src, lib = str(d / "s.cpp"), str(d / "s.so")
    with open(src, "w") as f:
        f.write('#include <math.h>\n#include <string.h>\n'
                'static float off(float x) { float r = 1.0f / x; int b; memcpy(&b, &r, 4);\n'
                '  b += %d; memcpy(&r, &b, 4); return r; }\n'
                '#define ASORA_QD_SEED(x) off(x)\n#include "%s/quick_div.cuh"\n'
                'extern "C" double qdiv(double a, double b) { return asora::quick_div(a, b); }\n'
                'extern "C" double qrec(double b) { return asora::quick_recip(b); }\n'
                % (request.param, CSRC))
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", src,
                    "-o", lib], check=True)
    so = C.CDLL(lib)
    so.qdiv.restype, so.qdiv.argtypes = C.c_double, [C.c_double] * 2
    so.qrec.restype, so.qrec.argtypes = C.c_double, [C.c_double]
    return so


def _close(got, exact):
    """Within half a unit in the last place, and 2^-30 of one for the error before rounding."""
    ulp = Fraction(2) ** (frexp(float(exact))[1] - 53)
    return abs(Fraction(got) - exact) <= ulp * (Fraction(1, 2) + Fraction(1, 2 ** 30))


def _mantissas(rng):
    edge = [0, 1, 2, 2 ** 52 - 1, 2 ** 52 - 2, 2 ** 51, 2 ** 29, 2 ** 29 - 1, 2 ** 52 - 2 ** 29,
            2 ** 52 - 2 ** 28, 2 ** 52 - 2 ** 30 + 1]
    return edge + [rng.getrandbits(52) for _ in range(3000)]


def test_quotients_round_like_the_exact_ones(lib):
    rng = random.Random(5)
    for mb in _mantissas(rng):
        b = ldexp(1 + mb / 2 ** 52, rng.randint(-399, 398))
        assert _close(lib.qrec(b), 1 / Fraction(b)), b
        for ma in (0, 2 ** 52 - 1, rng.getrandbits(52)):
            a = ldexp(1 + ma / 2 ** 52, rng.randint(-399, 398))
            assert _close(lib.qdiv(a, b), Fraction(a) / Fraction(b)), (a, b)
        assert lib.qdiv(b, b) == 1.0 and lib.qdiv(0.0, b) == 0.0


@pytest.mark.parametrize("a", [0.0, -0.0, 1.0, -3.0, 5e-324, 1e-310, 1e-130, 1e130, 1.7e308, inf,
                               -inf, nan])
def test_everything_else_as_the_plain_quotient(lib, a):
    for b in (1.0, 3.0, -7.0, 5e-324, 1e-310, 1e-200, 1e200, 1.7e308, inf, -inf, nan):
        want, got = C.c_double(a).value / b, lib.qdiv(a, b)
        assert (isnan(want) and isnan(got)) or want == got, (a, b)
        want, got = 1.0 / b if b else inf, lib.qrec(b)
        assert (isnan(want) and isnan(got)) or want == got, b
