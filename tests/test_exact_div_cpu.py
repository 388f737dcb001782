"""Quotients that have to have the bits of a / b (exact_div and exact_recip of
quick_div.cuh), compiled for the host with seeds as far off as the hardware's may be: next to
rounding ties and everywhere else."""
import ctypes as C
import os
import random
import subprocess
from math import inf, isnan, ldexp, nan

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2311_01492_gb300", "csrc")


@pytest.fixture(scope="module", params=[-1, 0, 1])  # units in the last place of the seed
def lib(request, tmp_path_factory):
    d = tmp_path_factory.mktemp("exact_div")
    src, lib = str(d / "s.cpp"), str(d / "s.so")
    with open(src, "w") as f:
        f.write('#include <math.h>\n#include <string.h>\n'
                'static float off(float x) { float r = 1.0f / x; int b; memcpy(&b, &r, 4);\n'
                '  b += %d; memcpy(&r, &b, 4); return r; }\n'
                '#define ASORA_QD_SEED(x) off(x)\n#include "%s/quick_div.cuh"\n'
                'extern "C" double qdiv(double a, double b) { return asora::exact_div(a, b); }\n'
                'extern "C" double qrec(double b) { return asora::exact_recip(b); }\n'
                % (request.param, CSRC))
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", src,
                    "-o", lib], check=True)
    so = C.CDLL(lib)
    so.qdiv.restype, so.qdiv.argtypes = C.c_double, [C.c_double] * 2
    so.qrec.restype, so.qrec.argtypes = C.c_double, [C.c_double]
    return so


def near_ties(B, most=40):
    """Numerators a (53 bits) for which a / B (B odd, 53 bits) is d / (2^54 B) away from a
    number of 54 bits, halfway between two doubles, for small odd d."""
    out = []
    for d in range(1, most, 2):
        for sign in (1, -1):
            M = sign * d * pow(B, -1, 2 ** 54) % 2 ** 54  # B M = sign d (mod 2^54)
            a = (B * M - sign * d) >> 54
            if M >> 53 and a >> 52 == 1:
                out.append(a)
    return out


def test_bits_of_the_quotient_next_to_ties(lib):
    rng = random.Random(7)
    bs = [int(ldexp(6.3e-18, 110)) | 1, 2 ** 52 + 1, 2 ** 53 - 1]
    bs += [2 ** 52 | rng.getrandbits(52) | 1 for _ in range(1500)]
    n = 0
    for B in bs:
        for a in near_ties(B):
            for e in (0, rng.randint(-390, 390)):
                x, y = ldexp(a, -52 + e), ldexp(B, -52)
                assert lib.qdiv(x, y) == x / y, (x, y)
                n += 1
    assert n > 10000


def test_bits_of_the_quotient_everywhere_else(lib):
    rng = random.Random(9)
    edge = [0, 1, 2, 3, 2 ** 52 - 1, 2 ** 52 - 2, 2 ** 51, 2 ** 29, 2 ** 29 - 1, 2 ** 52 - 2 ** 29]
    ms = edge + [rng.getrandbits(52) for _ in range(2000)]
    for mb in ms:
        b = ldexp(1 + mb / 2 ** 52, rng.randint(-399, 398))
        assert lib.qrec(b) == 1.0 / b, b
        for ma in (0, 1, 2 ** 52 - 1, mb, max(mb - 1, 0), min(mb + 1, 2 ** 52 - 1), rng.getrandbits(52)):
            a = ldexp(1 + ma / 2 ** 52, rng.randint(-399, 398))
            assert lib.qdiv(a, b) == a / b, (a, b)
        assert lib.qdiv(0.0, b) == 0.0


@pytest.mark.parametrize("a", [0.0, -0.0, 1.0, -3.0, 5e-324, 1e-310, 1e-130, 1e130, 1.7e308, inf,
                               -inf, nan])
def test_out_of_the_range_as_the_plain_quotient(lib, a):
    for b in (1.0, 3.0, -7.0, 5e-324, 1e-310, 1e-200, 1e200, 1.7e308, inf, -inf, nan):
        want, got = a / b, lib.qdiv(a, b)
        assert (isnan(want) and isnan(got)) or want == got, (a, b)
        want, got = 1.0 / b, lib.qrec(b)
        assert (isnan(want) and isnan(got)) or want == got, b
