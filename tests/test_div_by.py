"""The division step of the Lanczos vectors (csrc/div_by.h), compiled for the host,
against exact quotients: within 1/2 ulp and 2^-50 of one."""
import ctypes as C
import os
import random
import subprocess
from fractions import Fraction
from math import ulp

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_08523_gb300", "csrc")


@pytest.fixture(scope="module")
def div_by(tmp_path_factory):
    d = tmp_path_factory.mktemp("div")
    src, so = str(d / "div.cc"), str(d / "div.so")
    with open(src, "w") as f:
        f.write('#include "div_by.h"\nextern "C" double q(double w, double b) '
                '{ const double r = 1.0 / b; return ftsp2::div_by(w, b, r); }\n')
    # products that the header writes apart stay apart, as in nvcc's rounding of w * r
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    f = C.CDLL(so).q
    f.restype, f.argtypes = C.c_double, [C.c_double, C.c_double]
    return f


def check(div_by, w, b):
    got, exact = div_by(w, b), Fraction(w) / Fraction(b)
    bound = (Fraction(1, 2) + Fraction(1, 2 ** 50)) * Fraction(ulp(float(exact)))
    assert abs(Fraction(got) - exact) <= bound, (w, b, got)


def test_against_exact_quotients(div_by):
    r = random.Random(5)
    betas = [1e-12, 1.0000000000000002e-12, 0.5, 1.0, 1.9999999999999998, 3.0, 1e3, 1e38, 1e-38]
    betas += [r.uniform(1.0, 2.0) * 2.0 ** r.randint(-40, 40) for _ in range(3000)]
    for b in betas:
        for w in (b, -b, b * (1 - 2.0 ** -53), b * (1 + 2.0 ** -52), r.uniform(-1, 1) * b, r.uniform(-1, 1),
                  r.uniform(-1, 1) * 1e-200, 5e-250):
            check(div_by, w, b)


def test_quotients_beside_a_midpoint(div_by):
    # w = the number next to (q + 1/2 ulp) b: quotients a hair off the middle of two numbers
    r = random.Random(6)
    for _ in range(3000):
        b, q = r.uniform(1.0, 2.0), r.uniform(1.0, 2.0)
        w = float((Fraction(q) + Fraction(ulp(q)) / 2) * Fraction(b))
        check(div_by, w, b)


def test_zero(div_by):
    assert div_by(0.0, 3.7) == 0.0 and div_by(-0.0, 1e-12) == 0.0
