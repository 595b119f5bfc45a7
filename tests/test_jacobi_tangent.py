"""The Jacobi rotation's tangent (csrc/bbp_jacobi.h), compiled for the host,
against its root in 50 digits.  Its last Newton step rounds twice at t's own
scale: the inner product-sum c t + d, which the derivative 2 c t + d (same sign,
no smaller) carries over to t at most unchanged, and the step itself.  What the
steps leave of the FP32 root's error (1e-7 times 1e-7 twice) is below 1e-18, so
the bound is 2 u with u = 2^-53, stated here with a quarter more."""

import ctypes
import decimal
import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2402_04834_gb300", "csrc")
TOL = 2.25 * 2.0 ** -53


@pytest.fixture(scope="module")
def tangent(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("jacobi")
    src, lib = d / "t.cpp", d / "t.so"
    src.write_text('#include "bbp_jacobi.h"\n'
                   'extern "C" double tangent(double d, double c) { return bbp::jacobi_tangent(d, c); }\n')
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib),
                    str(src)], check=True)
    f = ctypes.CDLL(str(lib)).tangent
    f.argtypes, f.restype = [ctypes.c_double, ctypes.c_double], ctypes.c_double
    return f


# Squared norms with the larger in [1, 2), as the kernel scales them; the other
# close by, of any size down to the rounding floor, or equal.
@pytest.mark.parametrize("ratio", ["near", "any", "equal"])
def test_tangent_has_the_bits_of_fp64(tangent, ratio):
    rng = random.Random(11)
    with decimal.localcontext(decimal.Context(prec=50)):
        for _ in range(4000):
            a = rng.uniform(1.0, 2.0)
            b = a if ratio == "equal" else a * (1 - 10 ** rng.uniform(-14, 0)) if ratio == "near" else \
                a * 10 ** rng.uniform(-30, 0)
            if rng.random() < 0.5:
                a, b = b, a
            c = (a * b) ** 0.5 * 10 ** rng.uniform(-15, 0) * rng.choice((-1, 1))
            d = b - a
            D, C = decimal.Decimal(d), decimal.Decimal(c)
            s = (D * D + 4 * C * C).sqrt()
            want = 2 * C / (D + s) if D >= 0 else 2 * C / (D - s)      # the root of c t^2 + d t - c with |t| <= 1
            got = decimal.Decimal(tangent(d, c))
            if D == 0:
                assert abs(got) == 1
            else:
                assert abs(got - want) <= decimal.Decimal(TOL) * abs(want), (d, c)
