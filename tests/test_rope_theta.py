"""The rotary frequencies that every call forms on the host, against 50-digit arithmetic."""
import ctypes as C
import decimal
import math
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rope_theta(tmp_path_factory):
    d = tmp_path_factory.mktemp("theta")
    src, so = d / "theta.cpp", d / "theta.so"
    src.write_text('#include "rope_theta.h"\nextern "C" void rope_theta(double b, int d, double* t) { ads_rope_theta(b, d, t); }\n')
    subprocess.run(["g++", "-O3", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2605_03644_b200", "csrc"),
                    str(src), "-o", str(so)], check=True)
    fn = C.CDLL(str(so)).rope_theta
    fn.argtypes, fn.restype = [C.c_double, C.c_int, C.POINTER(C.c_double)], None

    def run(base, d):
        t = (C.c_double * (d // 2))()
        fn(base, d, t)
        return list(t)
    return run


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("base", [1e4, 5e5, 1e6, 7e6, 500000.1, 1.0, 1.7, 0.3, 1e-99, 9.9e99])
def test_frequencies_are_the_nearest_doubles(rope_theta, base, d):
    # every product is good to some 2^-100, so only a value that close to the middle of two doubles could be rounded the other way
    with decimal.localcontext() as ctx:
        ctx.prec = 50
        for i, got in enumerate(rope_theta(base, d)):
            want = decimal.Decimal(base) ** (decimal.Decimal(-2 * i) / d)
            assert abs(decimal.Decimal(got) - want) <= decimal.Decimal(0.5000001 * math.ulp(got)), (base, d, i)


@pytest.mark.parametrize("base,d", [(0.0, 64), (-3.0, 64), (1e150, 128), (1e-150, 64), (math.inf, 64), (math.nan, 128), (1e4, 96)])
def test_other_bases_and_sizes_are_what_pow_gives(rope_theta, base, d):
    pow_ = C.CDLL(None).pow
    pow_.argtypes, pow_.restype = [C.c_double, C.c_double], C.c_double
    for i, got in enumerate(rope_theta(base, d)):
        want = pow_(base, -2.0 * i / d)
        assert got == want or (math.isnan(got) and math.isnan(want))
