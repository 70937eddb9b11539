"""u^e in 64-bit fixed point (csrc/of_pow.cuh), compiled for the host and compared with decimal
arithmetic of 50 digits: 0.5 units in the last place from the rounding and 0.01 from the 2^-60 to
which the result is known before it (one unit is 2^-53 to 2^-52 of the value).
"""
import ctypes
import math
import subprocess
from decimal import Decimal, getcontext
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1412_8250_gb300" / "csrc"
SOURCE = """
#include "of_pow.cuh"
extern "C" int power(double u, double e, double* v) {
    const of::PowExp p = of::pow_exp(e);
    int k;
    long long f;
    return p.fixed != 0 && of::log2_fixed(u, k, f) && of::exp2_fixed(p, k, f, *v);
}
"""


@pytest.fixture(scope="module")
def power(tmp_path_factory):
    d = tmp_path_factory.mktemp("pow")
    (d / "p.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(CSRC), str(d / "p.cpp"), "-o",
                    str(d / "p.so")], check=True)
    f = ctypes.CDLL(str(d / "p.so")).power
    f.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.POINTER(ctypes.c_double)]

    def call(u, e):
        v = ctypes.c_double()
        return v.value if f(u, e, ctypes.byref(v)) else None
    return call


@pytest.mark.parametrize("e", [(5 + math.sqrt(5)) / 3, (5 - math.sqrt(5)) / 3, -0.8, 1.0, 15.75])
def test_power_is_rounded(power, e):
    getcontext().prec = 50
    rng = np.random.default_rng(1)
    us = list(np.exp(rng.uniform(math.log(1e-12), math.log(1e3), 300)))
    # powers of two and their neighbours, and the edges of the table's intervals
    for k in (-40, -1, 0, 1, 10):
        us += [2.0 ** k, np.nextafter(2.0 ** k, 0), np.nextafter(2.0 ** k, 1e300)]
    us += [2.0 ** ((j + 0.5) / 128) for j in range(128)]
    for u in us:
        v = power(float(u), e)
        ref = (Decimal(float(u)).ln() * Decimal(e)).exp()
        ulp = Decimal(math.ulp(float(ref)))
        assert abs(Decimal(v) - ref) <= Decimal("0.51") * ulp, (u, v)


def test_outside_the_range_is_left_to_pow(power):
    assert power(0.0, 0.9) is None and power(-1.0, 0.9) is None and power(math.inf, 0.9) is None
    assert power(math.nan, 0.9) is None and power(1e-30, 0.9) is None and power(2.0, 17.0) is None
    assert power(2.0, 1e-18) is None and power(2.0, 0.0) is None
