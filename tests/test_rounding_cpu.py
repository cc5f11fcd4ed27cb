"""The test whether a CG quotient's float is certain (csrc/rounding.h), against
exact rational arithmetic: wherever it says yes, every quotient within the stated
relative bound rounds to that float.  No tolerance."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2407_20026_gb300", "csrc")
BOUND = Fraction(93, 100) / 2**34


@pytest.fixture(scope="module")
def certain(tmp_path_factory):
    d = tmp_path_factory.mktemp("rounding")
    src = d / "r.cpp"
    src.write_text('#include "rounding.h"\n'
                   'extern "C" int certain(float f, float rest) '
                   '{ return sso::quotient_certain(f, rest); }\n')
    lib = d / "r.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).certain
    fn.argtypes = [ctypes.c_float, ctypes.c_float]
    return lambda f, rest: bool(fn(f, rest))


@pytest.mark.parametrize("lo,hi", [(0.5, 0.75), (0.75, 1.0), (1.0, 1.25), (1.25, 2.0)])
def test_certain_quotients_round_to_their_float(certain, lo, hi):
    rng = np.random.default_rng(int(8 * lo))
    last = 2.0**-24 if hi <= 1.0 else 2.0**-23  # a unit of f's last place
    yes = 0
    for _ in range(400):
        f = np.float32(rng.uniform(lo, hi))
        if float(f) in (0.5, 1.0) or float(f) >= hi:
            continue
        # what f leaves, close to half of that unit, on either side
        rest = np.float32((last / 2 - 2.0**-36 * rng.uniform(0, 16)) * rng.choice([-1, 1]))
        if not certain(f, rest):
            continue
        yes += 1
        q = Fraction(float(f)) + Fraction(float(rest))
        for e in (q * (1 - BOUND), q * (1 + BOUND)):
            assert abs(e - Fraction(float(f))) < Fraction(last) / 2, (float(f), float(rest))
    assert yes > 50 and certain(np.float32(lo + 0.1), np.float32(0.0))
