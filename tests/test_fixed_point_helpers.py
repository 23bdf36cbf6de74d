"""The integer helpers of the FP64 step's fixed-point sums, compiled for the host, against Python's integers:
a term of a node's force is a sum that fits63 accepts (up to 2^63 - 1 in magnitude), shifted right by the
difference of two exponents and rounded, halves away from zero."""
import ctypes
import os
import random
import subprocess

import pytest

from conftest import ROOT

SRC = """
#include "hmc_fixed.h"
extern "C" long long rshift_(long long x, int n) { return hmc::rshift(x, n); }
extern "C" int fits63_(int t) { return hmc::fits63(t); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "f.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_1009_0457_gb300", "csrc"),
                    str(d / "f.cpp"), "-o", str(d / "f.so")], check=True)
    lib = ctypes.CDLL(str(d / "f.so"))
    lib.rshift_.argtypes, lib.rshift_.restype = [ctypes.c_longlong, ctypes.c_int], ctypes.c_longlong
    return lib


def _nearest(x, n):
    q = (abs(x) + (1 << n >> 1)) >> n
    return q if x >= 0 else -q


@pytest.mark.parametrize("n", [-3, 0, 1, 2, 17, 38, 39, 53, 60, 61, 62, 63, 64, 65, 90, 2046])
def test_rounded_shift(lib, n):
    rng = random.Random(n)
    top = (1 << 63) - 1
    xs = [0, 1, top, top - 1, top - (1 << 38), 1 << 62, (1 << 62) - 1, (1 << 62) + 1, int(2 ** 62.3)]
    if 0 < n < 64:
        half = 1 << (n - 1)
        xs += [half, half - 1, half + 1, 3 * half, 3 * half - 1, 3 * half + 1, top // half * half]
    xs += [rng.getrandbits(rng.randint(1, 63)) for _ in range(2000)]
    for x in xs:
        if x > top:
            continue
        for y in (x, -x):
            assert lib.rshift_(y, n) == (_nearest(y, n) if n > 0 else y), (y, n)


def test_accepted_sums_fit(lib):
    rng = random.Random(1)
    edge, lim = 0, (1 << 63) - 1
    for _ in range(40000):
        k = rng.choice([2, 4])
        aim = rng.choice([-1, 1]) * (lim + rng.randint(-(1 << 39), 1 << 39))
        xs = [rng.randint(-(1 << 62), 1 << 62) for _ in range(k - 1)]
        xs.append(aim - sum(xs))
        if abs(xs[-1]) > lim:
            continue
        fits = bool(lib.fits63_(sum(x >> 35 for x in xs)))
        assert not fits or abs(sum(xs)) <= lim
        assert fits or abs(sum(xs)) > lim - 9 * (1 << 35)      # and refuses none that is clear of the edge
        edge += fits
    assert edge > 1000
    # the lowest sum, -2^63, would have no magnitude
    assert not lib.fits63_(-(1 << 28)) and lib.fits63_(-(1 << 28) + 1)
