"""Sums on images aligned to a common exponent (csrc/fxsum.cuh, built here for
the host) against exact rationals: the error is at most the truncated bits,
one unit of 2^-6 ulp of the image's largest exponent per unit of weight (12),
and half an ulp of the result; sums without truncated bits are rounded to
nearest, ties to even.  fx_to_float equals the FP64 conversion bit for bit."""
import os
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    e = str(tmp_path_factory.mktemp("fximage") / "fximage_host")
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", e, os.path.join(ROOT, "tests", "fximage_host.cpp")], check=True)
    return e


def bits(x):
    return "%016x" % struct.unpack("<Q", struct.pack("<d", x))[0]


def expo(x):
    return (struct.unpack("<Q", struct.pack("<d", x))[0] >> 52) & 0x7FF


@pytest.mark.parametrize("spread", [0, 1, 4, 8])
def test_sums(exe, spread):
    rng = np.random.default_rng(40 + spread)
    cases = []
    for n in range(3000):
        x = rng.uniform(1, 2, 7) * 2.0 ** rng.integers(-spread, 1, 7) * rng.choice([-1, 1], 7)
        if n % 3 == 0:  # nearly cancelling, as in a converged solution
            x = x[0] * (1 + 1e-6 * rng.normal(size=7))
        if n % 7 == 0:
            x[rng.integers(0, 7)] = 0.0
        x *= 2.0 ** int(rng.integers(-300, 300))
        cases.append((max(expo(v) for v in x) + int(rng.integers(0, spread + 1)), x))
    inp = "\n".join("%d %s" % (E, " ".join(bits(v) for v in x)) for E, x in cases)
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout.split()
    for (E, x), o in zip(cases, out):
        got = Fraction(struct.unpack("<d", struct.pack("<Q", int(o, 16)))[0])
        want = sum(Fraction(float(v)) for v in x[1:]) - 6 * Fraction(float(x[0]))
        unit = Fraction(2) ** (E - 1075 - 6)
        ulp = Fraction(2) ** (max(expo(float(got)), 1) - 1075)
        assert abs(got - want) <= 12 * unit + ulp / 2
        if all((Fraction(float(v)) / unit).denominator == 1 for v in x):
            assert float(got) == float(want)  # Fraction -> float rounds to nearest even


def test_to_float(exe):
    rng = np.random.default_rng(7)
    x = np.concatenate([rng.normal(size=2000), rng.normal(size=500) * 10.0 ** rng.integers(-60, 60, 500),
                        rng.integers(0, 2 ** 63, 500, dtype=np.uint64).view(np.float64),
                        [0.0, -0.0, 1e-45, 2 ** -126, 3.4028235677973366e38, np.inf, -np.inf, 1 + 2 ** -24, 1 + 3 * 2 ** -24,
                         2 ** -126 - 2 ** -151, 1e300]])
    x = x[~np.isnan(x)]
    out = subprocess.run([exe, "f"], input="\n".join(bits(v) for v in x), capture_output=True, text=True,
                         check=True).stdout.split()
    with np.errstate(all="ignore"):
        want = x.astype(np.float32).view(np.uint32)
    assert [int(o, 16) for o in out] == [int(w) for w in want]


def test_to_double(exe):
    rng = np.random.default_rng(8)
    x = rng.integers(0, 2 ** 32, 4000, dtype=np.uint32).view(np.float32)
    x = np.concatenate([x[~np.isnan(x)], np.array([0.0, -0.0, 1e-45, 1.17549435e-38, np.inf, -np.inf], np.float32)])
    inp = "\n".join("%08x" % v for v in x.view(np.uint32))
    out = subprocess.run([exe, "d"], input=inp, capture_output=True, text=True, check=True).stdout.split()
    assert [int(o, 16) for o in out] == [int(w) for w in x.astype(np.float64).view(np.uint64)]
