"""Which images are aligned to a common exponent, and the sums formed on them
(csrc/fxsum.cuh, built here for the host), for every operator that uses them: a
set of values is aligned exactly when that loses no bit of any of them, each
value counting by itself, and then every sum is the exact one rounded once --
so never further from it than the sums that are formed otherwise."""
import os
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
COUNT = {"h": 7, "l": 7, "m": 5, "r": 32}
GUARD = {"h": 7, "l": 6, "m": 7, "r": 4}  # 63 - 53 - headroom of weights 6, 12, 8, 48


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    e = str(tmp_path_factory.mktemp("fxspan") / "fxspan_host")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-o", e, os.path.join(ROOT, "tests", "fxspan_host.cpp")],
                   check=True)
    return e


def expo(x):
    return (struct.unpack("<Q", struct.pack("<d", x))[0] >> 52) & 0x7FF


def exact(op, x):
    x = [Fraction(float(v)) for v in x]
    if op == "r":
        return [sum(x[:8]) / 8, (sum(x[8:]) - 3 * sum(x[:8])) / 8]
    return [sum(x[1:]) - (0 if op == "h" else len(x) - 1) * x[0]]


def run(exe, op, cases):
    inp = "\n".join(op + " " + " ".join("%016x" % struct.unpack("<Q", struct.pack("<d", v))[0] for v in x) for x in cases)
    out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout.splitlines()
    for x, line in zip(cases, out):
        E, *v = line.split()
        v = [struct.unpack("<d", struct.pack("<Q", int(b, 16)))[0] for b in v]
        n = len(v) // 2
        yield x, int(E), v[:n], v[n:]


@pytest.mark.parametrize("op", "hlmr")
@pytest.mark.parametrize("spread", [0, 1, 3, 4, 5, 6, 7, 8, 12])
def test_exact_or_not_aligned(exe, op, spread):
    rng = np.random.default_rng([ord(op), spread])
    n, cases = COUNT[op], []
    for k in range(600):
        x = rng.uniform(1, 2, n) * 2.0 ** -rng.integers(0, spread + 1, n) * rng.choice([-1, 1], n)
        if k % 3 == 0:  # one large value, all others `spread` bits below it
            x = rng.uniform(1, 2, n) * 2.0 ** -spread * rng.choice([-1, 1], n)
            x[rng.integers(0, n)] = 1.5
        if k % 4 == 1:  # nearly cancelling, as in a converged solution
            x = x[0] * (1 + 1e-6 * rng.normal(size=n))
        if k % 7 == 0:
            x[rng.integers(0, n)] = 0.0
        if k % 11 == 0:
            x[rng.integers(0, n)] = 5e-324
        cases.append(x * 2.0 ** int(rng.integers(-300, 300)) if k % 11 else x)
    aligned = 0
    for x, E, sums, plain in run(exe, op, cases):
        e = [expo(float(v)) for v in x if abs(v) > 1e-310]
        fits = max(e) - min(e) <= GUARD[op]
        assert E == (max(e) if fits else -1), (x, E)
        if not fits:
            continue
        aligned += 1
        for got, old, want in zip(sums, plain, exact(op, x)):
            if any(0 < abs(v) < 1e-310 for v in x):  # below every guard bit: dropped
                assert abs(Fraction(got) - want) <= Fraction(2) ** (max(expo(got), 1) - 1075) / 2 + Fraction(1e-320)
                continue
            assert got == float(want)  # Fraction -> float rounds to nearest even
            assert abs(Fraction(got) - want) <= abs(Fraction(old) - want)
    assert aligned > 100  # the nearly cancelling ones fit at any spread


@pytest.mark.parametrize("op", "hlmr")
def test_a_small_value_beside_a_large_one(exe, op):
    """Each value counts, not the larger one of a pair; and the ends of the exponent range."""
    n = COUNT[op]
    for at in range(n):
        for small, fits in ((1e-12, False), (1e-19, False), (2.0 ** -GUARD[op], True), (2.0 ** -GUARD[op] * 0.999, False)):
            x = np.ones(n)
            x[at] = small
            (_, E, _, _), = run(exe, op, [x])
            assert E == (1023 if fits else -1)
    for scale, E in ((2.0 ** (64 - 1023), 64), (2.0 ** (63 - 1023), -1), (2.0 ** (2040 - 1023), 2040), (2.0 ** (2041 - 1023), -1),
                     (0.0, -1), (np.inf, -1), (np.nan, -1)):
        (_, got, _, _), = run(exe, op, [scale * np.ones(n)])
        assert got == E, scale
