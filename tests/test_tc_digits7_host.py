"""The seven-digit arithmetic of the tensor-core row stages above degree 39 (csrc/tc_digits.cuh) on the host, against
exact rational arithmetic: digit bounds, reconstruction of split values, recombination of the seven diagonal sums, and a
whole product with the shape of the folded Fourier stage and of the Legendre stage at degree 64."""
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1811_10270_gb300", "csrc")
ND = 7


@pytest.fixture(scope="module")
def tcd(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("tcd7") / "tc_digits7_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I" + CSRC,
                    os.path.join(HERE, "native", "tc_digits7_check.cpp"), "-o", exe], check=True)

    def go(lines):
        return subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True,
                              check=True).stdout.strip().splitlines()
    return go


def split_df(x):
    h = float(np.float32(x))
    return h, float(np.float32(x - h))


def row_digits(tcd, pairs):
    return [list(map(int, s.split())) for s in tcd(["D %s %s" % (h.hex(), l.hex()) for h, l in pairs])]


def test_row_digits(tcd):
    rng = np.random.default_rng(5)
    xs = rng.choice([-1.0, 1.0], 4000) * 2.0 ** rng.uniform(-35, 7, 4000) * rng.uniform(0.5, 1.0, 4000)
    pairs = [p for p in map(split_df, xs) if abs(p[0]) < 128.0]
    for (h, l), d in zip(pairs, row_digits(tcd, pairs)):
        assert abs(d[6]) <= 128 and abs(d[5]) <= 64 and abs(d[4]) <= 64 and abs(d[3]) <= 72
        assert max(map(abs, d[:3])) <= 65
        val = sum(Fraction(d[j]) * Fraction(2) ** (7 * (j - 6)) for j in range(ND))
        # half a unit of the last digit, and the remainder's rounding below the fourth
        assert abs(val - (Fraction(h) + Fraction(l))) <= Fraction(1, 2 ** 43) + Fraction(1, 2 ** 46)


def test_table_digits(tcd):
    rng = np.random.default_rng(6)
    xs = rng.uniform(-1.0, 1.0, 2000)
    for x, s in zip(xs, tcd(["H %s 0" % float(x).hex() for x in xs])):
        d = list(map(int, s.split()))
        assert max(map(abs, d[:6])) <= 64 and abs(d[6]) <= 128
        val = sum(Fraction(d[j]) * Fraction(2) ** (7 * (j - 7)) for j in range(ND))
        assert abs(val - Fraction(float(x))) <= Fraction(1, 2 ** 50)


@pytest.mark.parametrize("K", [66, 80, 130, 144])
def test_digit_product(tcd, K):
    """One output of a K-term product: exact diagonal sums below 2^24, the result within 2^-46 of the sum of magnitudes
    (28 of the 49 digit products; the neglected ones are below 2^-49 each, six diagonals of them)."""
    rng = np.random.default_rng(K)
    worst = 0.0
    for trial in range(20):
        x = rng.standard_normal(K) * 2.0 ** rng.uniform(-20, 0, K)
        t = np.cos(rng.uniform(0, 2 * math.pi, K))
        e = int(np.frexp(np.abs(x).max())[1])
        pairs = [split_df(v) for v in x]
        rd = row_digits(tcd, [(h * 2.0 ** (7 - e), l * 2.0 ** (7 - e)) for h, l in pairs])
        td = [list(map(int, s.split())) for s in tcd(["H %s 1" % float(v).hex() for v in t])]
        acc = [0] * ND
        for a, b in zip(rd, td):
            for ja in range(ND):
                for jb in range(ND - 1 - ja, ND):
                    acc[ja + jb - (ND - 1)] += a[ja] * b[jb]
        assert max(map(abs, acc)) < 2 ** 24
        hi, lo = (float.fromhex(v) for v in tcd(["C " + " ".join(float(a).hex() for a in acc[::-1])])[0].split())
        got = (Fraction(hi) + Fraction(lo)) * Fraction(2) ** (e - 13)
        want = sum((Fraction(h) + Fraction(l)) * Fraction(float(v)) for (h, l), v in zip(pairs, t))
        scale = Fraction(2) ** e * K
        worst = max(worst, float(abs(got - want) / scale))
    assert worst <= 2.0 ** -46
