"""The error bound of a difference of FP32 pairs (the window statistics decide by
it which windows are evaluated from their samples), against exact rational
arithmetic: the code itself, compiled for the host."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "fp_pair.cuh"
#include <cstdio>
using namespace dtws;
int main() {
    f2 x, y;
    while (scanf("%a %a %a %a", &x.hi, &x.lo, &y.hi, &y.lo) == 4) {
        float err;
        const f2 d = f2_diff(x, y, err);
        printf("%a %a %a\n", d.hi, d.lo, err);
    }
}
"""


def _store(v):
    """The pair that stores a number: hi its nearest float, lo the rest's."""
    hi = np.float32(float(v))  # (v has at most 53 bits)
    return hi, np.float32(float(v - Fraction(float(hi))))


def test_a_difference_stays_within_its_bound(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I" + os.path.join(ROOT, "paper_1812_10302_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    rng = np.random.default_rng(1)
    pairs = []
    for _ in range(30000):  # numbers near and far, of either sign, low parts near their largest, just below a power of two
        X = Fraction(float(rng.choice([1.0, 2.0, 1.99999994, 1.5, 1.0000001]) * (1 + rng.uniform(-2.0 ** -22, 2.0 ** -22))))
        Y = X * Fraction(float(rng.choice([1.0, -1.0, 0.5, 0.999999, 0.25]))) + Fraction(float(rng.uniform(-1, 1) * 2.0 ** rng.uniform(-40, 0)))
        pairs.append((Fraction(float(X)), Fraction(float(Y))))
    text = ""
    for X, Y in pairs:
        text += " ".join(float(v).hex() for v in (*_store(X), *_store(Y))) + "\n"
    out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout.split("\n")
    worst = tight = 0.0
    for (X, Y), line in zip(pairs, out):
        hi, lo, bound = (Fraction(float.fromhex(t)) for t in line.split())
        err = abs(hi + lo - (X - Y)) * 2 ** 48
        assert err <= bound, (float(X), float(Y), float(err), float(bound))
        worst = max(worst, float(err / (abs(X) + abs(Y))))
        tight = max(tight, float(err / bound))
    assert worst > 1.5  # (a bound of 1.5 times |X| + |Y|, which stood here, does not hold)
    assert tight > 0.7  # (nor does one much below it)
    print("largest error:", worst, "x 2^-48 (|X| + |Y|),", tight, "of its bound")
