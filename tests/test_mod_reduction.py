"""The residue reduction of the FP64 products (csrc/mod_arith.h), compiled for the host: every
integer an exact fp32 sum can hold, for each modulus."""
import math
import os
import shutil
import subprocess
from itertools import combinations

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_08990_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "mod_arith.h"
using namespace dme;
int main() {
    for (int m = 0; m < MOD_NM; ++m) {
        const int p = kModuli[m];
        const float inv = 1.0f / (float)p;
        long wrong = 0;
        float lo = 1e9f, hi = -1e9f;
        for (int x = -(1 << 24); x <= (1 << 24); ++x) {
            const float r = mod_centred((float)x, (float)p, inv);
            if ((x - (int)r) % p != 0) ++wrong;
            lo = r < lo ? r : lo;
            hi = r > hi ? r : hi;
        }
        std::printf("%d %ld %g %g\n", p, wrong, lo, hi);
    }
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("needs a C++ compiler")
    d = tmp_path_factory.mktemp("mod")
    (d / "m.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(d / "m.cpp"), "-o", str(d / "m")], check=True)
    out = subprocess.run([str(d / "m")], check=True, capture_output=True, text=True).stdout
    return [[float(v) for v in line.split()] for line in out.splitlines()]


def test_every_sum_reduces_to_a_byte(rows):
    assert len(rows) == 16
    for p, wrong, lo, hi in rows:
        assert wrong == 0, p
        # a byte holds -128 .. 127; 128 stands for -128 modulo 256 only
        assert -128 <= lo and hi <= (128 if p == 256 else 127), (p, lo, hi)


def test_moduli_span_the_outputs(rows):
    moduli = [int(r[0]) for r in rows]
    assert all(math.gcd(a, b) == 1 for a, b in combinations(moduli, 2))
    assert math.prod(moduli) >= 8 * 2 ** 122
