"""The register transforms' compile-time twiddles against 50-digit arithmetic:
each constant is the double nearest to its cosine or sine, for every length up
to 32 and the longer compiled ones.  A host program prints them."""
import os
import shutil
import subprocess
from decimal import Decimal, getcontext

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_06237_gb300", "csrc")
LENGTHS = list(range(1, 33)) + [40, 45, 48, 50]
PROGRAM = """
#include <cstdio>
#include <utility>
#include "%s"
template <int L, int... K>
void line(std::integer_sequence<int, K...>) {
  (std::printf("%%d %%d %%a %%a\\n", L, K, vie::TwConst<L, K>::c, vie::TwConst<L, K>::s), ...);
}
int main() {
%s
}
"""


def _cos_sin(k, L):
    """cos and sin of 2 pi k / L, |angle| <= pi, by their series."""
    getcontext().prec = 50
    pi = Decimal("3.14159265358979323846264338327950288419716939937510582097494459")
    x = 2 * pi * (k if 2 * k <= L else k - L) / L
    out = []
    for n, term in ((0, Decimal(1)), (1, x)):
        total = term
        while abs(term) > Decimal("1e-45"):
            term *= -x * x / ((n + 1) * (n + 2))
            n += 2
            total += term
        out.append(total)
    return out


def test_constants_are_the_nearest_doubles(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "twiddles.cpp"
    src.write_text(PROGRAM % (os.path.join(CSRC, "twiddle.cuh"),
                              "\n".join("  line<%d>(std::make_integer_sequence<int, %d>{});" % (L, L) for L in LENGTHS)))
    exe = tmp_path / "twiddles"
    subprocess.run([cxx, "-std=c++17", "-x", "c++", str(src), "-o", str(exe)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    seen = 0
    for text in filter(None, lines):
        L, k, c, s = text.split()
        cos, sin = _cos_sin(int(k), int(L))
        for got, exact in ((float.fromhex(c), cos), (float.fromhex(s), -sin)):
            # the nearest double; where the exact value is zero the series ends at 1e-45
            assert got == float(exact) or (got == 0.0 and abs(exact) < Decimal("1e-40")), (L, k, got)
        seen += 1
    assert seen == sum(LENGTHS)
