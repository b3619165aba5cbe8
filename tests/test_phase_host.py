"""The inlet's fixed-point phase (host part) against exact rational arithmetic:
frac(1 / T) to FP64's relative 2^-100 or 2^-127, frac(phase / 2 pi) to 2^-63
and the 2^-104 relative error of the two-part 1 / 2 pi, for periods around and
far from powers of two, below one step, and phases of both signs."""
import os
import subprocess
from fractions import Fraction

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2108_08783_gb300", "csrc")
MAIN = r"""
#include "lbm_internal.h"
#include <cstdio>
#include <cstdlib>
int main(int c, char** v) {
  for (int i = 1; i + 1 < c; i += 2) {
    uint64_t h, l, o;
    lbm::fixed_phase(strtod(v[i], 0), strtod(v[i + 1], 0), &h, &l, &o);
    printf("%llu %llu %llu\n", (unsigned long long)h, (unsigned long long)l, (unsigned long long)o);
  }
}
"""
# 1 / 2 pi to 60 digits
INV_2PI = Fraction(159154943091895335768883763372514362034459645740456448747667, 10 ** 60)
CASES = [(4000.0, 0.0), (100003.0, 0.7), (1e6, -0.7), (2048.0, 3.0), (37.0, -1e-20), (1 / 3, 6.2),
         (0.3, 100.0), (1.0, -7.5), (0.1 + 1e9, 1e-18), (3.0, 2.0), (1e300, 1.0)]


def test_fixed_phase_is_exact_to_its_last_bits(tmp_path):
    src, exe = tmp_path / "p.cpp", str(tmp_path / "p")
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o",
                    exe], check=True)
    args = [repr(float(v)) for case in CASES for v in case]
    out = subprocess.run([exe, *args], check=True, capture_output=True, text=True).stdout.split()
    for k, (T, phase) in enumerate(CASES):
        hi, lo, off = (int(v) for v in out[3 * k:3 * k + 3])

        def away(got, want):  # distance modulo one period
            d = (got - want) % 1
            return min(d, 1 - d)

        inv = 1 / Fraction(T)
        assert away(Fraction((hi << 64) + lo, 1 << 128), inv) <= inv / 2 ** 100 + Fraction(1, 2 ** 127)
        ph = Fraction(phase) * INV_2PI
        assert away(Fraction(off, 1 << 64), ph) <= abs(ph) / 2 ** 104 + Fraction(1, 2 ** 63)
