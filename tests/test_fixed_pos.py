"""Host check of the FP64 binning positions (csrc/fixed_pos.h): the integer
arithmetic on the bits of t against exact rational arithmetic, over zeros,
subnormals, every shift, rounding ties either way, the last node and values
that must be refused."""
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1508_02766_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include "fixed_pos.h"
int main() {
  unsigned long long t, top;
  while (std::scanf("%llx %llx", &t, &top) == 2) {
    uint64_t V = 0;
    const bool in = kde::fixed_position(t, top, &V);
    std::printf("%d %llu\n", (int)in, (unsigned long long)V);
  }
  return 0;
}
"""


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _cases():
    rng = np.random.default_rng(3)
    out = []
    for M in (2, 3, 128, 2001, 4097, 1 << 24):
        top = float(M - 1)
        t = list(rng.uniform(0, top, 200)) + list(np.exp(rng.uniform(-60, np.log(top), 200)))
        for i in {0, 1, M // 2, M - 2, M - 1}:
            for f in (0.0, 2.0 ** -33, 2.0 ** -32, 3 * 2.0 ** -33, 2.0 ** -34, 0.5, 1 - 2.0 ** -33,
                      1 - 2.0 ** -32, 1 - 3 * 2.0 ** -33):
                v = i + f
                t += [v, np.nextafter(v, np.inf), np.nextafter(v, -np.inf)]
        t += [0.0, -0.0, 5e-324, -5e-324, 2.0 ** -1022, -1.0, -1e300, top, np.nextafter(top, np.inf),
              1e300, np.inf, -np.inf, np.nan, -np.nan]
        out += [(float(v), top) for v in t]
    return out


def _expected(t, top):
    if not (0 <= t <= top):
        return 0, 0
    v = Fraction(t) * 2 ** 32
    r = v.numerator // v.denominator
    rest = v - r
    return 1, r + (rest > Fraction(1, 2) or (rest == Fraction(1, 2) and r % 2 == 1))


def test_positions_are_exactly_rounded(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROG)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    cases = _cases()
    text = "\n".join("%x %x" % (_bits(t), _bits(top)) for t, top in cases)
    got = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout
    for (t, top), line in zip(cases, got.splitlines(), strict=True):
        assert tuple(map(int, line.split())) == _expected(t, top), (t, top)
