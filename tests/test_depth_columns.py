"""The depth table's entries from their columns (csrc/pcr_certified.cuh: table_columns, depth_entry), on the CPU,
against exact rational arithmetic: round half up of |S M| 2^(e - 150 + 40) in magnitude, zero and unusable from the
first entry that reaches 2^62."""
from __future__ import annotations

import math
import os
import subprocess
from fractions import Fraction

import pytest

from paper_1908_02681_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "pcr_certified.cuh"
int main(int argc, char** argv) {
  const double s = strtod(argv[1], nullptr), m = strtod(argv[2], nullptr), m3[4] = {m, -m, m, 0.0};
  pcr::DepthColumn col[3];
  int32_t e_max[3] = {0, 0, 0};
  __int128 b;
  if (!pcr::host::table_columns(s, m3, 0.0, col, e_max, &b)) { printf("refused\n"); return 0; }
  printf("%d %d %d\n", e_max[0], col[0].neg, col[1].neg);
  for (int e = 0; e < pcr::kTableExp; ++e) {
    unsigned long long f;
    const bool ok = pcr::depth_entry(col[0], e, &f);
    printf("%d %llu\n", ok ? 1 : 0, f);
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("columns")
    src, exe = d / "columns.cu", d / "columns"
    src.write_text(PROGRAM)
    subprocess.check_call([build.NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                           build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe)])
    return str(exe)


# LINEAR scales of ordinary views, METRIC, PIECEWISE nanometres; entries of magnitude 1, tiny, exact powers of two,
# 0, products of one bit and of 106 bits, and values whose shift is 0, just left and just right
@pytest.mark.parametrize("s", [2.0 ** 40 / 2999.9, 2.0 ** 40 / 9.9, 1000.0, 1e9, 1.0, 2.0 ** 90, math.nextafter(2.0, 0.0)])
@pytest.mark.parametrize("m", [0.0, -0.6180339887, 1.0, 1e-17, -2.0 ** -80, math.nextafter(1.0, 0.0), 3.75, 2.0 ** -52])
def test_entries(program, s, m):
    out = subprocess.run([program, s.hex(), m.hex()], capture_output=True, text=True, check=True).stdout.split("\n")
    want, exact = [], abs(Fraction(s) * Fraction(m))
    for e in range(256):
        v = exact * Fraction(2) ** ((e or 1) - 150 + 40)
        f = math.floor(v + Fraction(1, 2))
        want.append((1, f) if e < 255 and f < 2 ** 62 else (0, 0))
    usable = max(e for e in range(256) if want[e][0])
    if abs(s * m) >= 2.0 ** 80 or usable < 127:
        assert out[0] == "refused"
        return
    e_max, neg, neg1 = (int(x) for x in out[0].split())
    assert e_max == usable
    assert m == 0.0 or (neg, neg1) == ((1, 0) if m < 0 else (0, 1))
    assert [tuple(int(x) for x in line.split()) for line in out[1:257]] == want
