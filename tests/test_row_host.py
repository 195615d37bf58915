"""Host side of the row-segment kernels' index arithmetic: the header's
host-device functions, compiled into a small program that runs on the CPU."""
import os
import subprocess

import pytest

from paper_2103_10114_gb300 import agcm

PROGRAM = r"""
#include <cstdio>
#include "agcm_row.cuh"
using namespace agcm;
// Rows that are not 16-byte aligned: four columns a thread, a quarter of the
// segment apart.  Every own column is read once, no other is.
static int own_columns_once() {
  for (int H = 4; H <= 32; H += 4)
    for (int own = 1; own + 2 * H <= kRowB; ++own) {
      const int NTW = (own + 2 * H + 31) & ~31, tr = NTW >> 2;
      int seen[kRowB] = {};
      for (int cc = 0; cc < tr; ++cc)
        for (int e = 0; e < 4; ++e)
          if (own_columns(cc, tr, H, own) >> 8 * e & 128u) ++seen[cc + e * tr];
      for (int c = 0; c < NTW; ++c)
        if (seen[c] != (c >= H && c < H + own ? 1 : 0)) return printf("own_columns %d %d %d\n", H, own, c), 1;
    }
  return 0;
}
// A block holds the rows of as many levels as the row-segment ensemble has ever
// taken: 4449 in FP32, 1732 in FP64.
static int levels_of_a_block() {
  const size_t most = 227 * 1024;
  if (row_smem_bytes<float>(4449) > most) return puts("FP32 levels"), 1;
  if (row_smem_bytes<double>(1732) > most) return puts("FP64 levels"), 1;
  return 0;
}
int main() { return own_columns_once() | levels_of_a_block(); }
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("row_host")
    src, exe = d / "main.cu", d / "main"
    src.write_text(PROGRAM)
    subprocess.check_call(["nvcc", *agcm.ARCH, "-std=c++17", "-I", agcm._CSRC, "-o", str(exe), str(src)])
    return str(exe)


def test_row_arithmetic(program):
    r = subprocess.run([program], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
