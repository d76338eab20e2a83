"""Whether a host operand is one block of page-locked memory (which the device then reads by itself): the decision of
rg_gemm_plan_host, compiled on its own and asked about blocks that a table stands for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "rg_internal.h"
#include <cstdio>
// two registrations with a hole between them: [4096, 8192) and [12288, 16384)
static bool block(uintptr_t p, uintptr_t* start, size_t* size) {
  for (uintptr_t at : {uintptr_t(4096), uintptr_t(12288)})
    if (p >= at && p < at + 4096) {
      *start = at;
      *size = 4096;
      return true;
    }
  return false;
}
int main() {
  unsigned long long p;
  long long bytes;
  while (std::scanf("%llu %lld", &p, &bytes) == 2) std::printf("%d\n", rg::in_one_block(p, bytes, block) ? 1 : 0);
}
"""

CASES = [
    (4096, 4096, 1),            # a whole registration
    (4098, 4094, 1),            # up to its last byte
    (8191, 1, 1),
    (4098, 4095, 0),            # one byte further
    (4096, 12288, 0),           # both ends are page-locked, the bytes between them are not
    (8000, 4300, 0),
    (8192, 1, 0),               # in the hole
    (4000, 200, 0),             # starts before it
    (12288, 2 ** 62, 0),
    (4096, 0, 0),
]


def test_one_block(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "block.cpp", tmp_path / "block"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2605_29752_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], input="".join(f"{p} {n}\n" for p, n, _ in CASES), text=True, check=True,
                         capture_output=True).stdout.split()
    assert [int(x) for x in out] == [want for _, _, want in CASES]
