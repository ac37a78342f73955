"""A chunk's metadata is read only after the wait for it succeeded (CPU: the kernel's helper run on the host)."""
import os
import subprocess

from conftest import ROOT
from paper_1503_06203_gb300 import builder

HARNESS = r"""
#include <stdio.h>
#include "xe_dual.cuh"
int main() {
  const int4 current = make_int4(0x201, 2, 3, 4), next = make_int4(0x301, 6, 7, 8);
  for (int arrives = 0; arrives < 2; ++arrives) {
    int waits = 0, reads = 0;
    bool ok = true;
    const int4 m = xe::next_meta(ok, current, [&] { ++waits; return arrives != 0; }, [&] { ++reads; return next; });
    printf("%d %d %d %d %d %d %d\n", ok, waits, reads, m.x, m.y, m.z, m.w);
  }
}
"""


def test_meta_of_a_chunk_that_never_came_is_not_read(tmp_path):
    src, exe = tmp_path / "h.cu", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run([builder._nvcc(), *builder.ARCH, "-std=c++17", "--extended-lambda", "-I", builder.CSRC, "-I",
                    os.path.join(ROOT, "include"), "-o", str(exe), str(src)], check=True)
    lines = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")
    assert lines[0] == f"0 1 0 {0x201} 2 3 4"  # the wait ran out: the current chunk's stays, nothing is read
    assert lines[1] == f"1 1 1 {0x301} 6 7 8"
