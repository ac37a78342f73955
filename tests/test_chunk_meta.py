"""No chunk's metadata is there before one was written (CPU: the kernel's set-up helper run on the host)."""
import os
import subprocess

from conftest import ROOT
from paper_1503_06203_gb300 import builder

HARNESS = r"""
#include <stdio.h>
#include <string.h>
#include <memory>
#include "xe_dual.cuh"
int main() {
  std::unique_ptr<char[]> mem(new char[sizeof(xe::DualSmem) + 128]);
  char* p = mem.get() + (128 - reinterpret_cast<uintptr_t>(mem.get()) % 128) % 128;
  memset(p, 0xA7, sizeof(xe::DualSmem));  // what shared memory may hold
  xe::DualSmem& sm = *reinterpret_cast<xe::DualSmem*>(p);
  for (int k = 0; k < xe::kDualThreads; ++k) xe::clear_smem(sm, k, xe::kDualThreads);
  int flags = 0, sums = 0;
  for (const auto& m : sm.pmeta) flags |= m.flags;
  for (const int32_t v : sm.part[0]) sums |= v;
  for (const int32_t v : sm.part[1]) sums |= v;
  printf("%d %d %llx\n", flags, sums, (unsigned long long)sm.full[0]);
}
"""


def test_a_cta_starts_without_chunks_or_sums(tmp_path):
    src, exe = tmp_path / "h.cu", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run([builder._nvcc(), *builder.ARCH, "-std=c++17", "-I", builder.CSRC, "-I", os.path.join(ROOT, "include"),
                    "-o", str(exe), str(src)], check=True)
    # no kMetaValid and no operand offset in any buffer; the barriers after them untouched
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0", "0", "a7" * 8]
