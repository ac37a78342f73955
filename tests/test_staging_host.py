"""The staging copy of unaligned rows reads nothing outside the caller's frame (CPU: its 16-byte step run on the host)."""
import os
import subprocess

import pytest

from conftest import ROOT
from paper_1503_06203_gb300 import builder

# One frame [T][F][N] at `base` bytes past an aligned address, staged step by step; the
# frame's bytes are k * 37 + 11, its neighbours are absent: a load outside [0, bytes) ends the run with status 1.
HARNESS = r"""
#include <stdio.h>
#include <stdlib.h>
#include <vector>
#include "xe_corr.cuh"
static int64_t bytes;
static uint8_t at(int64_t o) {
  if (o < 0 || o >= bytes) {
    printf("byte %lld of a frame of %lld read\n", (long long)o, (long long)bytes);
    exit(1);
  }
  return (uint8_t)(o * 37 + 11);
}
int main(int argc, char** argv) {
  const int N = atoi(argv[1]), F = atoi(argv[2]), T = atoi(argv[3]), Np = (N + 15) / 16 * 16;
  const int64_t rows = (int64_t)T * F;
  bytes = rows * N;
  for (uint64_t base = 0; base < 16; ++base) {
    std::vector<uint4> buf(rows * Np / 16);
    uint8_t* got = reinterpret_cast<uint8_t*>(buf.data());
    for (int64_t row = 0; row < rows; ++row)
      for (int e0 = 0; e0 < Np; e0 += 16) {
        auto word = [base](int64_t o) {
          if ((base + o) & 3) exit(2);
          return at(o) | at(o + 1) << 8 | at(o + 2) << 16 | (uint32_t)at(o + 3) << 24;
        };
        auto byte = [](int64_t o) { return at(o); };
        const int live = N - e0 < 16 ? N - e0 : 16;
        if (row < xe::kEndRows || row >= rows - xe::kEndRows)  // (as the kernel)
          xe::stage_16<true>(base, row * N + e0, live, bytes, word, byte, got + row * Np + e0);
        else
          xe::stage_16<false>(base, row * N + e0, live, bytes, word, byte, got + row * Np + e0);
      }
    for (int64_t row = 0; row < rows; ++row)
      for (int e = 0; e < Np; ++e)
        if (got[row * Np + e] != (e < N ? at(row * N + e) : 0x88)) {
          printf("base %d row %lld byte %d: %02x\n", (int)base, (long long)row, e, got[row * Np + e]);
          return 1;
        }
  }
  return 0;
}
"""


def compiled(d, code):
    src, exe = d / "h.cu", d / "h"
    src.write_text(code)
    subprocess.run([builder._nvcc(), *builder.ARCH, "-std=c++17", "--extended-lambda", "-I", builder.CSRC, "-I",
                    os.path.join(ROOT, "include"), "-o", str(exe), str(src)], check=True)
    return str(exe)


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("staging"), HARNESS)


@pytest.mark.parametrize("N,F,T", [(1, 1, 1), (2, 1, 1), (1, 5, 1), (1, 2, 3), (7, 1, 1), (3, 1, 2), (4, 1, 1), (15, 1, 1), (16, 1, 1), (17, 1, 1), (18, 2, 3),
                                   (31, 1, 2), (64, 1, 2), (66, 3, 2), (1, 4, 6), (2, 1, 9), (5, 1, 8),
                                   (19, 3, 4), (64, 1, 9)])
def test_only_the_frame_is_read(harness, N, F, T):
    r = subprocess.run([harness, str(N), str(F), str(T)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


BLOCKS = r"""
#include <stdio.h>
#include <stdlib.h>
#include "xe_corr.cuh"
int main(int, char** argv) { printf("%d\n", xe::repack_rows_per_block(atoll(argv[1]), atoi(argv[2]), 152)); }
"""


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("blocks"), BLOCKS)


@pytest.mark.parametrize("N,F,T", [(1, 1, 1), (8, 1, 2048), (8, 256, 64), (30, 1, 640), (65, 16, 200), (250, 3, 128),
                                   (250, 61, 4001), (1000, 64, 64), (40001, 1, 7)])
def test_rows_are_spread_over_the_gpu(blocks, N, F, T):
    rows, Np = T * F, -(-N // 16) * 16
    per = int(subprocess.run([blocks, str(rows), str(Np)], capture_output=True, text=True, check=True).stdout)
    steps, n = rows * Np // 16, -(-rows // per)  # 16-byte steps of the frame; blocks of 256 threads
    assert per >= 1 and (per == 1 or per * Np <= 32768)
    # every SM has four blocks, or no thread has more than one step (and a row's rounding)
    assert n >= min(4 * 152 // 2, steps // (256 + Np // 16))
