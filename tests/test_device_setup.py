"""Device set-up reports the CUDA call that failed (CPU: the library's object linked against fakes of the calls)."""
import os
import subprocess
import sys

import pytest

import paper_1503_06203_gb300 as xe
from paper_1503_06203_gb300 import builder

# The calls of corr_create up to its first allocation, which always fails: no GPU is touched.
FAKES = r"""
#include <cuda_runtime.h>
#include <string.h>
extern "C" {
static int sets, gets, fail_set = -1, fail_get = -1;
void fake_plan(int s, int g) { sets = gets = 0; fail_set = s; fail_get = g; }
int fake_sets() { return sets; }
int fake_gets() { return gets; }
cudaError_t __wrap_cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t __wrap_cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
  return sets++ == fail_set ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t __wrap_cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  a->numRegs = 128;
  return gets++ == fail_get ? cudaErrorInvalidDeviceFunction : cudaSuccess;
}
cudaError_t __wrap_cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t __wrap_cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t __wrap_cudaMalloc(void**, size_t) { return cudaErrorMemoryAllocation; }
cudaError_t __wrap_cudaGetLastError() { return cudaSuccess; }
}
"""
WRAPPED = ["cudaGetDevice", "cudaFuncSetAttribute", "cudaFuncGetAttributes", "cudaDeviceGetAttribute", "cudaMalloc",
           "cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags", "cudaGetLastError"]

# argv: the library, then set:get pairs; prints the error of each corr_create
CALLER = """
import ctypes, sys
L = ctypes.CDLL(sys.argv[1])
L.corr_create.restype = ctypes.c_void_p
L.corr_last_error.restype = ctypes.c_char_p
for p in sys.argv[2:]:
    s, g = map(int, p.split(":"))
    L.fake_plan(s, g)
    h = L.corr_create(64, 1, 128)
    print(bool(h), L.fake_sets(), L.fake_gets(), L.corr_last_error().decode(), sep="|")
"""


@pytest.fixture(scope="module")
def faked(tmp_path_factory):
    xe.build()
    obj = os.path.join(os.path.dirname(builder.LIB), "_build", "xengine.o")
    if not os.path.exists(obj):
        builder.build(force=True)
    d = tmp_path_factory.mktemp("fakes")
    src, lib = d / "fakes.cu", d / "libfaked.so"
    src.write_text(FAKES)
    wraps = [f"-Xlinker=--wrap={s}" for s in WRAPPED]
    subprocess.run([builder._nvcc(), "-shared", "-Xcompiler", "-fPIC", *wraps, "-o", str(lib), str(src), obj], check=True)

    def run(*plans):
        r = subprocess.run([sys.executable, "-c", CALLER, str(lib), *(f"{s}:{g}" for s, g in plans)],
                           capture_output=True, text=True, check=True)
        return [line.split("|", 3) for line in r.stdout.splitlines()]
    return run


def test_every_failed_call_is_reported(faked):
    (made, sets, gets, msg), = faked((-1, -1))  # none fails: set-up passes, the first allocation does not
    assert made == "False" and "cudaMalloc" in msg
    sets, gets = int(sets), int(gets)
    assert sets >= gets > 0
    for (made, n, _, msg), k in zip(faked(*((k, -1) for k in range(sets))), range(sets)):
        assert made == "False" and int(n) == k + 1 and "cudaFuncSetAttribute" in msg, (k, msg)
    for (made, _, n, msg), k in zip(faked(*((-1, k) for k in range(gets))), range(gets)):
        assert made == "False" and int(n) == k + 1 and "cudaFuncGetAttributes" in msg, (k, msg)
