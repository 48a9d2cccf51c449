"""The direct sum's scratch is freed when the call fails on the way: direct.cu's
host code, compiled against a fake CUDA runtime and a fake allocator (no GPU, no
CUDA library), with the n-th runtime call made to fail."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2012_06925_gb300", "csrc")
FAKE = r"""
#include <stddef.h>
#include <stdlib.h>
struct CUstream_st;
typedef CUstream_st* Stream;
struct Dim { unsigned x, y, z; };
namespace bldtt {
int direct_sum(const double*, long, const double*, long, const double*, int, double, double*, Stream);
void set_error(const char*, ...);
int dalloc(void** p, size_t, Stream);
void dfree(void* p, Stream);
}
static int live = 0, calls = 0, fail_at = 0, last = 0;
static int failing() { return ++calls == fail_at ? 999 : 0; }
extern "C" {
int cudaGetDevice(int* d) { *d = 0; return failing(); }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return failing(); }
int cudaMemsetAsync(void*, int, size_t, Stream) { return failing(); }
int cudaLaunchKernel(const void*, Dim, Dim, void**, size_t, Stream) { return last = failing(); }
int cudaGetLastError() { int e = last; last = 0; return e; }
const char* cudaGetErrorString(int) { return "fake"; }
unsigned __cudaPushCallConfiguration(Dim, Dim, size_t, Stream) { return 0; }
int __cudaPopCallConfiguration(Dim*, Dim*, size_t*, void*) { return 0; }
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaLaunchKernel(void*, Dim, Dim, void**, size_t, Stream) { return last = failing(); }
void** __cudaRegisterFatBinary(void*) { return 0; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
// returns the status; *leaked: allocations left, *made: runtime and allocator calls made
int run(long m, long n, int kernel, int fail, int* leaked, int* made) {
  live = calls = last = 0;
  fail_at = fail;
  double x;
  const int st = bldtt::direct_sum(&x, m, &x, n, &x, kernel, 0.5, &x, 0);
  *leaked = live;
  *made = calls;
  return st;
}
}
namespace bldtt {
void set_error(const char*, ...) {}
int dalloc(void** p, size_t, Stream) {
  if (failing()) return 2;
  ++live;
  *p = malloc(1);
  return 0;
}
void dfree(void* p, Stream) {
  if (!p) return;
  free(p);
  --live;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("direct")
    (d / "fake.cpp").write_text(FAKE)
    flags = ["-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-Xcompiler", "-fPIC",
             "--expt-relaxed-constexpr", "-w", "-I", CSRC, "-I", os.path.join(ROOT, "include")]
    subprocess.run([nvcc, *flags, "-c", os.path.join(CSRC, "direct.cu"), "-o", str(d / "direct.o")], check=True)
    so = str(d / "direct.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-Wl,-z,defs", str(d / "fake.cpp"), str(d / "direct.o"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("kernel", [0, 1, 2, 3])
@pytest.mark.parametrize("m,n", [(10, 20), (100, 5000), (500, 100000)])    # no scratch, splits, splits and extent
def test_no_scratch_is_left(lib, m, n, kernel):
    leaked, made = ctypes.c_int(), ctypes.c_int()
    call = lambda fail: lib.run(ctypes.c_long(m), ctypes.c_long(n), kernel, fail, ctypes.byref(leaked),
                                ctypes.byref(made))
    assert call(0) == 0 and leaked.value == 0
    steps = made.value
    for k in range(1, steps + 1):
        assert call(k) != 0 and leaked.value == 0, (k, leaked.value)
