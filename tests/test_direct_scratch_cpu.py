"""The direct sum's scratch is freed when the call fails on the way: direct.cu's
host code with a fake CUDA runtime and a fake allocator, the n-th of whose calls
fails.  They make a program of their own that links no CUDA library: loaded into
this process, the fake's names would give way to the real runtime's."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2012_06925_gb300", "csrc")
FAKE = r"""
#include <stddef.h>
#include <stdio.h>
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
static int run(long m, long n, int kernel, int fail) {
  live = calls = last = 0;
  fail_at = fail;
  double x;
  return bldtt::direct_sum(&x, m, &x, n, &x, kernel, 0.5, &x, 0);
}
// prints a line "failing call, status, allocations left" for no failure (0) and for every call made
int main(int, char** a) {
  const long m = atol(a[1]), n = atol(a[2]);
  const int kernel = atoi(a[3]);
  int st = run(m, n, kernel, 0);
  const int made = calls;
  printf("0 %d %d\n", st, live);
  for (int k = 1; k <= made; ++k) {
    st = run(m, n, kernel, k);
    printf("%d %d %d\n", k, st, live);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("direct")
    (d / "fake.cpp").write_text(FAKE)
    flags = ["-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "--expt-relaxed-constexpr", "-w",
             "-I", CSRC, "-I", os.path.join(ROOT, "include")]
    subprocess.run([nvcc, *flags, "-c", os.path.join(CSRC, "direct.cu"), "-o", str(d / "direct.o")], check=True)
    exe = str(d / "run")
    subprocess.run(["g++", str(d / "fake.cpp"), str(d / "direct.o"), "-o", exe], check=True)
    libs = subprocess.run(["ldd", exe], capture_output=True, text=True, check=True).stdout
    assert "cuda" not in libs
    return exe


@pytest.mark.parametrize("kernel", [0, 1, 2, 3])
@pytest.mark.parametrize("m,n", [(10, 20), (100, 5000), (500, 100000)])    # no scratch, splits, splits and extent
def test_no_scratch_is_left(program, m, n, kernel):
    out = subprocess.run([program, str(m), str(n), str(kernel)], capture_output=True, text=True, check=True,
                         env={"PATH": os.environ.get("PATH", "")}).stdout
    rows = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    assert rows[0] == (0, 0, 0) and len(rows) >= 4
    for call, status, left in rows[1:]:
        assert status != 0 and left == 0, (call, status, left)
