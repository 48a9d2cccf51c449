// Pipe-throughput microbenchmark behind the benchmark's issue ceilings.  It is
// measurement tooling, built into its own library (libbldtt_pipes.so) that only
// bench.py and its test load; the BLDTT library does not contain it.
//
// One CTA of 1024 threads per SM (each CTA reserves more than half of an SM's
// shared memory, so no SM holds two) runs eight independent dependency chains
// per thread of one operation, and the SM's own cycle counter (clock64) times
// it, so the rate is in operations (lanes) per clock per SM whatever the clock
// frequency.
//
// C ABI:
//   int pipes_rates(double* out, void* cuda_stream)
//     out: host, 5 doubles: lanes per clock per SM of FP32 FMA, packed FP32x2
//     FMA (two lanes per instruction), MUFU rsqrt, MUFU exp2 and FP64 FMA
//     (median CTA).  Synchronous on cuda_stream.  Returns 0, or the CUDA error
//     code of the first failing call (message from pipes_last_error()).
//   int pipes_pair_loop(double* out, void* cuda_stream)
//     out: host, 2 doubles: evaluations per clock per SM of the interaction
//     kernel's packed inner loop by itself, Coulomb and Yukawa: 24 warps on an SM
//     (six CTAs of four), two targets a thread, 256 staged sources read again and
//     again for a fixed number of cycles, no producer, ring, lists or chunk sums.
//     Returns as pipes_rates.
//   const char* pipes_last_error(void)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <vector>

namespace {

constexpr int kRateThreads = 1024;
constexpr int kRateSmem = 120 * 1024;   // dynamic shared memory reserved, unused

enum RateOp { kOpFfma = 0, kOpFfma2 = 1, kOpRsqrt = 2, kOpEx2 = 3, kOpDfma = 4 };

char g_msg[256] = "";

template <int OP>
__global__ void __launch_bounds__(kRateThreads) k_rate(int iters, float seed, float* __restrict__ sink,
                                                       long long* __restrict__ cycles) {
  float a[8];
  double d[8];
  unsigned long long p[4];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    a[k] = seed + 1e-3f * (float)(threadIdx.x + k);
    d[k] = (double)a[k];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) asm("mov.b64 %0, {%1, %2};" : "=l"(p[k]) : "f"(a[2 * k]), "f"(a[2 * k + 1]));
  unsigned long long c2;
  {
    const float c = 0.999f;
    asm("mov.b64 %0, {%1, %1};" : "=l"(c2) : "f"(c));
  }
  __syncthreads();
  const long long t0 = clock64();
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (OP == kOpFfma) a[k] = fmaf(a[k], 0.999f, 1e-4f);
      if (OP == kOpRsqrt) asm volatile("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(a[k]));
      if (OP == kOpEx2)   // 2^-a: a bounded chain (a -> ~0.64)
        asm volatile("{ .reg .f32 t; neg.f32 t, %0; ex2.approx.ftz.f32 %0, t; }" : "+f"(a[k]));
      if (OP == kOpDfma) d[k] = fma(d[k], 0.999, 1e-4);
    }
    if (OP == kOpFfma2) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {   // 4 packed chains, twice: 8 packed operations = 16 lanes
        asm volatile("fma.rn.f32x2 %0, %0, %1, %1;" : "+l"(p[k]) : "l"(c2));
        asm volatile("fma.rn.f32x2 %0, %0, %1, %1;" : "+l"(p[k]) : "l"(c2));
      }
    }
  }
  __syncthreads();
  const long long t1 = clock64();
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) s += a[k] + (float)d[k];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p[k]));
    s += lo + hi;
  }
  sink[blockIdx.x * blockDim.x + threadIdx.x] = s;
  if (threadIdx.x == 0) cycles[blockIdx.x] = t1 - t0;
}

// ---- the packed pair loop ----------------------------------------------------
constexpr int kPairThreads = 128, kPairCtas = 6, kPairRecords = 128, kPairTargets = 2;
constexpr int kPairMaxPasses = 1 << 20;
constexpr int kPairSmem = 32 * 1024;    // dynamic shared memory reserved, unused: with 4 KB of records and 1 KB a CTA
                                        // six CTAs fit the 228 KB of an SM, seven do not
typedef unsigned long long f2_t;

__device__ __forceinline__ f2_t f2(float a, float b) {
  f2_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ void f2_halves(f2_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2_t f2_sub(f2_t a, f2_t b) {
  f2_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t f2_mul(f2_t a, f2_t b) {
  f2_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t f2_fma(f2_t a, f2_t b, f2_t c) {
  f2_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

template <bool YUKAWA>
__global__ void __launch_bounds__(kPairThreads, kPairCtas) k_pair_loop(long long limit, float seed,
                                                                       float* __restrict__ sink,
                                                                       int* __restrict__ done) {
  __shared__ ulonglong2 rec[2 * kPairRecords];       // (x0, x1) (y0, y1) | (z0, z1) (q0, q1)
  for (int i = threadIdx.x; i < kPairRecords; i += kPairThreads) {
    const float v = seed + 1e-3f * (float)i;
    rec[2 * i] = make_ulonglong2(f2(v, -v), f2(0.5f * v, v));
    rec[2 * i + 1] = make_ulonglong2(f2(v, 0.25f * v), f2(1.f, -1.f));
  }
  f2_t x[kPairTargets][3], acc[kPairTargets];
  for (int k = 0; k < kPairTargets; ++k) {
    for (int d = 0; d < 3; ++d) {
      const float v = 3.f + seed + 0.01f * (float)(threadIdx.x + 7 * k + d);
      x[k][d] = f2(v, v);
    }
    acc[k] = 0ull;
  }
  const f2_t prm = f2(-seed, -seed);
  __syncthreads();
  // Each warp counts the passes it makes in `limit` cycles: the warps of an SM do
  // not progress alike, so the time of a fixed number of passes each would include a
  // phase of fewer warps.
  const long long t0 = clock64();
  int it = 0;
#pragma unroll 1
  for (; it < kPairMaxPasses && clock64() - t0 < limit; ++it) {
#pragma unroll 8
    for (int j = 0; j < kPairRecords; ++j) {
      const ulonglong2 a = rec[2 * j], b = rec[2 * j + 1];
#pragma unroll
      for (int k = 0; k < kPairTargets; ++k) {
        const f2_t dx = f2_sub(x[k][0], a.x), dy = f2_sub(x[k][1], a.y), dz = f2_sub(x[k][2], b.x);
        const f2_t r2 = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
        float r0, r1;
        f2_halves(r2, r0, r1);
        asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(r0));
        asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(r1));
        const f2_t ri = f2(r0, r1);
        if (YUKAWA) {
          float e0, e1;
          f2_halves(f2_mul(f2_mul(r2, ri), prm), e0, e1);
          asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(e0));
          asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(e1));
          acc[k] = f2_fma(f2_mul(b.y, ri), f2(e0, e1), acc[k]);
        } else {
          acc[k] = f2_fma(b.y, ri, acc[k]);
        }
      }
    }
    for (int k = 0; k < kPairTargets; ++k) asm volatile("" : "+l"(x[k][0]));   // the same work again
  }
  float s = 0.f;
  for (int k = 0; k < kPairTargets; ++k) {
    float lo, hi;
    f2_halves(acc[k], lo, hi);
    s += lo + hi;
  }
  sink[blockIdx.x * kPairThreads + threadIdx.x] = s;
  if (threadIdx.x % 32 == 0) done[(blockIdx.x * kPairThreads + threadIdx.x) / 32] = it;
}

int fail(cudaError_t e, const char* what) {
  std::snprintf(g_msg, sizeof(g_msg), "%s failed: %s", what, cudaGetErrorString(e));
  return (int)e;
}

#define PIPES_CUDA(call)                          \
  do {                                            \
    cudaError_t e_ = (call);                      \
    if (e_ != cudaSuccess) return fail(e_, #call); \
  } while (0)

template <int OP>
int rate(int sms, int iters, float* sink, long long* cycles, cudaStream_t s, double* out) {
  PIPES_CUDA(cudaFuncSetAttribute(k_rate<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRateSmem));
  k_rate<OP><<<sms, kRateThreads, kRateSmem, s>>>(iters, 0.75f, sink, cycles);
  PIPES_CUDA(cudaGetLastError());
  std::vector<long long> h(sms);
  PIPES_CUDA(cudaMemcpyAsync(h.data(), cycles, sms * sizeof(long long), cudaMemcpyDeviceToHost, s));
  PIPES_CUDA(cudaStreamSynchronize(s));
  std::sort(h.begin(), h.end());
  const double lanes = (double)kRateThreads * iters * (OP == kOpFfma2 ? 16 : 8);
  *out = lanes / (double)h[sms / 2];   // median CTA
  return 0;
}

int rates_all(int sms, float* sink, long long* cycles, cudaStream_t s, double* out) {
  int rc = rate<kOpFfma>(sms, 4096, sink, cycles, s, &out[0]);
  if (rc == 0) rc = rate<kOpFfma2>(sms, 2048, sink, cycles, s, &out[1]);
  if (rc == 0) rc = rate<kOpRsqrt>(sms, 1024, sink, cycles, s, &out[2]);
  if (rc == 0) rc = rate<kOpEx2>(sms, 1024, sink, cycles, s, &out[3]);
  if (rc == 0) rc = rate<kOpDfma>(sms, 256, sink, cycles, s, &out[4]);
  return rc;
}

template <bool YUKAWA>
int pair_loop(int sms, long long limit, float* sink, int* done, cudaStream_t s, double* out) {
  PIPES_CUDA(cudaFuncSetAttribute(k_pair_loop<YUKAWA>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  (int)cudaSharedmemCarveoutMaxShared));
  PIPES_CUDA(cudaFuncSetAttribute(k_pair_loop<YUKAWA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem));
  const int ctas = sms * kPairCtas;
  std::vector<int> h((size_t)ctas * kPairThreads / 32);
  for (int rep = 0; rep < 2; ++rep) {                // the first run warms up
    k_pair_loop<YUKAWA><<<ctas, kPairThreads, kPairSmem, s>>>(limit, 0.75f, sink, done);
    PIPES_CUDA(cudaGetLastError());
    PIPES_CUDA(cudaMemcpyAsync(h.data(), done, h.size() * sizeof(int), cudaMemcpyDeviceToHost, s));
    PIPES_CUDA(cudaStreamSynchronize(s));
  }
  double passes = 0.0;
  for (int v : h) passes += v;
  *out = passes * 32 * kPairTargets * 2 * kPairRecords / ((double)limit * sms);
  return 0;
}

}  // namespace

extern "C" int pipes_pair_loop(double* out, void* cuda_stream) {
  if (!out) {
    std::snprintf(g_msg, sizeof(g_msg), "pipes_pair_loop: out is NULL");
    return -1;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  int dev = 0, sms = 0;
  PIPES_CUDA(cudaGetDevice(&dev));
  PIPES_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  float* sink = nullptr;
  int* done = nullptr;
  PIPES_CUDA(cudaMalloc(&sink, (size_t)sms * kPairCtas * kPairThreads * sizeof(float)));
  cudaError_t e = cudaMalloc(&done, (size_t)sms * kPairCtas * kPairThreads / 32 * sizeof(int));
  if (e != cudaSuccess) {
    cudaFree(sink);
    return fail(e, "cudaMalloc");
  }
  int rc = pair_loop<false>(sms, 40000000ll, sink, done, s, &out[0]);
  if (rc == 0) rc = pair_loop<true>(sms, 40000000ll, sink, done, s, &out[1]);
  cudaFree(sink);
  cudaFree(done);
  return rc;
}

extern "C" int pipes_rates(double* out, void* cuda_stream) {
  if (!out) {
    std::snprintf(g_msg, sizeof(g_msg), "pipes_rates: out is NULL");
    return -1;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  int dev = 0, sms = 0;
  PIPES_CUDA(cudaGetDevice(&dev));
  PIPES_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  float* sink = nullptr;
  long long* cycles = nullptr;
  PIPES_CUDA(cudaMalloc(&sink, (size_t)sms * kRateThreads * sizeof(float)));
  cudaError_t e = cudaMalloc(&cycles, (size_t)sms * sizeof(long long));
  if (e != cudaSuccess) {
    cudaFree(sink);
    return fail(e, "cudaMalloc");
  }
  const int rc = rates_all(sms, sink, cycles, s, out);
  cudaFree(sink);
  cudaFree(cycles);
  return rc;
}

extern "C" const char* pipes_last_error(void) { return g_msg; }
