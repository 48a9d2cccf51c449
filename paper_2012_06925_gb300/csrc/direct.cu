// FP64 direct summation, Eq. (1), for error measurements on sampled targets.
// One thread per target and source split (the sources are split so that few
// targets still fill the device); sources are staged through shared memory
// and the splits are summed in order.  Pairs at distance 0 contribute nothing.
// Each tile of 256 sources has its own sum, so the sum's rounding grows with
// the tile's length and the number of tiles, not with the number of sources.
// Bound by the FP64 pipe (1.7 lanes per clock and SM): 12 instructions an
// evaluation in FP64, 4 with G in integer arithmetic; Coulomb, 2000 targets x
// 1E6 sources: 48.3 -> 15.3 ms.
#include <float.h>

#include "fixed64.cuh"
#include "internal.cuh"

namespace bldtt {

constexpr int kDirectThreads = 256;

// FIXED: G in integer arithmetic (fixed64.cuh).  It wants a finite kappa >= 0,
// as plans do; the direct sum takes any, and evaluates the others in FP64.
template <int KERN, bool FIXED>
__global__ void __launch_bounds__(kDirectThreads) k_direct(const double* __restrict__ t, int64_t M,
                                                           const double* __restrict__ src, int64_t N,
                                                           const double* __restrict__ q, double kappa,
                                                           int64_t span, double* __restrict__ part) {
  // blockIdx.y takes sources [y * span, min(N, (y + 1) * span)); part[y][i]
  __shared__ double4 tile[kDirectThreads];
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double x = 0, y = 0, z = 0;
  if (i < M) {
    x = t[i];
    y = t[M + i];
    z = t[2 * M + i];
  }
  const int64_t s0 = (int64_t)blockIdx.y * span, s1 = min(N, s0 + span);
  const fixed64::Screen screen = FIXED && KERN == BLDTT_YUKAWA ? fixed64::make_screen(kappa) : fixed64::Screen{0, 0};
  double acc = 0.0;
  for (int64_t base = s0; base < s1; base += kDirectThreads) {
    int64_t j = base + threadIdx.x;
    tile[threadIdx.x] = j < s1 ? make_double4(src[j], src[N + j], src[2 * N + j], q[j])
                               : make_double4(0, 0, 0, 0);
    __syncthreads();
    int cnt = (int)min((int64_t)kDirectThreads, s1 - base);
    double a = 0.0;
    for (int k = 0; k < cnt; ++k) {
      double4 p = tile[k];
      double dx = x - p.x, dy = y - p.y, dz = z - p.z;
      double g = 0.0;
      if (FIXED) {
        g = KERN == BLDTT_COULOMB  ? fixed64::inv_r(dx, dy, dz)
            : KERN == BLDTT_YUKAWA ? fixed64::screened_inv_r(dx, dy, dz, screen)
                                   : fixed64::inv_sqrt_r2_kappa2(dx, dy, dz, kappa);
      } else {
        const double r2 = dx * dx + dy * dy + dz * dz;
        if (r2 > 0.0) {
          const double r = sqrt(r2);
          if (KERN == BLDTT_YUKAWA)
            g = exp(-kappa * r) / r;
          else if (KERN == BLDTT_OSCILLATORY)
            g = sin(kappa * r) / r;
          else if (KERN == BLDTT_REG_COULOMB)
            g = 1.0 / sqrt(r2 + kappa * kappa);
          else
            g = 1.0 + dx - 2.0 * dy + 3.0 * dz + dx * dy - dy * dz + dx * dx * dz * dz - 0.5 * dy * dy;
        }
      }
      a = fma(g, p.w, a);
    }
    acc += a;
    __syncthreads();
  }
  if (i < M) part[(int64_t)blockIdx.y * M + i] = acc;
}

// phi[i] = sum over the source splits, in split order, with each addition's
// rounding error (Knuth's two-sum) added at the end: hundreds of splits one
// after the other were most of the sum's error.
__global__ void k_direct_reduce(const double* __restrict__ part, int64_t M, int splits,
                                double* __restrict__ phi) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  double a = 0.0, err = 0.0;
  for (int k = 0; k < splits; ++k) {
    const double b = part[(int64_t)k * M + i], t = a + b, w = t - a;
    err += (a - (t - w)) + (b - w);
    a = t;
  }
  phi[i] = err - err == 0.0 ? a + err : a;      // infinite sums have no error term
}

int direct_sum(const double* targets, int64_t M, const double* sources, int64_t N,
               const double* charges, int kernel, double kappa, double* phi, cudaStream_t s) {
  const unsigned blocks = (unsigned)((M + kDirectThreads - 1) / kDirectThreads);
  // Split the sources so that the grid fills the device (few targets, many sources).
  int dev = 0, sms = 0;
  BL_CUDA(cudaGetDevice(&dev));
  BL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  int64_t splits = ((int64_t)4 * sms + blocks - 1) / blocks;
  const int64_t max_splits = (N + kDirectThreads - 1) / kDirectThreads;
  if (splits > max_splits) splits = max_splits;
  if (splits > 1024) splits = 1024;
  if (splits < 1) splits = 1;
  const int64_t span = (N + splits - 1) / splits;
  double* part = phi;
  if (splits > 1) BL_TRY(dalloc_n(&part, (size_t)(splits * M), s));
  const dim3 grid(blocks, (unsigned)splits);
  const bool fixed = kappa >= 0.0 && kappa <= DBL_MAX;
  void (*k)(const double*, int64_t, const double*, int64_t, const double*, double, int64_t, double*) =
      k_direct<BLDTT_TEST_POLY, false>;
  if (kernel == BLDTT_COULOMB)
    k = k_direct<BLDTT_COULOMB, true>;
  else if (kernel == BLDTT_YUKAWA)
    k = fixed ? k_direct<BLDTT_YUKAWA, true> : k_direct<BLDTT_YUKAWA, false>;
  else if (kernel == BLDTT_OSCILLATORY)
    k = k_direct<BLDTT_OSCILLATORY, false>;
  else if (kernel == BLDTT_REG_COULOMB)
    k = fixed ? k_direct<BLDTT_REG_COULOMB, true> : k_direct<BLDTT_REG_COULOMB, false>;
  k<<<grid, kDirectThreads, 0, s>>>(targets, M, sources, N, charges, kappa, span, part);
  int64_t dummy = 0;
  BL_LAUNCHED(dummy);
  if (splits > 1) {
    k_direct_reduce<<<blocks, kDirectThreads, 0, s>>>(part, M, (int)splits, phi);
    BL_LAUNCHED(dummy);
    dfree(part, s);
  }
  return BLDTT_OK;
}

}  // namespace bldtt
