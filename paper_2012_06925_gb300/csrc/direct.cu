// FP64 direct summation, Eq. (1), for error measurements on sampled targets.
// One thread per target and source split (the sources are split so that few
// targets still fill the device); sources are staged through shared memory
// and the splits are summed in order.  Pairs at distance 0 contribute nothing,
// whatever their charge (this entry point takes infinities and NaN).
// Each tile of 256 sources has its own sum, so the sum's rounding grows with
// the tile's length and the number of tiles, not with the number of sources.
// In FP64 the pipe (1.7 lanes per clock and SM) bounds the sum at 12
// instructions an evaluation; with G in integer arithmetic (fixed64.cuh) at 4,
// the differences among them; with the coordinates in fixed point at 1, where
// the integer pipe bounds it.  Coulomb, 2000 targets x 1E6 sources: 48.3 ms in
// FP64 expressions, 9.9 in the last form.
#include <float.h>

#include <algorithm>

#include "fixed64.cuh"
#include "internal.cuh"

namespace bldtt {

constexpr int kDirectThreads = 256;

// Extent of the coordinates of both sets, by dimension: key[d] and key[3 + d]
// are the largest order-preserving keys of v and -v (0 before the first).
__device__ __forceinline__ unsigned long long order_key(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return b >> 63 ? ~b : b | 0x8000000000000000ull;
}
__device__ __forceinline__ double order_value(unsigned long long k) {
  return __longlong_as_double((long long)(k >> 63 ? k & 0x7fffffffffffffffull : ~k));
}
__global__ void __launch_bounds__(kDirectThreads) k_extent(const double* __restrict__ t, int64_t M,
                                                           const double* __restrict__ src, int64_t N,
                                                           unsigned long long* __restrict__ key) {
  const int d = blockIdx.y;
  unsigned long long hi = 0, lo = 0;
  for (int64_t i = (int64_t)blockIdx.x * kDirectThreads + threadIdx.x; i < M + N;
       i += (int64_t)gridDim.x * kDirectThreads) {
    const double v = i < M ? t[d * M + i] : src[d * N + i - M];
    hi = max(hi, order_key(v));
    lo = max(lo, order_key(-v));
  }
  for (int o = 16; o; o >>= 1) {
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    lo = max(lo, __shfl_xor_sync(0xffffffffu, lo, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(key + d, hi);
    atomicMax(key + 3 + d, lo);
  }
}

// Form of G: FP64 expressions; integer arithmetic on FP64 differences, for a
// finite kappa >= 0 (the direct sum takes any); the same on coordinates in fixed
// point, in units of the two sets' common extent (key), with FP64 differences
// for pairs closer than 1/64 of it, and for all if the extent is 0 or not finite.
enum DirectForm { kFormFp64, kFormFixed, kFormFixedCoords };

// q G in FP64 expressions added to a; nothing for a pair at distance 0.
template <int KERN>
__device__ __forceinline__ double add_fp64(double dx, double dy, double dz, double q, double kappa, double a) {
  const double r2 = dx * dx + dy * dy + dz * dz;
  if (!(r2 > 0.0)) return a;
  const double r = sqrt(r2);
  double g;
  if (KERN == BLDTT_COULOMB)
    g = 1.0 / r;
  else if (KERN == BLDTT_YUKAWA)
    g = exp(-kappa * r) / r;
  else if (KERN == BLDTT_OSCILLATORY)
    g = sin(kappa * r) / r;
  else if (KERN == BLDTT_REG_COULOMB)
    g = 1.0 / sqrt(r2 + kappa * kappa);
  else
    g = 1.0 + dx - 2.0 * dy + 3.0 * dz + dx * dy - dy * dz + dx * dx * dz * dz - 0.5 * dy * dy;
  return fma(g, q, a);
}
// The fixed-point forms give a pair at distance 0 the factor 0, which does not
// leave out a charge that is not finite: a split's sum that is not finite is
// taken again here, from the sources in memory and out of line, so that the
// forms' loops keep their registers.
template <int KERN>
__device__ __noinline__ double split_again(const double* t, int64_t M, int64_t i, const double* src, int64_t N,
                                           const double* q, double kappa, int64_t s0, int64_t s1) {
  const double x = t[i], y = t[M + i], z = t[2 * M + i];
  double acc = 0.0, a = 0.0;
#pragma unroll 1
  for (int64_t j = s0; j < s1; ++j) {
    if ((j - s0) % kDirectThreads == 0) {
      acc += a;
      a = 0.0;
    }
    a = add_fp64<KERN>(x - src[j], y - src[N + j], z - src[2 * N + j], q[j], kappa, a);
  }
  return acc + a;
}

// CTAs of a form that an SM holds (their registers; split_again's must not take more).
template <int KERN, int FORM>
constexpr int direct_ctas() {
  return FORM == kFormFp64 ? 0 : KERN == BLDTT_YUKAWA ? 5 : FORM == kFormFixedCoords ? 6 : 8;
}
template <int KERN, int FORM>
__global__ void __launch_bounds__(kDirectThreads, direct_ctas<KERN, FORM>()) k_direct(const double* __restrict__ t, int64_t M,
                                                           const double* __restrict__ src, int64_t N,
                                                           const double* __restrict__ q, double kappa,
                                                           int64_t span, const unsigned long long* __restrict__ key,
                                                           double* __restrict__ part) {
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
  __shared__ long long fx[FORM == kFormFixedCoords ? kDirectThreads : 1], fy[FORM == kFormFixedCoords ? kDirectThreads : 1],
      fz[FORM == kFormFixedCoords ? kDirectThreads : 1];
  int k2 = 0;                                       // unit 2^-k2
  uint32_t top_min = ~0u;
  long long X = 0, Y = 0, Z = 0;
  if (FORM == kFormFixedCoords) {
    double w = 0.0;
    for (int d = 0; d < 3; ++d) w = fmax(w, order_value(key[d]) + order_value(key[3 + d]));
    bool ok = true;
    for (int d = 0; d < 3; ++d) ok = ok && order_value(key[d]) <= DBL_MAX && order_value(key[3 + d]) <= DBL_MAX;
    if (ok && w >= 0x1p-900 && w <= 0x1p900) {
      k2 = 61 - ilogb(w);                           // w < 2^(62 - k2)
      top_min = fixed64::kFixedTop;
    }
    X = fixed64::to_fixed(x, k2);
    Y = fixed64::to_fixed(y, k2);
    Z = fixed64::to_fixed(z, k2);
  }
  const fixed64::Screen screen = FORM != kFormFp64 && KERN == BLDTT_YUKAWA ? fixed64::make_screen(kappa) : fixed64::Screen{0, 0};
  double acc = 0.0;
  for (int64_t base = s0; base < s1; base += kDirectThreads) {
    int64_t j = base + threadIdx.x;
    tile[threadIdx.x] = j < s1 ? make_double4(src[j], src[N + j], src[2 * N + j], q[j])
                               : make_double4(0, 0, 0, 0);
    if (FORM == kFormFixedCoords) {
      const double4 p = tile[threadIdx.x];
      fx[threadIdx.x] = fixed64::to_fixed(p.x, k2);
      fy[threadIdx.x] = fixed64::to_fixed(p.y, k2);
      fz[threadIdx.x] = fixed64::to_fixed(p.z, k2);
    }
    __syncthreads();
    int cnt = (int)min((int64_t)kDirectThreads, s1 - base);
    double a = 0.0;
#pragma unroll 2
    for (int k = 0; k < cnt; ++k) {
      if (FORM == kFormFixedCoords) {
        const long long ux = X - fx[k], uy = Y - fy[k], uz = Z - fz[k];
        const uint32_t top = fixed64::fixed_top(ux, uy, uz);
        if (top >= top_min) {
          int E;
          const fixed64::u64 S = fixed64::sum_squares_fixed(ux, uy, uz, top, k2, &E);
          const double g = KERN == BLDTT_COULOMB ? fixed64::inv_r_of(S, E) : fixed64::screened_inv_r_of(S, E, screen);
          a = fma(g, tile[k].w, a);
          continue;
        }
      }
      const double4 p = tile[k];
      const double dx = x - p.x, dy = y - p.y, dz = z - p.z;
      if (FORM != kFormFp64) {
        const double g = KERN == BLDTT_COULOMB  ? fixed64::inv_r(dx, dy, dz)
                         : KERN == BLDTT_YUKAWA ? fixed64::screened_inv_r(dx, dy, dz, screen)
                                                : fixed64::inv_sqrt_r2_kappa2(dx, dy, dz, kappa);
        a = fma(g, p.w, a);
      } else {
        a = add_fp64<KERN>(dx, dy, dz, p.w, kappa, a);
      }
    }
    acc += a;
    __syncthreads();
  }
  if (i >= M) return;
  if (FORM != kFormFp64 && fixed64::exponent_of(fixed64::bits_of(acc)) == 0x7ff)
    acc = split_again<KERN>(t, M, i, src, N, q, kappa, s0, s1);
  part[(int64_t)blockIdx.y * M + i] = acc;
}

// phi[i] = sum over the source splits, with each addition's rounding error
// (Knuth's two-sum) added at the end: hundreds of splits one after the other were
// most of the sum's error.  One warp per target, in an order fixed by the number
// of splits (a thread per target: 0.16 ms for 500 targets).
__device__ __forceinline__ void add_split(double& a, double& err, double b) {
  const double t = a + b, w = t - a;
  err += (a - (t - w)) + (b - w);
  a = t;
}
__global__ void __launch_bounds__(kDirectThreads) k_direct_reduce(const double* __restrict__ part, int64_t M,
                                                                  int splits, double* __restrict__ phi) {
  const int64_t i = ((int64_t)blockIdx.x * kDirectThreads + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= M) return;                               // whole warps
  double a = 0.0, err = 0.0;
  for (int k = lane; k < splits; k += 32) add_split(a, err, part[(int64_t)k * M + i]);
  for (int o = 16; o; o >>= 1) {
    const double b = __shfl_down_sync(0xffffffffu, a, o), e = __shfl_down_sync(0xffffffffu, err, o);
    add_split(a, err, b);
    err += e;
  }
  if (lane == 0) phi[i] = err - err == 0.0 ? a + err : a;   // infinite sums have no error term
}

int direct_sum(const double* targets, int64_t M, const double* sources, int64_t N,
               const double* charges, int kernel, double kappa, double* phi, cudaStream_t s) {
  const unsigned blocks = (unsigned)((M + kDirectThreads - 1) / kDirectThreads);
  // Split the sources so that the grid fills the device (few targets, many
  // sources): up to eight CTAs to an SM (with four 2E4 x 2E5 takes 24.6 ms, with
  // eight 21.5), and of those numbers of splits down to half of it the one whose
  // fullest SM has the least to do.
  int dev = 0, sms = 0;
  BL_CUDA(cudaGetDevice(&dev));
  BL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t most = std::max<int64_t>(
      1, std::min({((int64_t)8 * sms + blocks - 1) / blocks, (N + kDirectThreads - 1) / kDirectThreads, (int64_t)1024}));
  int64_t splits = most, least = INT64_MAX;
  for (int64_t k = most; 2 * k > most; --k) {
    const int64_t load = (blocks * k + sms - 1) / sms * ((N + k - 1) / k);
    if (load < least) {
      least = load;
      splits = k;
    }
  }
  const int64_t span = (N + splits - 1) / splits;
  const dim3 grid(blocks, (unsigned)splits);
  const bool fixed = kappa >= 0.0 && kappa <= DBL_MAX;
  // The extent takes two launches, about 6 us: worth it from some millions of evaluations.
  int64_t dummy = 0;
  const bool coords = (double)M * (double)N >= 0x1p23 &&
                      (kernel == BLDTT_COULOMB || (kernel == BLDTT_YUKAWA && fixed));
  double* part = phi;
  unsigned long long* key = nullptr;
  Arena scratch;                       // freed, in stream order, when it goes out of scope
  if (splits > 1) scratch.add(&part, (size_t)(splits * M));
  if (coords) scratch.add(&key, 6);
  if (splits > 1 || coords) BL_TRY(scratch.alloc(s));
  if (coords) {
    BL_CUDA(cudaMemsetAsync(key, 0, 6 * sizeof(*key), s));
    const int64_t need = (M + N + kDirectThreads - 1) / kDirectThreads;
    k_extent<<<dim3((unsigned)(need < 2 * sms ? need : 2 * sms), 3), kDirectThreads, 0, s>>>(targets, M, sources, N,
                                                                                            key);
    BL_LAUNCHED(dummy);
  }
  void (*k)(const double*, int64_t, const double*, int64_t, const double*, double, int64_t, const unsigned long long*,
            double*) = k_direct<BLDTT_TEST_POLY, kFormFp64>;
  if (kernel == BLDTT_COULOMB)
    k = coords ? k_direct<BLDTT_COULOMB, kFormFixedCoords> : k_direct<BLDTT_COULOMB, kFormFixed>;
  else if (kernel == BLDTT_YUKAWA)
    k = coords  ? k_direct<BLDTT_YUKAWA, kFormFixedCoords>
        : fixed ? k_direct<BLDTT_YUKAWA, kFormFixed>
                : k_direct<BLDTT_YUKAWA, kFormFp64>;
  else if (kernel == BLDTT_OSCILLATORY)
    k = k_direct<BLDTT_OSCILLATORY, kFormFp64>;
  else if (kernel == BLDTT_REG_COULOMB)
    k = fixed ? k_direct<BLDTT_REG_COULOMB, kFormFixed> : k_direct<BLDTT_REG_COULOMB, kFormFp64>;
  k<<<grid, kDirectThreads, 0, s>>>(targets, M, sources, N, charges, kappa, span, key, part);
  BL_LAUNCHED(dummy);
  if (splits > 1) {
    k_direct_reduce<<<(unsigned)((M * 32 + kDirectThreads - 1) / kDirectThreads), kDirectThreads, 0, s>>>(part, M, (int)splits, phi);
    BL_LAUNCHED(dummy);
  }
  return BLDTT_OK;
}

}  // namespace bldtt
