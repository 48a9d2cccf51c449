// Learned pair selector: a bfloat16 network that replaces the MAC of Alg. 2
// by a per-pair choice of interaction type and interpolation degree, its
// training kernels, and the per-pair error labels it is trained on.
//
// Features of a pair (t, s), R = |c_t - c_s| > 0, (r_t + r_s)/R < 1:
//   f = (plog2|C_t|/16, plog2|C_s|/16, r_t/R, r_s/R, (r_t + r_s)/R, kR/(1 + kR))
// in FP64 (plog2(m) = e + (f - 1) for m = f 2^e, 1 <= f < 2), rounded to
// float and then to bfloat16.  Network: three hidden ReLU layers of 64 and a
// linear output of 3 per degree, y[3 i + t] ~ log10 of the relative error of
// (PC, CP, CC)[t] at degree d[i] on the pair.  Every layer computes
// z_j = b_j + sum_k w_jk a_k in float, k in increasing order, with bf16
// weights and activations (their products are exact in float), then
// a_j = bf16(max(z_j, 0)); the same arithmetic on any device gives the same
// bits.  The cheapest option with y <= log10(budget) is taken (PP if it costs
// no more); none feasible means no approximation; features outside the
// training box fall back to the MAC.
#include <cuda_bf16.h>

#include <cmath>
#include <vector>

#include "internal.cuh"

namespace bldtt {

constexpr int kSelWarps = 8;   // pairs (or samples) per block, one warp each

__host__ __device__ inline int64_t sel_weight_count(int nout) {
  return (int64_t)kHidden * kFeatures + 2 * (int64_t)kHidden * kHidden + (int64_t)nout * kHidden;
}
__host__ __device__ inline int64_t sel_bias_count(int nout) { return 3 * (int64_t)kHidden + nout; }
// Offsets of W1..W4 and b1..b4 inside the packed master-parameter array.
struct ParamLayout {
  int64_t w[4], b[4], total;
  __host__ __device__ explicit ParamLayout(int nout) {
    const int64_t in[4] = {kFeatures, kHidden, kHidden, kHidden};
    const int64_t out[4] = {kHidden, kHidden, kHidden, nout};
    int64_t o = 0;
    for (int l = 0; l < 4; ++l) {
      w[l] = o;
      o += in[l] * out[l];
      b[l] = o;
      o += out[l];
    }
    total = o;
  }
};

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ---- features ---------------------------------------------------------------
__device__ __forceinline__ double plog2(int64_t m) {
  int e;
  const double f = frexp((double)m, &e);   // m = f 2^e, 0.5 <= f < 1
  return __dadd_rn((double)(e - 1), __dsub_rn(__dmul_rn(2.0, f), 1.0));
}

struct PairTrees {
  const int32_t *tb, *te, *sb, *se;
  const double *tc, *sc, *tr, *sr;
};

// The FP64 features of pair (t, s); false if it cannot be approximated.
__device__ bool pair_features(const PairTrees& T, int t, int s, double kappa, double* f) {
  const double* ct = T.tc + (int64_t)t * 3;
  const double* cs = T.sc + (int64_t)s * 3;
  const double dx = __dsub_rn(ct[0], cs[0]), dy = __dsub_rn(ct[1], cs[1]), dz = __dsub_rn(ct[2], cs[2]);
  const double R = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
  if (!(R > 0.0)) return false;
  const double rt = T.tr[t], rs = T.sr[s];
  const double sep = __ddiv_rn(__dadd_rn(rt, rs), R);
  if (!(sep < 1.0)) return false;
  const double kr = __dmul_rn(kappa, R);
  f[0] = __ddiv_rn(plog2(T.te[t] - T.tb[t]), 16.0);
  f[1] = __ddiv_rn(plog2(T.se[s] - T.sb[s]), 16.0);
  f[2] = __ddiv_rn(rt, R);
  f[3] = __ddiv_rn(rs, R);
  f[4] = sep;
  f[5] = __ddiv_rn(kr, __dadd_rn(1.0, kr));
  return true;
}

// ---- network forward (one warp per sample) -----------------------------------
struct NetSmem {
  const __nv_bfloat16* w;   // W1 | W2 | W3 | W4, each stored transposed [in][out] in shared memory
  const float* b;           // b1 | b2 | b3 | b4
  int nout;
};

// z_j for neurons j = lane, lane + 32 (or lane < n for the output layer);
// Wt is the layer's weights transposed ([K][J]), so the lanes of a warp read
// consecutive entries; the sum over k runs in increasing order.
__device__ __forceinline__ float neuron(const __nv_bfloat16* Wt, const float* b, int j, int K, int J,
                                        const float* a) {
  float z = b[j];
  for (int k = 0; k < K; ++k) z = fmaf(__bfloat162float(Wt[(int64_t)k * J + j]), a[k], z);
  return z;
}

// x: 6 bf16-rounded inputs in shared memory; act: 2 x 64 floats of this warp.
// Writes y[lane] for lane < nout.  If keep != NULL the pre-activations and
// activations of each layer are stored there ([z1 a1 z2 a2 z3 a3] x 64).
__device__ float mlp_forward_warp(const NetSmem& net, const float* x, float* act, float* keep) {
  const int lane = threadIdx.x & 31;
  const __nv_bfloat16* W = net.w;
  const float* b = net.b;
  const int K[3] = {kFeatures, kHidden, kHidden};
  const float* in = x;
  float* bufs[2] = {act, act + kHidden};
  for (int l = 0; l < 3; ++l) {
    float* out = bufs[l & 1];
    float zz[2];
    for (int h = 0; h < 2; ++h) {
      const int j = lane + 32 * h;
      zz[h] = neuron(W, b, j, K[l], kHidden, in);
    }
    __syncwarp();
    for (int h = 0; h < 2; ++h) {
      const int j = lane + 32 * h;
      const float a = bf16r(zz[h] > 0.f ? zz[h] : 0.f);
      out[j] = a;
      if (keep) {
        keep[(2 * l) * kHidden + j] = zz[h];
        keep[(2 * l + 1) * kHidden + j] = a;
      }
    }
    __syncwarp();
    W += (int64_t)kHidden * K[l];
    b += kHidden;
    in = out;
  }
  return lane < net.nout ? neuron(W, b, lane, kHidden, net.nout, in) : 0.f;
}

// The same network for kSelTogether inputs x[m] at once (the sums in the same
// order): a neuron's sum is a chain of dependent multiply-adds, so one input at
// a time left the warp waiting, 3.8 us each.  act: 2 x 64 x kSelTogether floats.
constexpr int kSelTogether = 4;
__device__ __forceinline__ void mlp_forward_together(const NetSmem& net, const float* const (&x)[kSelTogether],
                                                     float* act, float (&y)[kSelTogether]) {
  constexpr int M = kSelTogether;
  const int lane = threadIdx.x & 31;
  const __nv_bfloat16* W = net.w;
  const float* b = net.b;
  float4* bufs[2] = {reinterpret_cast<float4*>(act), reinterpret_cast<float4*>(act + kHidden * M)};
  if (lane < kFeatures) bufs[1][lane] = make_float4(x[0][lane], x[1][lane], x[2][lane], x[3][lane]);
  __syncwarp();
  for (int l = 0; l < 3; ++l) {
    const int K = l == 0 ? kFeatures : kHidden;
    const float4* in = bufs[(l + 1) & 1];
    float z[2][M];
    for (int h = 0; h < 2; ++h)
      for (int m = 0; m < M; ++m) z[h][m] = b[lane + 32 * h];
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      const float4 a = in[k];
      const float am[M] = {a.x, a.y, a.z, a.w};
      for (int h = 0; h < 2; ++h) {
        const float w = __bfloat162float(W[(int64_t)k * kHidden + lane + 32 * h]);
        for (int m = 0; m < M; ++m) z[h][m] = fmaf(w, am[m], z[h][m]);
      }
    }
    for (int h = 0; h < 2; ++h) {
      for (int m = 0; m < M; ++m) z[h][m] = bf16r(z[h][m] > 0.f ? z[h][m] : 0.f);
      bufs[l & 1][lane + 32 * h] = make_float4(z[h][0], z[h][1], z[h][2], z[h][3]);
    }
    __syncwarp();
    W += (int64_t)kHidden * K;
    b += kHidden;
  }
  for (int m = 0; m < M; ++m) y[m] = 0.f;
  if (lane < net.nout) {
    const float4* in = bufs[0];
    for (int m = 0; m < M; ++m) y[m] = b[lane];
#pragma unroll 4
    for (int k = 0; k < kHidden; ++k) {
      const float4 a = in[k];
      const float am[M] = {a.x, a.y, a.z, a.w};
      const float w = __bfloat162float(W[(int64_t)k * net.nout + lane]);
      for (int m = 0; m < M; ++m) y[m] = fmaf(w, am[m], y[m]);
    }
  }
  __syncwarp();
}

// Load bf16 weights ([in][out] per layer) and float biases.
__device__ void load_net(const __nv_bfloat16* gw, const float* gb, int nout, __nv_bfloat16* sw, float* sb) {
  static_assert(kHidden % 8 == 0, "the weights of every layer are whole 16-byte words");
  const int nw = (int)(sel_weight_count(nout) / 8), nb = (int)sel_bias_count(nout);
  for (int i = threadIdx.x; i < nw; i += blockDim.x)
    reinterpret_cast<uint4*>(sw)[i] = reinterpret_cast<const uint4*>(gw)[i];
  for (int i = threadIdx.x; i < nb; i += blockDim.x) sb[i] = gb[i];
  __syncthreads();
}

// ---- selection inside the traversal -----------------------------------------
struct SelParams {
  int nout, ndeg;
  int np[kMaxDegrees];
  float lo[kFeatures], hi[kFeatures];
  float log_eps;
  double kappa;
  int net;   // 0: no network (MAC fallback everywhere)
};

// Per-warp scratch of k_select: the networks' activations, then the inputs and
// outputs of the warp's 32 pairs.
constexpr int kSelOutMax = 3 * kMaxDegrees;
constexpr int kSelActFloats = 2 * kHidden * kSelTogether;
constexpr int kSelWarpFloats = kSelActFloats + 32 * 8 + 32 * kSelOutMax;

__host__ __device__ inline size_t select_smem_bytes(int nout) {
  size_t w = (size_t)sel_weight_count(nout) * sizeof(__nv_bfloat16);
  w = (w + 15) / 16 * 16;
  return w + (size_t)(sel_bias_count(nout) + 3) / 4 * 4 * sizeof(float) +
         (size_t)kSelWarps * kSelWarpFloats * sizeof(float);
}

// A warp takes `per_warp` pairs at a time (32 at most): each lane computes its
// pair's features (the FP64 divisions and square root run on all lanes at once),
// the warp runs the network for the pairs inside the box, kSelTogether at a
// time, and each lane decides its own pair.  Same arithmetic as one pair per
// warp.  Bound by latency: a front of a few thousand pairs, 32 to a warp on a
// few SMs, took 0.14 ms; spread over all SMs, 4 networks at a time, 0.017 (50000 pairs 0.21 -> 0.06).
__global__ void k_select(const int2* __restrict__ pairs, int32_t F, PairTrees T, SelParams sp,
                         const __nv_bfloat16* __restrict__ gw, const float* __restrict__ gb, int per_warp,
                         int16_t* __restrict__ choice) {
  extern __shared__ __align__(16) unsigned char sraw[];
  __nv_bfloat16* sw = reinterpret_cast<__nv_bfloat16*>(sraw);
  size_t wbytes = ((size_t)sel_weight_count(sp.nout) * sizeof(__nv_bfloat16) + 15) / 16 * 16;
  float* sb = reinterpret_cast<float*>(sraw + wbytes);
  float* swarp = sb + (sel_bias_count(sp.nout) + 3) / 4 * 4;   // 16-byte aligned
  if (sp.net) load_net(gw, gb, sp.nout, sw, sb);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* act = swarp + warp * kSelWarpFloats;
  float* xs = act + kSelActFloats;    // [32][8]
  float* ys = xs + 32 * 8;            // [32][kSelOutMax]
  const NetSmem net{sw, sb, sp.nout};
  const int64_t stride = (int64_t)gridDim.x * kSelWarps * per_warp;
  for (int64_t base = ((int64_t)blockIdx.x * kSelWarps + warp) * per_warp; base < F; base += stride) {
    const int64_t i = lane < per_warp ? base + lane : F;
    int state = 0;   // 0 no approximation, 1 fallback, 2 network
    int t = 0, s = 0;
    if (i < F) {
      t = pairs[i].x;
      s = pairs[i].y;
      double f[kFeatures];
      if (pair_features(T, t, s, sp.kappa, f)) {
        state = sp.net ? 2 : 1;
        for (int d = 0; d < kFeatures; ++d) {
          const float xd = bf16r(__double2float_rn(f[d]));
          xs[lane * 8 + d] = xd;
          if (xd < sp.lo[d] || xd > sp.hi[d]) state = 1;
        }
      }
    }
    __syncwarp();
    unsigned todo = __ballot_sync(0xffffffffu, state == 2);
    while (todo) {
      int j[kSelTogether];
      const float* x[kSelTogether];
      float y[kSelTogether];
      for (int m = 0; m < kSelTogether; ++m) {       // the last round repeats its last pair
        j[m] = todo ? __ffs(todo) - 1 : j[m > 0 ? m - 1 : 0];
        todo &= todo - 1;
        x[m] = xs + j[m] * 8;
      }
      mlp_forward_together(net, x, act, y);
      if (lane < sp.nout)
        for (int m = 0; m < kSelTogether; ++m) ys[j[m] * kSelOutMax + lane] = y[m];
      __syncwarp();
    }
    if (i < F) {
      int16_t c = state == 0 ? kChoiceNoApprox : kChoiceFallback;
      if (state == 2) {
        const float* y = ys + lane * kSelOutMax;
        const int64_t ct = T.te[t] - T.tb[t], cs = T.se[s] - T.sb[s];
        int best = -1;
        int64_t best_cost = 0;
        for (int di = 0; di < sp.ndeg; ++di) {
          const int64_t np = sp.np[di];
          const int64_t cost[3] = {ct * np, np * cs, np * np};
          for (int ty = 0; ty < 3; ++ty)
            if (y[3 * di + ty] <= sp.log_eps && (best < 0 || cost[ty] < best_cost)) {
              best = 1 + 3 * di + ty;
              best_cost = cost[ty];
            }
        }
        c = best < 0 ? kChoiceNoApprox : (ct * cs <= best_cost ? (int16_t)0 : (int16_t)best);
      }
      choice[i] = c;
    }
    __syncwarp();
  }
}

static inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

static PairTrees pair_trees(const bldtt_plan* p) {
  return PairTrees{p->tt.begin, p->tt.end, p->st.begin, p->st.end,
                   p->tt.center, p->st.center, p->tt.radius, p->st.radius};
}

int select_pairs(bldtt_plan* p, const int2* pairs, int32_t F, int16_t* choice, cudaStream_t s) {
  SelParams sp{};
  sp.nout = p->sel_nout;
  sp.ndeg = p->deg.n;
  for (int i = 0; i < p->deg.n; ++i) sp.np[i] = p->deg.np[i];
  for (int d = 0; d < kFeatures; ++d) {
    sp.lo[d] = p->sel_lo[d];
    sp.hi[d] = p->sel_hi[d];
  }
  sp.log_eps = p->sel_log_eps;
  sp.kappa = p->kappa;
  sp.net = p->selector_net ? 1 : 0;
  const size_t sm = select_smem_bytes(p->sel_nout);
  BL_CUDA(cudaFuncSetAttribute(k_select, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  int sms = 0;
  BL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device));
  const int64_t spread = (F + (int64_t)sms * 2 * kSelWarps - 1) / ((int64_t)sms * 2 * kSelWarps);
  const int per_warp = (int)std::min<int64_t>(32, (spread + kSelTogether - 1) / kSelTogether * kSelTogether);
  unsigned g = nblk(F, kSelWarps * per_warp);
  if (g > 4096) g = 4096;
  k_select<<<g, 32 * kSelWarps, sm, s>>>(pairs, F, pair_trees(p), sp,
                                          reinterpret_cast<const __nv_bfloat16*>(p->sel_w), p->sel_b,
                                          per_warp, choice);
  BL_LAUNCHED(p->setup_counter.launches);
  return BLDTT_OK;
}

// ---- training ------------------------------------------------------------------
// The master parameters of all layers into shared memory as bf16, per layer Wt[k][j] (the
// forward pass: a warp's lanes read neighbouring neurons) and, if Wr is given,
// Wr[j][k] (the backward pass: neighbouring inputs).
__device__ void load_params(const float* __restrict__ params, const ParamLayout& L, int nout, __nv_bfloat16* wt,
                            __nv_bfloat16* wr, float* sb) {
  const int K[4] = {kFeatures, kHidden, kHidden, kHidden};
  const int J[4] = {kHidden, kHidden, kHidden, nout};
  int o = 0, ob = 0;
  for (int l = 0; l < 4; ++l) {
    const int n = K[l] * J[l];
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const __nv_bfloat16 v = __float2bfloat16_rn(params[L.w[l] + i]);
      wt[o + (i % K[l]) * J[l] + i / K[l]] = v;
      if (wr) wr[o + i] = v;
    }
    for (int i = threadIdx.x; i < J[l]; i += blockDim.x) sb[ob + i] = params[L.b[l] + i];
    o += n;
    ob += J[l];
  }
}

__host__ __device__ inline size_t train_weight_bytes(int nout) {
  return ((size_t)sel_weight_count(nout) * sizeof(__nv_bfloat16) + 15) / 16 * 16;
}
// Per-warp scratch of the training kernels: two activation or gradient rows and the inputs.
constexpr int kTrainWarpFloats = 2 * kHidden + 8;
__host__ __device__ inline size_t train_smem_bytes(int nout, bool backward) {
  return train_weight_bytes(nout) * (backward ? 2 : 1) + (size_t)sel_bias_count(nout) * sizeof(float) +
         (size_t)kSelWarps * kTrainWarpFloats * sizeof(float);
}

// What a sample's backward pass and the weight gradients read: [x(8) | z1 a1 z2
// a2 z3 a3 (6 x 64)] and [dL/dy (24) | dL/dz3, dL/dz2, dL/dz1 (3 x 64)].
constexpr int kKeep = 8 + 6 * kHidden;
constexpr int kGradOut = 24;
constexpr int kGradRow = kGradOut + 3 * kHidden;

__global__ void k_mlp_forward(const float* __restrict__ xin, int64_t B, const float* __restrict__ params,
                              ParamLayout L, int nout, float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char sraw[];
  __nv_bfloat16* sw = reinterpret_cast<__nv_bfloat16*>(sraw);
  float* sb = reinterpret_cast<float*>(sraw + train_weight_bytes(nout));
  float* swarp = sb + sel_bias_count(nout);
  load_params(params, L, nout, sw, nullptr, sb);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* act = swarp + warp * kTrainWarpFloats;
  float* x = act + 2 * kHidden;
  const NetSmem net{sw, sb, nout};
  for (int64_t i = (int64_t)blockIdx.x * kSelWarps + warp; i < B; i += (int64_t)gridDim.x * kSelWarps) {
    if (lane < kFeatures) x[lane] = bf16r(xin[i * kFeatures + lane]);
    __syncwarp();
    const float v = mlp_forward_warp(net, x, act, nullptr);
    if (lane < nout) y[i * nout + lane] = v;
    __syncwarp();
  }
}

// Forward and backward pass of every sample, one warp each, in one launch (the
// layers used to be a launch each: conversion, forward, loss, output gradient
// and three backward steps).  The output gradient is left undivided by the mask
// count, dL/dy cnt = 2 mask (y - T), because the count is known only after all
// samples; the weight gradients divide their sums.  Backward through a layer:
// gz[k] = (sum_j g[j] W[j][k]) [z[k] > 0], j in increasing order.  part[block] =
// (sum mask, sum (mask (y - T))^2) of the block's samples.
__global__ void __launch_bounds__(32 * kSelWarps) k_train_samples(
    const float* __restrict__ xin, const float* __restrict__ T, const float* __restrict__ mask, int64_t B,
    const float* __restrict__ params, ParamLayout L, int nout, float* __restrict__ keep,
    float* __restrict__ grad, double2* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char sraw[];
  __shared__ double2 sred[kSelWarps];
  const size_t wbytes = train_weight_bytes(nout);
  __nv_bfloat16* wt = reinterpret_cast<__nv_bfloat16*>(sraw);
  __nv_bfloat16* wr = reinterpret_cast<__nv_bfloat16*>(sraw + wbytes);
  float* sb = reinterpret_cast<float*>(sraw + 2 * wbytes);
  float* swarp = sb + sel_bias_count(nout);
  load_params(params, L, nout, wt, wr, sb);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* act = swarp + warp * kTrainWarpFloats;
  float* x = act + 2 * kHidden;
  const NetSmem net{wt, sb, nout};
  double sm = 0.0, sl = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * kSelWarps + warp; i < B; i += (int64_t)gridDim.x * kSelWarps) {
    float* kp = keep + i * kKeep;
    float* gr = grad + i * kGradRow;
    if (lane < kFeatures) {
      x[lane] = bf16r(xin[i * kFeatures + lane]);
      kp[lane] = x[lane];
    }
    __syncwarp();
    const float y = mlp_forward_warp(net, x, act, kp + 8);
    float* g = act;                            // dL/dy, then the hidden layers' dL/dz, alternating
    float* gn = act + kHidden;
    __syncwarp();
    if (lane < nout) {
      const float mk = mask[i * nout + lane], t = T[i * nout + lane];
      const float v = 2.f * mk * (y - t);
      g[lane] = v;
      gr[lane] = v;
      const double d = (double)mk * ((double)y - (double)t);
      sm += mk;
      sl += d * d;
    }
    __syncwarp();
    const __nv_bfloat16* W = wr + kHidden * kFeatures + 2 * kHidden * kHidden;   // the output layer's
    for (int l = 3; l >= 1; --l) {
      const int J = l == 3 ? nout : kHidden;
      float v[2];
      for (int h = 0; h < 2; ++h) {
        const int k = lane + 32 * h;
        float a = 0.f;
        for (int j = 0; j < J; ++j) a = fmaf(g[j], __bfloat162float(W[j * kHidden + k]), a);
        // this thread wrote its own pre-activations z[k] of layer l
        v[h] = kp[8 + 2 * (l - 1) * kHidden + k] > 0.f ? a : 0.f;
      }
      for (int h = 0; h < 2; ++h) {
        gn[lane + 32 * h] = v[h];
        gr[kGradOut + (3 - l) * kHidden + lane + 32 * h] = v[h];
      }
      __syncwarp();
      float* tmp = g;
      g = gn;
      gn = tmp;
      W -= kHidden * kHidden;
    }
  }
  for (int o = 16; o; o >>= 1) {
    sm += __shfl_xor_sync(0xffffffffu, sm, o);
    sl += __shfl_xor_sync(0xffffffffu, sl, o);
  }
  if (lane == 0) sred[warp] = make_double2(sm, sl);
  __syncthreads();
  if (threadIdx.x == 0) {
    double2 v = sred[0];
    for (int w = 1; w < kSelWarps; ++w) {
      v.x += sred[w].x;
      v.y += sred[w].y;
    }
    part[blockIdx.x] = v;
  }
}

// Weight and bias gradients of all layers in one launch: dW[j][k] = sum_b
// g[b][j] a[b][k] / cnt, db[j] = sum_b g[b][j] / cnt, each sum in float over
// kGradB samples, then over those sums, in order.  A block takes kGradJ neurons of one layer, a thread one
// input k of them (thread 64: the biases), so a sample's activation is read
// once for kGradJ products; kGradB samples at a time come through shared memory
// (one thread per weight reading both factors from memory took 4 x ~100 us at
// 1024 samples, the latency of 1024 dependent steps).
constexpr int kGradJ = 4;
constexpr int kGradB = 64;
constexpr int kGradThreads = 96;
__global__ void __launch_bounds__(kGradThreads) k_weight_grads(const float* __restrict__ keep,
                                                              const float* __restrict__ grad, int64_t B,
                                                              ParamLayout L, int nout,
                                                              const double2* __restrict__ part, int nparts,
                                                              float* __restrict__ out, float* __restrict__ loss) {
  __shared__ __align__(16) float sa[2][kGradB][kHidden];
  __shared__ __align__(16) float sg[2][kGradB][kGradJ];
  __shared__ float scnt;
  const int per = kHidden / kGradJ;             // blocks per hidden layer
  const int l = blockIdx.x / per < 3 ? blockIdx.x / per : 3;
  const int j0 = (blockIdx.x - l * per) * kGradJ;
  const int J = l == 3 ? nout : kHidden, K = l == 0 ? kFeatures : kHidden;
  const int aoff = l == 0 ? 0 : 8 + (2 * l - 1) * kHidden;               // x, a1, a2, a3
  const int goff = l == 3 ? 0 : kGradOut + (2 - l) * kHidden;            // dL/dy, dL/dz3, dL/dz2, dL/dz1
  const int tid = threadIdx.x;
  if (tid < 32) {                               // the mask count and the loss, in block order
    double m = 0.0, q = 0.0;
    for (int i = tid; i < nparts; i += 32) {
      m += part[i].x;
      q += part[i].y;
    }
    for (int o = 16; o; o >>= 1) {
      m += __shfl_xor_sync(0xffffffffu, m, o);
      q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    if (tid == 0) {
      const double cnt = m > 1.0 ? m : 1.0;
      scnt = (float)cnt;
      if (blockIdx.x == 0 && loss) *loss = (float)(q / cnt);
    }
  }
  auto stage = [&](int buf, int64_t base) {     // asynchronous copies of one set of samples
    const int n = (int)min((int64_t)kGradB, B - base);
    for (int i = tid; i < n * (kHidden / 4); i += kGradThreads) {
      const int b = i / (kHidden / 4), k = (i % (kHidden / 4)) * 4;
      if (k < (K + 3) / 4 * 4) {
        const float* src = keep + (base + b) * kKeep + aoff + k;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&sa[buf][b][k])),
                     "l"(src));
      }
    }
    for (int b = tid; b < n; b += kGradThreads) {
      const float* src = grad + (base + b) * kGradRow + goff + j0;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(&sg[buf][b][0])),
                   "l"(src));
    }
    asm volatile("cp.async.commit_group;");
  };
  float total[kGradJ] = {0.f, 0.f, 0.f, 0.f};
  const bool mine = tid < K || tid == kHidden;
  stage(0, 0);
  for (int64_t base = 0, it = 0; base < B; base += kGradB, ++it) {
    const int buf = (int)(it & 1);
    if (base + kGradB < B) {
      stage(buf ^ 1, base + kGradB);
      asm volatile("cp.async.wait_group 1;");
    } else {
      asm volatile("cp.async.wait_group 0;");
    }
    __syncthreads();
    const int n = (int)min((int64_t)kGradB, B - base);
    if (mine) {
      float acc[kGradJ] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
      for (int b = 0; b < n; ++b) {
        const float a = tid < kHidden ? sa[buf][b][tid] : 1.f;
        const float4 g = *reinterpret_cast<const float4*>(sg[buf][b]);
        acc[0] = fmaf(g.x, a, acc[0]);
        acc[1] = fmaf(g.y, a, acc[1]);
        acc[2] = fmaf(g.z, a, acc[2]);
        acc[3] = fmaf(g.w, a, acc[3]);
      }
      for (int r = 0; r < kGradJ; ++r) total[r] += acc[r];
    }
    __syncthreads();
  }
  if (!mine) return;
  for (int r = 0; r < kGradJ; ++r) {
    const int j = j0 + r;
    if (j >= J) break;
    if (tid < kHidden)
      out[L.w[l] + (int64_t)j * K + tid] = total[r] / scnt;
    else
      out[L.b[l] + j] = total[r] / scnt;
  }
}

__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, int64_t n, float lr, float c1, float c2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float b1 = 0.9f, b2 = 0.999f;
  const float mi = b1 * m[i] + (1.f - b1) * g[i];
  const float vi = b2 * v[i] + (1.f - b2) * g[i] * g[i];
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

// ---- per-pair error labels ------------------------------------------------------
template <int KERN>
__device__ __forceinline__ double g64(double dx, double dy, double dz, double kappa) {
  const double r2 = dx * dx + dy * dy + dz * dz;
  if (!(r2 > 0.0)) return 0.0;
  if (KERN == BLDTT_REG_COULOMB) return rsqrt(r2 + kappa * kappa);
  const double ri = rsqrt(r2);
  if (KERN == BLDTT_COULOMB) return ri;
  if (KERN == BLDTT_OSCILLATORY) return ri * sin(kappa * (r2 * ri));
  if (KERN == BLDTT_YUKAWA) return ri * exp(-kappa * (r2 * ri));
  return 1.0 + dx - 2.0 * dy + 3.0 * dz + dx * dy - dy * dz + dx * dx * dz * dz - 0.5 * dy * dy;
}

__device__ __forceinline__ double bary_w(int k, int n) {
  const double w = (k == 0 || k == n) ? 0.5 : 1.0;
  return (k & 1) ? -w : w;
}
// L_k(x), k = 0..n, on the grid `nodes` with the coincident-point guard.
__device__ void basis(double x, const double* nodes, int n, double* out, int stride) {
  double sum = 0.0;
  int hit = -1;
  for (int k = 0; k <= n; ++k) {
    const double d = x - nodes[k];
    if (d == 0.0 && hit < 0) hit = k;
    const double r = d == 0.0 ? 0.0 : bary_w(k, n) / d;
    out[k * stride] = r;
    sum += r;
  }
  for (int k = 0; k <= n; ++k) out[k * stride] = hit >= 0 ? (k == hit ? 1.0 : 0.0) : out[k * stride] / sum;
}

constexpr int kErrThreads = 256;
constexpr int kErrChunk = 32;
constexpr int kErrMaxSources = 4096;   // larger source clusters: an evenly strided subset

struct ErrTrees {
  const int32_t *tb, *te, *sb, *se;
  const double *tbox, *sbox;
  const double *tx, *ty, *tz, *sx, *sy, *sz, *q;
};

// One block per (pair, degree): the relative l2 errors of PC, CP and CC at
// degree d against the exact pair sum (Eq. (6)), on up to S target samples
// spread evenly over C_t.  A source cluster of more than kErrMaxSources
// particles is represented by every stride-th particle (stride =
// ceil(|C_s| / kErrMaxSources)) in the exact sum and in all three
// approximations alike.  err[(pair * ndeg + di) * 3 + type].
template <int KERN>
__global__ void __launch_bounds__(kErrThreads) k_pair_errors(const int32_t* __restrict__ pairs, int64_t npairs,
                                                            ErrTrees T, DegreeSet deg, int S, double kappa,
                                                            double* __restrict__ err) {
  extern __shared__ double sm[];
  const int64_t blk = blockIdx.x;
  const int64_t pi = blk / deg.n;
  const int di = (int)(blk % deg.n);
  if (pi >= npairs) return;
  const int t = pairs[2 * pi], s = pairs[2 * pi + 1];
  const int d = deg.d[di], P = d + 1, np = P * P * P;
  const int32_t tb = T.tb[t], nt = T.te[t] - tb, sb = T.sb[s], ns_all = T.se[s] - sb;
  const int32_t sst = (ns_all + kErrMaxSources - 1) / kErrMaxSources;   // source stride
  const int32_t ns = (ns_all + sst - 1) / sst;                          // sources used
  const int m = nt < S ? nt : S;
  double* tn = sm;                     // [3][P] target nodes
  double* sn = tn + 3 * P;             // [3][P] source nodes
  double* qh = sn + 3 * P;             // [np] proxy charges of C_s
  double* ph = qh + np;                // [np] CP potentials at C_t's proxies
  double* pc2 = ph + np;               // [np] CC potentials at C_t's proxies
  double* Bj = pc2 + np;               // [3][P][kErrChunk] source basis of a chunk
  double* Bm = Bj + 3 * P * kErrChunk; // [3][P][S] target basis at the samples
  double* sv = Bm + 3 * P * S;         // [4][S]: exact, PC, CP, CC at the samples
  double* red = sv + 4 * S;            // [3][2] error sums
  for (int i = threadIdx.x; i < 3 * P; i += blockDim.x) {
    const int dd = i / P, k = i % P;
    const double* bt = T.tbox + (int64_t)t * 6;
    const double* bs = T.sbox + (int64_t)s * 6;
    double c = __dmul_rn(__dadd_rn(bt[dd], bt[3 + dd]), 0.5), h = __dmul_rn(__dsub_rn(bt[3 + dd], bt[dd]), 0.5);
    tn[i] = __dadd_rn(c, __dmul_rn(h, cheb_point(k, d)));
    c = __dmul_rn(__dadd_rn(bs[dd], bs[3 + dd]), 0.5);
    h = __dmul_rn(__dsub_rn(bs[3 + dd], bs[dd]), 0.5);
    sn[i] = __dadd_rn(c, __dmul_rn(h, cheb_point(k, d)));
  }
  for (int i = threadIdx.x; i < np; i += blockDim.x) qh[i] = 0.0;
  __syncthreads();
  // Eq. (9): proxy charges of C_s at degree d.
  for (int base = 0; base < ns; base += kErrChunk) {
    const int cnt = min(kErrChunk, ns - base);
    for (int task = threadIdx.x; task < 3 * kErrChunk; task += blockDim.x) {
      const int dd = task / kErrChunk, j = task % kErrChunk;
      const double* crd = dd == 0 ? T.sx : (dd == 1 ? T.sy : T.sz);
      if (j < cnt)
        basis(crd[sb + (int64_t)(base + j) * sst], sn + dd * P, d, Bj + (dd * P) * kErrChunk + j, kErrChunk);
      else
        for (int k = 0; k < P; ++k) Bj[(dd * P + k) * kErrChunk + j] = 0.0;
    }
    __syncthreads();
    for (int o = threadIdx.x; o < np; o += blockDim.x) {
      const int k1 = o / (P * P), k2 = (o / P) % P, k3 = o % P;
      double a = 0.0;
      for (int j = 0; j < cnt; ++j)
        a += Bj[k1 * kErrChunk + j] * Bj[(P + k2) * kErrChunk + j] * Bj[(2 * P + k3) * kErrChunk + j] *
             T.q[sb + (int64_t)(base + j) * sst];
      qh[o] += a;
    }
    __syncthreads();
  }
  // Target samples and their basis; the exact and PC sums at the samples.
  for (int task = threadIdx.x; task < 3 * m; task += blockDim.x) {
    const int dd = task / m, i = task % m;
    const int64_t pos = tb + (int64_t)i * nt / m;
    const double* crd = dd == 0 ? T.tx : (dd == 1 ? T.ty : T.tz);
    basis(crd[pos], tn + dd * P, d, Bm + (dd * P) * S + i, S);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int i = warp; i < m; i += nw) {
    const int64_t pos = tb + (int64_t)i * nt / m;
    const double x = T.tx[pos], y = T.ty[pos], z = T.tz[pos];
    double ex = 0.0, pc = 0.0;
    for (int j = lane; j < ns; j += 32) {
      const int64_t y0 = sb + (int64_t)j * sst;
      ex += g64<KERN>(x - T.sx[y0], y - T.sy[y0], z - T.sz[y0], kappa) * T.q[y0];
    }
    for (int o = lane; o < np; o += 32) {
      const int k1 = o / (P * P), k2 = (o / P) % P, k3 = o % P;
      pc += g64<KERN>(x - sn[k1], y - sn[P + k2], z - sn[2 * P + k3], kappa) * qh[o];
    }
    for (int off = 16; off; off >>= 1) {
      ex += __shfl_xor_sync(0xffffffffu, ex, off);
      pc += __shfl_xor_sync(0xffffffffu, pc, off);
    }
    if (lane == 0) {
      sv[i] = ex;
      sv[S + i] = pc;
    }
  }
  // CP (Eq. (12)) and CC (Eq. (15)) at C_t's proxies.
  for (int o = threadIdx.x; o < np; o += blockDim.x) {
    const int k1 = o / (P * P), k2 = (o / P) % P, k3 = o % P;
    const double x = tn[k1], y = tn[P + k2], z = tn[2 * P + k3];
    double cp = 0.0, cc = 0.0;
    for (int j = 0; j < ns; ++j) {
      const int64_t y0 = sb + (int64_t)j * sst;
      cp += g64<KERN>(x - T.sx[y0], y - T.sy[y0], z - T.sz[y0], kappa) * T.q[y0];
    }
    for (int r = 0; r < np; ++r) {
      const int r1 = r / (P * P), r2 = (r / P) % P, r3 = r % P;
      cc += g64<KERN>(x - sn[r1], y - sn[P + r2], z - sn[2 * P + r3], kappa) * qh[r];
    }
    ph[o] = cp;
    pc2[o] = cc;
  }
  __syncthreads();
  // Interpolate to the samples (Eq. (21)).
  for (int i = warp; i < m; i += nw) {
    double a = 0.0, b = 0.0;
    for (int o = lane; o < np; o += 32) {
      const int k1 = o / (P * P), k2 = (o / P) % P, k3 = o % P;
      const double L = Bm[k1 * S + i] * Bm[(P + k2) * S + i] * Bm[(2 * P + k3) * S + i];
      a += L * ph[o];
      b += L * pc2[o];
    }
    for (int off = 16; off; off >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, off);
      b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (lane == 0) {
      sv[2 * S + i] = a;
      sv[3 * S + i] = b;
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double num = 0.0, den = 0.0;
    for (int i = 0; i < m; ++i) {
      const double e = sv[i], dlt = sv[(1 + threadIdx.x) * S + i] - e;
      num += dlt * dlt;
      den += e * e;
    }
    red[threadIdx.x] = den > 0.0 ? sqrt(num / den) : (num > 0.0 ? INFINITY : 0.0);
  }
  __syncthreads();
  if (threadIdx.x < 3) err[(pi * deg.n + di) * 3 + threadIdx.x] = red[threadIdx.x];
}

static size_t err_smem_bytes(int P, int S) {
  const int np = P * P * P;
  return sizeof(double) * (size_t)(6 * P + 3 * np + 3 * P * kErrChunk + 3 * P * S + 4 * S + 8);
}

__global__ void k_pair_features(const int32_t* __restrict__ pairs, int64_t n, PairTrees T, double kappa,
                                double* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double f[kFeatures];
  const bool ok = pair_features(T, pairs[2 * i], pairs[2 * i + 1], kappa, f);
  for (int d = 0; d < kFeatures; ++d) out[i * kFeatures + d] = ok ? f[d] : NAN;
}

}  // namespace bldtt

using namespace bldtt;

extern "C" {

int64_t bldtt_selector_param_count(int num_degrees) {
  if (num_degrees < 1 || num_degrees > kMaxDegrees) return -1;
  return ParamLayout(3 * num_degrees).total;
}

int bldtt_mlp_forward(const float* params, int num_out, const float* x, int64_t batch, float* y,
                      void* cuda_stream) {
  if (!params || !x || !y || batch < 1 || num_out < 1 || num_out > 3 * kMaxDegrees) {
    set_error("mlp_forward: bad arguments");
    return BLDTT_EINVAL;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const size_t sm = train_smem_bytes(num_out, false);
  k_mlp_forward<<<nblk(batch, kSelWarps) > 4096 ? 4096 : nblk(batch, kSelWarps), 32 * kSelWarps, sm, s>>>(
      x, batch, params, ParamLayout(num_out), num_out, y);
  int64_t dummy = 0;
  BL_LAUNCHED(dummy);
  return BLDTT_OK;
}

int bldtt_mlp_gradients(const float* params, int num_out, const float* x, const float* target,
                        const float* mask, int64_t batch, float* grads, float* loss, void* cuda_stream) {
  if (!params || !x || !target || !mask || !grads || batch < 1 || num_out < 1 ||
      num_out > 3 * kMaxDegrees) {
    set_error("mlp_gradients: bad arguments");
    return BLDTT_EINVAL;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const ParamLayout L(num_out);
  const unsigned blocks = nblk(batch, kSelWarps) > 4096 ? 4096 : nblk(batch, kSelWarps);
  float *keep = nullptr, *grad = nullptr;
  double2* part = nullptr;
  Arena scratch;                       // freed, in stream order, when it goes out of scope
  scratch.add(&keep, (size_t)batch * kKeep);
  scratch.add(&grad, (size_t)batch * kGradRow);
  scratch.add(&part, blocks);
  BL_TRY(scratch.alloc(s));
  int64_t dummy = 0;
  const size_t sm = train_smem_bytes(num_out, true);
  k_train_samples<<<blocks, 32 * kSelWarps, sm, s>>>(x, target, mask, batch, params, L, num_out, keep, grad, part);
  BL_LAUNCHED(dummy);
  const unsigned jb = 3 * (kHidden / kGradJ) + nblk(num_out, kGradJ);
  k_weight_grads<<<jb, kGradThreads, 0, s>>>(keep, grad, batch, L, num_out, part, (int)blocks, grads, loss);
  BL_LAUNCHED(dummy);
  return BLDTT_OK;
}

int bldtt_mlp_adam(float* params, float* m, float* v, const float* grads, int64_t count, int step,
                   float lr, void* cuda_stream) {
  if (!params || !m || !v || !grads || count < 1 || step < 1) {
    set_error("mlp_adam: bad arguments");
    return BLDTT_EINVAL;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const float c1 = 1.f - powf(0.9f, (float)step), c2 = 1.f - powf(0.999f, (float)step);
  k_adam<<<nblk(count, 256), 256, 0, s>>>(params, m, v, grads, count, lr, c1, c2);
  int64_t dummy = 0;
  BL_LAUNCHED(dummy);
  return BLDTT_OK;
}

int bldtt_pair_features(bldtt_plan* p, int64_t npairs, const int32_t* pairs, double* features,
                        void* cuda_stream) {
  if (!p || !pairs || !features || npairs < 1) {
    set_error("pair_features: bad arguments");
    return BLDTT_EINVAL;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  k_pair_features<<<nblk(npairs, 128), 128, 0, s>>>(pairs, npairs, pair_trees(p), p->kappa, features);
  int64_t dummy = 0;
  BL_LAUNCHED(dummy);
  return BLDTT_OK;
}

int bldtt_pair_errors(bldtt_plan* p, int64_t npairs, const int32_t* pairs, int samples, int num_degrees,
                      const int* degrees, double* err, void* cuda_stream) {
  if (!p || !pairs || !err || !degrees || npairs < 1 || samples < 1 || samples > 256 ||
      num_degrees < 1 || num_degrees > kMaxDegrees) {
    set_error("pair_errors: bad arguments");
    return BLDTT_EINVAL;
  }
  DegreeSet deg;
  deg.n = num_degrees;
  int pmax = 1;
  for (int i = 0; i < num_degrees; ++i) {
    if (degrees[i] < 1 || degrees[i] > kMaxDegree) {
      set_error("pair_errors: degree %d outside [1, %d]", degrees[i], kMaxDegree);
      return BLDTT_EINVAL;
    }
    deg.d[i] = degrees[i];
    deg.np[i] = (degrees[i] + 1) * (degrees[i] + 1) * (degrees[i] + 1);
    if (degrees[i] + 1 > pmax) pmax = degrees[i] + 1;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  ErrTrees T{p->tt.begin, p->tt.end, p->st.begin, p->st.end, p->tt.box, p->st.box,
             p->tt.x, p->tt.y, p->tt.z, p->st.x, p->st.y, p->st.z, p->q_tree};
  const size_t sm = err_smem_bytes(pmax, samples);
  if (sm > 200 * 1024) {
    set_error("pair_errors: degree and sample count need %zu bytes of shared memory", sm);
    return BLDTT_EINVAL;
  }
  const int64_t blocks = npairs * num_degrees;
  int64_t dummy = 0;
#define BL_ERR_LAUNCH(K)                                                                              \
  do {                                                                                               \
    BL_CUDA(cudaFuncSetAttribute(k_pair_errors<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)); \
    k_pair_errors<K><<<(unsigned)blocks, kErrThreads, sm, s>>>(pairs, npairs, T, deg, samples, p->kappa, err); \
    BL_LAUNCHED(dummy);                                                                              \
  } while (0)
  switch (p->kernel) {
    case BLDTT_COULOMB: BL_ERR_LAUNCH(BLDTT_COULOMB); break;
    case BLDTT_YUKAWA: BL_ERR_LAUNCH(BLDTT_YUKAWA); break;
    case BLDTT_OSCILLATORY: BL_ERR_LAUNCH(BLDTT_OSCILLATORY); break;
    case BLDTT_REG_COULOMB: BL_ERR_LAUNCH(BLDTT_REG_COULOMB); break;
    default: BL_ERR_LAUNCH(BLDTT_TEST_POLY); break;
  }
#undef BL_ERR_LAUNCH
  return BLDTT_OK;
}

}  // extern "C"
