// PP, PC, CP and CC interactions (Sec. 2.4, Eqs. (6), (8), (12), (15)) in one
// persistent kernel, launched once per kernel type of the plan.
//
// All four interaction types are "targets x sources" sums (Sec. 3.3): the
// targets are particles (PP, PC) or proxy points (CP, CC) of a target cluster,
// the sources are particles (PP, CP) or proxy points with proxy charges
// (PC, CC) of a source cluster.  A work item is a tile of up to kTile targets
// of one target cluster; its sources are the concatenation of
//   particle tiles: PP and PC (every degree) entries of the leaf and of every
//                   ancestor (an entry on an ancestor applies to all its
//                   particles)
//   proxy tiles:    CP and CC entries of one degree on the cluster itself
//                   (the targets are that degree's proxy points).
// Each item owns its outputs and its summation order is fixed.
//
// An item with many source chunks is split into tasks over its chunks
// (plan_parts), so that a plan with few items still fills the device and the
// last tasks are short: 2E4 points make ~200 items for 152 SMs x 6 CTAs, and
// the launch would last as long as the longest of them (this kernel on a GB300,
// whole items and tasks: FP64 at 2E4 points, n = 4, 9.5 and 2.3 ms; FP32 on a sphere
// of 2E4 0.31 and 0.14 ms; 1E6 points 31.7 and 31.2 ms).
//
// Per CTA, one producer warp takes tasks from a global counter, walks their
// lists and streams the sources, kChunk at a time, from the source pool into
// a shared-memory ring (3 or 4 stages) with cp.async.bulk (TMA) copies that
// complete on mbarriers; NCW consumer warps evaluate G for K targets per
// thread against every staged source (NCW * 32 * K == kTile).
//
// FP32_BULK: every chunk of kChunk pool entries has its own frame centre c, a
// float near the chunk (particles inside a source leaf are in Morton order, so
// a chunk is spatially compact).  Entries hold y - c in FP32, formed from the
// split y = hi + lo (hi = fl(y), lo = fl(y - hi)) as fl(fl(hi - c) + lo), and
// are stored as pair records {x0,x1, y0,y1, z0,z1, q0,q1} so that one target
// meets two sources in packed f32x2 arithmetic (7 packed FP32 instructions and
// 2 MUFU.RSQ per two Coulomb evaluations).  Targets keep the same split and
// are moved into each chunk's frame with the same expression, so the
// coordinate rounding error is relative to the chunk size, and a target that
// coincides with a source gets exactly the same FP32 coordinates (r = 0).
// The two halves of the packed accumulator are two interleaved partial sums;
// each chunk's sum is added into an FP64 accumulator.
// FP64: pool entries are double4 (y, q) in absolute coordinates.
// Chunks carry their real source count, so padding is neither copied nor
// evaluated.
//
// Close pairs (FP32_BULK): every chunk also carries its half-extents and a
// near distance tau; the producer flags the 32-target groups whose box comes
// within tau of a particle chunk and then also stages the chunk's frame
// residuals; a flagged warp adds the residuals of both points to the
// coordinate differences of its near targets (see eval_chunk_f32).
//
// A pair at distance 0 contributes nothing.  Only a target near a chunk (or in
// it) can meet one, so the guard stands in the careful path alone, for warps
// with a target inside the chunk's box (and in proxy chunks of plans whose
// clusters may overlap); the plain path evaluates unguarded, and a sum that is
// not finite all the same (r^2 underflows, a charge beyond float) is redone with
// such pairs left out.  The arithmetic and the order are the same throughout, so a target's
// result never depends on which warp or consumer layout evaluated it.
#include <type_traits>

#include "fixed64.cuh"
#include "internal.cuh"

namespace bldtt {

constexpr uint64_t kWaitNs = 20ull * 1000ull * 1000ull * 1000ull;   // 20 s bound on any wait

struct InteractView {
  const int4* items;
  const int4* parts;            // {first chunk, chunks, first group of segment sums or -1, segments | segment length << 8}
  double* seg_sums;             // [groups][32]: from a split tile's first group on, [segments][groups of the tile]
  int32_t* arrived;             // [groups]: at a split tile's first groups, segments finished per consumer warp
  int32_t nitems;
  int32_t* counter;
  // lists and source layout (producer)
  const int32_t* list_ptr;
  const int32_t* list_src;
  int32_t nct;
  const int32_t* t_parent;
  const int32_t* s_leaf_first;
  const int32_t* s_leaf_last;
  const int32_t* pad_prefix;
  const float4* chunk_frame;   // [chunks][2]: frame centre + real count (int bits), extents + tau
  const float* pool_res;       // FP32: frame residuals of the pool's particles (pair records)
  const float4* item_box;      // FP32: [items][kItemGroups][2] target group boxes (lo, hi)
  DegreeSet deg;               // degrees, proxies per cluster and pool offsets per degree
  const void* pool;
  // targets and outputs (consumers)
  const double* tx;
  const double* ty;
  const double* tz;
  const double* t_nodes[kMaxDegrees];   // target proxy nodes per degree index
  double* phi_near;
  double* phit[kMaxDegrees];            // target proxy potentials per degree index
  int* err;
  // per-problem kernel parameters (read once per work item)
  const int32_t* t_problem;    // target cluster -> problem
  const float* prob_prm;       // FP32 kernel parameter (fp32_parameter)
  const double* prob_kappa;
  const int* prob_kernel;      // kernel of each problem (read per item by the fused launch)
  bool overlap;                // a target may lie at a source proxy (clusters_may_overlap)
};

// Flags of a staged chunk: first of its task, last of its segment, last of its task.
constexpr unsigned kTaskStart = 1, kSegEnd = 2, kTaskEnd = 4;

struct StageMeta {
  int item;                     // task index (-1: no more work)
  int count;                    // real sources in the staged chunk
  int slot;                     // split item: first group of its segment sums (-1: the task is a whole item)
  int seg;                      // the chunk's segment
  unsigned flags;               // kTaskStart | kSegEnd | kTaskEnd
  unsigned near;                // bit g: target group g may be near the chunk (residuals staged)
  float c[3];                   // frame centre
  float4 ext;                   // half-extents and near distance tau (-inf: proxies)
};

// ---- PTX helpers: mbarrier, bulk copy, timer -------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after kWaitNs, raising the plan's error flag.  The
// clock is read every 256th attempt only, and the producer sleeps between
// attempts: a waiting warp shares the issue slots with the warps that compute.
__device__ __noinline__ bool mbar_wait_slow(uint64_t* b, uint32_t parity, int* err, uint32_t sleep_ns) {
  const uint64_t t0 = global_ns();
  for (uint32_t n = 1;; ++n) {
    if (sleep_ns) __nanosleep(sleep_ns);
    if (mbar_try_wait(b, parity)) return true;
    if ((n & 255u) == 0 && global_ns() - t0 > kWaitNs) {
      atomicExch(err, kDevErrTimeout);
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int* err, uint32_t sleep_ns = 0) {
  return mbar_try_wait(b, parity) || mbar_wait_slow(b, parity, err, sleep_ns);
}
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes,
                                              uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float exp2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ bool not_finite(float v) {
  return (__float_as_uint(v) & 0x7f800000u) == 0x7f800000u;
}

// ---- packed FP32 (f32x2) helpers: low half = first element -----------------
typedef unsigned long long f2_t;
__device__ __forceinline__ f2_t f2_add(f2_t a, f2_t b) {
  f2_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
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
__device__ __forceinline__ f2_t f2_pack(float lo, float hi) {
  f2_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void f2_unpack(f2_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// ---- kernel functions (Sec. 4.6); d = x - y -------------------------------
template <typename T>
__device__ __forceinline__ T poly_kernel(T dx, T dy, T dz) {
  return (T)1 + dx - (T)2 * dy + (T)3 * dz + dx * dy - dy * dz + dx * dx * dz * dz -
         (T)0.5 * dy * dy;
}

// Kernels whose near chunks all take the guarded call: finite at r = 0, so that
// a coincident pair would not show in the sum (and their loop is long: a second
// copy of it beside the plain one spills registers).
template <int KERN>
struct AlwaysGuarded {
  static constexpr bool value = KERN == BLDTT_OSCILLATORY || KERN == BLDTT_REG_COULOMB ||
                                KERN == BLDTT_TEST_POLY;
};

// Kernel parameter of a work item in FP64: kappa, and for Yukawa its form in
// fixed point.
struct Param64 {
  double kappa;
  fixed64::Screen screen;
};
// Coulomb, Yukawa and regularized run in fixed point: the FP64 pipe (1.7 lanes
// per clock and SM) would take 12 to 45 instructions per evaluation, here 4.  2E4
// Coulomb particles (n 4, theta 0.7, leaves of 500) 2.3 ms in this kernel, a third
// of its time with FP64 expressions; 6E4 Yukawa (n 7, theta 0.8, leaves of 1000) 9.5
// ms, a fifth.
template <int KERN>
__device__ __forceinline__ double kernel_f64(double dx, double dy, double dz, const Param64& prm) {
  if (KERN == BLDTT_COULOMB) return fixed64::inv_r(dx, dy, dz);
  if (KERN == BLDTT_YUKAWA) return fixed64::screened_inv_r(dx, dy, dz, prm.screen);
  if (KERN == BLDTT_REG_COULOMB) return fixed64::inv_sqrt_r2_kappa2(dx, dy, dz, prm.kappa);
  const double r2 = dx * dx + dy * dy + dz * dz;
  if (!(r2 > 0.0)) return 0.0;
  if (KERN == BLDTT_TEST_POLY) return poly_kernel<double>(dx, dy, dz);
  const double ri = rsqrt(r2);
  return ri * sin(prm.kappa * (r2 * ri));
}

// ---- producer: walks a task's lists -----------------------------------------
// One warp.  The lanes read the lists 32 entries at a time (source cluster,
// pool range), so a task that starts in the middle of its item's chunks skips
// to it in a few memory latencies, and a chunk's near-group test runs on one
// lane per group; lane 0 issues the copies.
template <typename Vec, int RES, int STAGES>
struct Producer {
  const InteractView& v;
  Vec (*buf)[kChunk];
  float4 (*rbuf)[RES];
  StageMeta* meta;
  uint64_t* full;
  uint64_t* empty;
  const int lane;
  uint32_t it = 0;
  int cur_item = -1;
  int slot = -1, seg_len = 1;
  int seg = 0, seg_left = 1;    // the next chunk's segment, chunks left in it
  int skip = 0, left = 0;       // chunks before the task's first, chunks still to stage
  unsigned start = 0;           // kTaskStart until the task's first chunk is staged
  bool has_box = false;
  float4 glo, ghi;              // lane g: box of the task's target group g

  __device__ Producer(const InteractView& v_, Vec (*b)[kChunk], float4 (*r)[RES], StageMeta* m,
                      uint64_t* f, uint64_t* e, int lane_)
      : v(v_), buf(b), rbuf(r), meta(m), full(f), empty(e), lane(lane_) {}

  // Target groups of the current task whose box comes within tau of the
  // particle chunk's box (c +- e): a superset of the targets the consumers'
  // own test finds near.
  __device__ __forceinline__ unsigned near_groups(const float4& f, const float4& ext) const {
    if (!(ext.w >= 0.f)) return 0u;       // proxy chunk
    const float gap = fmaxf(fmaxf(fmaxf(glo.x - (f.x + ext.x), (f.x - ext.x) - ghi.x),
                                  fmaxf(glo.y - (f.y + ext.y), (f.y - ext.y) - ghi.y)),
                            fmaxf(glo.z - (f.z + ext.z), (f.z - ext.z) - ghi.z));
    return __ballot_sync(0xffffffffu, has_box && gap < ext.w);
  }

  __device__ __forceinline__ bool acquire(int& s) {
    s = (int)(it % STAGES);
    return __all_sync(0xffffffffu, mbar_wait(&empty[s], ((it / STAGES) & 1u) ^ 1u, v.err, 500u));
  }

  // Stage pool chunk q (real entries only).
  __device__ __forceinline__ bool stage(int q) {
    const float4 f = v.chunk_frame[(int64_t)kChunkInfo * q];
    float4 ext = make_float4(0.f, 0.f, 0.f, 0.f);
    unsigned near = 0;
    if (std::is_same<Vec, float4>::value) {
      ext = v.chunk_frame[(int64_t)kChunkInfo * q + 1];
      near = near_groups(f, ext);
    }
    int s;
    if (!acquire(s)) return false;
    if (lane == 0) {
      const int count = __float_as_int(f.w);
      StageMeta& m = meta[s];
      m.item = cur_item;
      m.count = count;
      m.slot = slot;
      m.seg = seg;
      m.flags = start | (seg_left == 1 || left == 1 ? kSegEnd : 0u) | (left == 1 ? kTaskEnd : 0u);
      m.near = near;
      uint32_t bytes;
      if (std::is_same<Vec, float4>::value) {
        m.c[0] = f.x;
        m.c[1] = f.y;
        m.c[2] = f.z;
        m.ext = ext;
        bytes = (uint32_t)(((count + 1) / 2) * 32);          // whole pair records
      } else {
        bytes = (uint32_t)(count * sizeof(Vec));
      }
      const char* src = reinterpret_cast<const char*>(v.pool) + (int64_t)q * (kChunk * (int64_t)sizeof(Vec));
      mbar_arrive_tx(&full[s], near ? 2 * bytes : bytes);
      bulk_copy_g2s(buf[s], src, bytes, &full[s]);
      if (RES == kChunk && near)       // the chunk's frame residuals, same record layout
        bulk_copy_g2s(rbuf[s], v.pool_res + (int64_t)q * (kChunk * 4), bytes, &full[s]);
    }
    __syncwarp();
    ++it;
    --left;
    if (--seg_left == 0) {
      seg_left = seg_len;
      ++seg;
    }
    start = 0;
    return true;
  }

  // Entries [e0, e1) of one list: the particles of the source clusters (i < 0;
  // all leaves under a cluster are one contiguous pool range, because they are
  // consecutive in leaf order) or their proxy blocks of degree index i.
  __device__ bool entries(int32_t e0, int32_t e1, int i) {
    for (int32_t base = e0; base < e1 && left > 0; base += 32) {
      int o = 0, n = 0;
      if (base + lane < e1) {
        const int32_t src = v.list_src[base + lane];
        if (i < 0) {
          const int32_t p0 = v.pad_prefix[v.s_leaf_first[src]], p1 = v.pad_prefix[v.s_leaf_last[src]];
          o = p0 / kChunk;
          n = (p1 - p0) / kChunk;
        } else {
          n = v.deg.np_pad[i] / kChunk;
          o = (int)(v.deg.proxy_base[i] / kChunk) + src * n;
        }
      }
      const int cnt = min(32, e1 - base);
      for (int j = 0; j < cnt && left > 0; ++j) {
        const int oj = __shfl_sync(0xffffffffu, o, j), nj = __shfl_sync(0xffffffffu, n, j);
        if (skip >= nj) {
          skip -= nj;
          continue;
        }
        for (int k = skip; k < nj && left > 0; ++k)
          if (!stage(oj + k)) return false;
        skip = 0;
      }
    }
    return true;
  }

  // The lists of a leaf's particles: on the leaf and on each of its ancestors, PP
  // and then PC of every degree.  Lane 0 holds an ancestor's PP range of the CSR,
  // lane i + 1 its PC range of degree index i.
  __device__ bool run_particles(int32_t leaf) {
    for (int32_t a = leaf; a >= 0 && left > 0;) {
      const int32_t up = v.t_parent[a];
      int32_t e0 = 0, e1 = 0;
      if (lane <= v.deg.n) {
        const int64_t k = (int64_t)(lane == 0 ? 0 : class_of(BLDTT_PC, lane - 1)) * v.nct + a;
        e0 = v.list_ptr[k];
        e1 = v.list_ptr[k + 1];
      }
      unsigned todo = __ballot_sync(0xffffffffu, e1 > e0);
      while (todo) {
        const int j = __ffs(todo) - 1;
        todo &= todo - 1;
        if (!entries(__shfl_sync(0xffffffffu, e0, j), __shfl_sync(0xffffffffu, e1, j), j - 1)) return false;
      }
      a = up;
    }
    return true;
  }

  __device__ void run() {
    bool ok = true;
    while (ok) {
      int idx = 0;
      if (lane == 0) idx = atomicAdd(v.counter, 1);
      idx = __shfl_sync(0xffffffffu, idx, 0);
      if (idx >= v.nitems) break;
      const int4 item = v.items[idx], part = v.parts[idx];
      cur_item = idx;
      skip = part.x;
      left = part.y;
      slot = part.z;
      seg_len = seg_left = part.w >> 8;           // a task starts at a segment's start
      seg = part.x / seg_len;
      start = kTaskStart;
      has_box = std::is_same<Vec, float4>::value && lane < (item.z + 31) / 32;
      if (has_box) {
        const float4* gb = v.item_box + (int64_t)idx * (2 * kItemGroups);
        glo = gb[2 * lane];
        ghi = gb[2 * lane + 1];
      }
      if (item.w == kItemParticles) {
        ok = run_particles(item.x);
      } else {                          // CP and CC of one degree on the cluster itself
        const int i = item.w - kItemProxies;
        const int64_t k0 = (int64_t)class_of(BLDTT_CP, i) * v.nct + item.x;
        const int64_t k1 = (int64_t)class_of(BLDTT_CC, i) * v.nct + item.x;
        const int32_t a0 = v.list_ptr[k0], a1 = v.list_ptr[k0 + 1], b0 = v.list_ptr[k1], b1 = v.list_ptr[k1 + 1];
        ok = entries(a0, a1, -1) && entries(b0, b1, i);
      }
    }
    if (ok) {
      int s;
      if (acquire(s)) {
        if (lane == 0) {
          meta[s].item = -1;
          mbar_arrive(&full[s]);
        }
        return;
      }
    }
    // Error path: let the copies already issued land before the CTA exits.
    uint32_t first = it > (uint32_t)STAGES ? it - STAGES : 0;
    for (uint32_t j = first; j < it; ++j) mbar_wait(&full[j % STAGES], (j / STAGES) & 1u, v.err);
  }
};

// ---- consumers --------------------------------------------------------------
// Kernel parameter of a work item in FP32: fp32_parameter's value k, and for the
// oscillatory kernel kappa / pi and pi k / (kappa kPiHigh) - 1 (see sin2); the
// second form has each value duplicated.
template <typename T>
struct PlainParam {
  T k;
};
template <typename T>
struct PhaseParam {
  T k, turns, rest;
};
template <int KERN, typename T>
using Param = std::conditional_t<KERN == BLDTT_OSCILLATORY, PhaseParam<T>, PlainParam<T>>;
__device__ __forceinline__ PlainParam<f2_t> duplicate(const PlainParam<float>& p) { return {f2_pack(p.k, p.k)}; }
__device__ __forceinline__ PhaseParam<f2_t> duplicate(const PhaseParam<float>& p) {
  return {f2_pack(p.k, p.k), f2_pack(p.turns, p.turns), f2_pack(p.rest, p.rest)};
}
constexpr float kPiHigh = 3.140625f;
__device__ __forceinline__ void set_param(PlainParam<float>& p, float k, const double*) { p.k = k; }
__device__ __forceinline__ void set_param(PhaseParam<float>& p, float k, const double* kappa) {
  const double pi = 3.14159265358979323846;
  const double scale = *kappa > 0.0 ? (double)k / *kappa : 1.0;
  p = {k, (float)(*kappa / pi), (float)(pi / (double)kPiHigh * scale - 1.0)};
}

// sin(kappa r) of two values: kappa r = n pi + f with n the nearest integer, sin =
// (-1)^n sin f.  n comes from adding 1.5 * 2^23 (its parity is the sum's last
// bit; rint and the conversion to int run on the MUFU's pipe, which the rsqrts
// fill).  With k the float nearest to kappa, f k / kappa = k r - n (pi k / kappa), and
// pi k / kappa is kPiHigh (1 + rest): n kPiHigh comes from one multiply-add, exact
// to n = 2^15.  So neither the product k r nor kappa's rounding counts n times;
// what is left of the latter scales f by less than 2^-24, as a product rounded to
// float would.
// Where n = 0 and kappa is a float nothing is rounded at all.
// sin f = f + f^3 Q(f^2), Q the degree-3 minimax polynomial of the relative error on
// |f| <= pi/2 (6.3e-9 with these float coefficients, found one after the other so
// that each absorbs the rounding of those before it).  For arguments
// beyond 2^22 pi the phase is noise in float; the clamp keeps |sin| <= 1.
__device__ __forceinline__ f2_t sin2(f2_t r, const PhaseParam<f2_t>& p) {
  const f2_t big = f2_pack(12582912.f, 12582912.f);
  const f2_t t = f2_fma(r, p.turns, big);
  const f2_t m = f2_fma(t, f2_pack(-kPiHigh, -kPiHigh), f2_pack(12582912.f * kPiHigh, 12582912.f * kPiHigh));   // -n kPiHigh
  float f0, f1, t0, t1, p0, p1;
  f2_unpack(f2_fma(m, p.rest, f2_fma(r, p.k, m)), f0, f1);
  f2_unpack(t, t0, t1);
  const f2_t f = f2_pack(fminf(fmaxf(f0, -1.5707964f), 1.5707964f), fminf(fmaxf(f1, -1.5707964f), 1.5707964f));
  const f2_t s = f2_mul(f, f);
  f2_t q = f2_fma(s, f2_pack(2.6060538402816746e-6f, 2.6060538402816746e-6f),
                  f2_pack(-1.9809768127743155e-4f, -1.9809768127743155e-4f));
  q = f2_fma(q, s, f2_pack(0.008333069272339344f, 0.008333069272339344f));
  q = f2_fma(q, s, f2_pack(-0.16666659712791443f, -0.16666659712791443f));
  f2_unpack(f2_fma(f2_mul(f, s), q, f), p0, p1);
  return f2_pack(__uint_as_float(__float_as_uint(p0) ^ (__float_as_uint(t0) << 31)),
                 __uint_as_float(__float_as_uint(p1) ^ (__float_as_uint(t1) << 31)));
}

// Packed evaluation of target k against the source pair (s0, s1) at
// differences d: acc += (q0 G(x - s0), q1 G(x - s1)).  A guard gives a pair at r =
// 0 the factor 0 (two compares and two selects a pair of evaluations); kGuardPair
// leaves its charge out as well, which may be infinite in float.  Evaluations
// per clock and SM: Coulomb 12.8, Yukawa 8.7, regularized 11.1 (9.4 with the guard
// on every pair instead of near chunks only, 2.6 in a scalar guarded loop),
// oscillatory 4.2 (0.67 in a scalar loop with sinf).
enum Guard { kNoGuard, kGuardFactor, kGuardPair };
template <int KERN, Guard GUARD = kNoGuard>
__device__ __forceinline__ f2_t pair2_eval(f2_t dx, f2_t dy, f2_t dz, f2_t q2, f2_t acc, const Param<KERN, f2_t>& prm) {
  f2_t r2 = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
  float r0, r1;
  f2_unpack(r2, r0, r1);
  const bool k0 = GUARD == kNoGuard || r0 > 0.f, k1 = GUARD == kNoGuard || r1 > 0.f;
  if (GUARD == kGuardPair) {
    float q0, q1;
    f2_unpack(q2, q0, q1);
    q2 = f2_pack(k0 ? q0 : 0.f, k1 ? q1 : 0.f);
  }
  if (KERN == BLDTT_REG_COULOMB) f2_unpack(f2_add(r2, prm.k), r0, r1);
  const float i0 = rsqrt_approx(r0), i1 = rsqrt_approx(r1);
  const f2_t ri = f2_pack(k0 ? i0 : 0.f, k1 ? i1 : 0.f);
  if (KERN == BLDTT_COULOMB || KERN == BLDTT_REG_COULOMB) return f2_fma(q2, ri, acc);
  const f2_t r = f2_mul(r2, ri);
  if constexpr (KERN == BLDTT_OSCILLATORY) return f2_fma(f2_mul(q2, ri), sin2(r, prm), acc);
  // Yukawa: q ri exp2(-kappa log2(e) r)
  float e0, e1;
  f2_unpack(f2_mul(r, prm.k), e0, e1);
  return f2_fma(f2_mul(q2, ri), f2_pack(exp2_approx(e0), exp2_approx(e1)), acc);
}
template <int KERN>
__device__ __forceinline__ f2_t pair2_f32(f2_t tx, f2_t ty, f2_t tz, const ulonglong2& a,
                                          const ulonglong2& b, f2_t acc, const Param<KERN, f2_t>& prm) {
  return pair2_eval<KERN>(f2_sub(tx, a.x), f2_sub(ty, a.y), f2_sub(tz, b.x), b.y, acc, prm);
}
// Careful variant: d = fma(m, x_r - y_r, x'' - y'') with m = 1 for a target
// near the chunk (frame residuals added) and m = 0 otherwise (exactly the
// packed difference x'' - y'').
template <int KERN, Guard GUARD>
__device__ __forceinline__ f2_t pair2_careful(f2_t tx, f2_t ty, f2_t tz, f2_t rx, f2_t ry, f2_t rz,
                                              f2_t m2, const ulonglong2& a, const ulonglong2& b,
                                              const ulonglong2& ra, const ulonglong2& rb, f2_t acc,
                                              const Param<KERN, f2_t>& prm) {
  return pair2_eval<KERN, GUARD>(f2_fma(m2, f2_sub(rx, ra.x), f2_sub(tx, a.x)),
                          f2_fma(m2, f2_sub(ry, ra.y), f2_sub(ty, a.y)),
                          f2_fma(m2, f2_sub(rz, rb.x), f2_sub(tz, b.x)), b.y, acc, prm);
}

// Sum over the staged chunk of q G for K targets; two partial sums per target.
// Full chunks have a loop of fixed length (the oscillatory kernel's loop body
// is long enough to do without); the others are unrolled as far: 1E6 particles,
// whose leaves end in a partial chunk, 31.5 ms unrolled by 2, 31.1 by 4 and 8.
template <int KERN, int K>
__device__ __forceinline__ void chunk_f32(const ulonglong2* __restrict__ sb, int npairs,
                                          const f2_t (&x2)[K][3], float (&a)[K], const Param<KERN, float>& prm) {
  f2_t acc[K];
  const Param<KERN, f2_t> prm2 = duplicate(prm);
#pragma unroll
  for (int k = 0; k < K; ++k) acc[k] = 0ull;
  if (KERN != BLDTT_OSCILLATORY && npairs == kChunk / 2) {
#pragma unroll 8
    for (int jp = 0; jp < kChunk / 2; ++jp) {
      const ulonglong2 A = sb[2 * jp], Bq = sb[2 * jp + 1];
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] = pair2_f32<KERN>(x2[k][0], x2[k][1], x2[k][2], A, Bq, acc[k], prm2);
    }
  } else {
#pragma unroll 8
    for (int jp = 0; jp < npairs; ++jp) {
      const ulonglong2 A = sb[2 * jp], Bq = sb[2 * jp + 1];
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] = pair2_f32<KERN>(x2[k][0], x2[k][1], x2[k][2], A, Bq, acc[k], prm2);
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    float lo, hi;
    f2_unpack(acc[k], lo, hi);
    a[k] = lo + hi;
  }
}

// A consumer thread's targets, split v = hi + lo in FP32 and kept in shared
// memory rather than registers, (hi, lo) in one word: entry (k, d) of the
// thread is v[(3k + d) * stride].  (Kept duplicated for the packed subtraction
// they took 12 KB of a CTA's shared memory; with the items' totals beside them
// only five of the six CTAs then fit an SM: 32.4 -> 32.9 ms at 1E6.)
struct TargetSplit {
  const f2_t* v;
  int stride;
  __device__ __forceinline__ void get(int k, int d, float& hi, float& lo) const {
    f2_unpack(v[(3 * k + d) * stride], hi, lo);
  }
};

// Frame residual (frame_resid) of target slot k in the chunk's frame c.
__device__ __forceinline__ void target_residual(const TargetSplit& ts, const float* c, int k, float (&xr)[3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    float h, l;
    ts.get(k, d, h, l);
    xr[d] = frame_resid(h, l, c[d]);
  }
}

// Careful packed sum over the staged chunk (sr: its frame residual records).
template <int KERN, int K, Guard GUARD>
__device__ __forceinline__ void chunk_f32_careful(const ulonglong2* __restrict__ sb,
                                                  const ulonglong2* __restrict__ sr, int npairs,
                                                  const f2_t (&x2)[K][3], const TargetSplit& ts,
                                                  const float* c, unsigned near, float (&a)[K],
                                                  const Param<KERN, float>& prm) {
  const Param<KERN, f2_t> prm2 = duplicate(prm);
  f2_t acc[K], m2[K], r2x[K][3];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const float m = ((near >> k) & 1u) ? 1.f : 0.f;
    m2[k] = f2_pack(m, m);
    float xr[3];
    target_residual(ts, c, k, xr);
#pragma unroll
    for (int d = 0; d < 3; ++d) r2x[k][d] = f2_pack(xr[d], xr[d]);
    acc[k] = 0ull;
  }
#pragma unroll 2
  for (int jp = 0; jp < npairs; ++jp) {
    const ulonglong2 A = sb[2 * jp], Bq = sb[2 * jp + 1], RA = sr[2 * jp], RB = sr[2 * jp + 1];
#pragma unroll
    for (int k = 0; k < K; ++k)
      acc[k] = pair2_careful<KERN, GUARD>(x2[k][0], x2[k][1], x2[k][2], r2x[k][0], r2x[k][1], r2x[k][2],
                                   m2[k], A, Bq, RA, RB, acc[k], prm2);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    float lo, hi;
    f2_unpack(acc[k], lo, hi);
    a[k] = lo + hi;
  }
}

// Scalar evaluation of a staged chunk by the test kernel, with the r = 0 guard:
// two partial sums (even and odd entries).  Targets whose bit is set in `near`
// use the corrected difference of the careful path.
template <int K>
__device__ __forceinline__ void chunk_f32_slow(const float* __restrict__ sf, const float* __restrict__ res,
                                               int count, const float (&xs)[K][3],
                                               const TargetSplit& ts, const float* c, unsigned near,
                                               float (&a)[K]) {
  // one target slot at a time: few live registers on this rare path
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const bool nr = (near >> k) & 1u;
    float xr[3] = {0.f, 0.f, 0.f};
    if (nr) target_residual(ts, c, k, xr);
    float acc0 = 0.f, acc1 = 0.f;
    for (int jp = 0; jp < (count + 1) / 2; ++jp) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = 2 * jp + h;
        if (j < count) {
          const float* r = sf + jp * 8 + h;   // pair record: x0 x1 y0 y1 z0 z1 q0 q1
          float dx = __fsub_rn(xs[k][0], r[0]), dy = __fsub_rn(xs[k][1], r[2]),
                dz = __fsub_rn(xs[k][2], r[4]);
          if (nr) {
            const float* e = res + jp * 8 + h;
            dx = __fadd_rn(dx, __fsub_rn(xr[0], e[0]));
            dy = __fadd_rn(dy, __fsub_rn(xr[1], e[2]));
            dz = __fadd_rn(dz, __fsub_rn(xr[2], e[4]));
          }
          const float r2 = fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
          if (r2 > 0.f) {
            const float t = r[6] * poly_kernel<float>(dx, dy, dz);
            if (h == 0)
              acc0 = __fadd_rn(acc0, t);
            else
              acc1 = __fadd_rn(acc1, t);
          }
        }
      }
    }
    a[k] = acc0 + acc1;
  }
}

// One staged chunk in FP64 for K targets.
template <int KERN, int K>
__device__ __forceinline__ void chunk_f64(const double4* __restrict__ sb, int count,
                                          const double (&x)[K][3], double (&a)[K], const Param64& prm) {
#pragma unroll
  for (int k = 0; k < K; ++k) a[k] = 0.0;
#pragma unroll 2
  for (int j = 0; j < count; ++j) {
    const double4 p = sb[j];
#pragma unroll
    for (int k = 0; k < K; ++k)
      a[k] = fma(p.w, kernel_f64<KERN>(x[k][0] - p.x, x[k][1] - p.y, x[k][2] - p.z, prm), a[k]);
  }
}

// The same for the warp's real rows: its last target slot is left out where
// none of its rows holds a target.  The FP64 pipe bounds this path, so an idle
// row costs what a real one does: 2E4 Coulomb particles in leaves of 312 (a
// full tile and one of 56 rows) 2.3 ms, 3.2 with the idle rows.
template <int KERN, int K>
__device__ __forceinline__ void rows_f64(const double4* __restrict__ sb, int count, const double (&x)[K][3],
                                         bool warp_full, double (&a)[K], const Param64& prm) {
  if (K == 1 || warp_full) {
    chunk_f64<KERN, K>(sb, count, x, a, prm);
    return;
  }
  constexpr int K1 = K > 1 ? K - 1 : 1;
  double a1[K1];
  chunk_f64<KERN, K1>(sb, count, *reinterpret_cast<const double(*)[K1][3]>(&x), a1, prm);
#pragma unroll
  for (int k = 0; k < K; ++k) a[k] = k < K1 ? a1[k < K1 ? k : 0] : 0.0;
}

// Absolute coordinates of target row r of an item (a particle or a proxy point).
__device__ __forceinline__ void target_coords(const InteractView& v, const int4& item, int r,
                                              double& X, double& Y, double& Z) {
  if (r >= item.z) {       // idle slot of a partial tile: far away, contributes nothing
    X = Y = Z = 1.0e15;
    return;
  }
  if (item.w == kItemParticles) {
    int64_t i = (int64_t)item.y + r;
    X = v.tx[i];
    Y = v.ty[i];
    Z = v.tz[i];
  } else {
    const int i = item.w - kItemProxies;
    const int P = v.deg.d[i] + 1;
    int l = item.y + r;
    int l1 = l / (P * P), l2 = (l / P) % P, l3 = l % P;
    const double* nd = v.t_nodes[i] + (int64_t)item.x * 3 * P;
    X = nd[l1];
    Y = nd[P + l2];
    Z = nd[2 * P + l3];
  }
}

__device__ __forceinline__ void store_output(const InteractView& v, const int4& item, int r,
                                             double value) {
  if (r < item.z) {
    if (item.w == kItemParticles)
      v.phi_near[(int64_t)item.y + r] = value;
    else
      v.phit[item.w - kItemProxies][(int64_t)item.x * v.deg.np[item.w - kItemProxies] + item.y + r] = value;
  }
}

template <int K>
struct SegSums {
  double v[K];
};
// End of a split item's segment or of an item, per consumer warp (out of line:
// no register of the packed loop).  A whole item adds the last segment's sums
// to its totals (tot, in shared memory) and stores them.  A split item's sums go to memory; the
// warp that finds every segment of the item finished adds them in segment
// order, the order in which a whole item adds them (so the split does not
// change the bits), and resets the count for the next compute.
template <int NCW, int K>
__device__ __noinline__ void end_segment(const InteractView& v, const int4 item, int task, int slot, int seg,
                                         unsigned flags, const SegSums<K> a, double* tot) {
  const int ct = threadIdx.x, lane = ct & 31;
  if (slot < 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int r = k * NCW * 32 + ct;
      store_output(v, item, r, tot[r] + a.v[k]);
    }
    return;
  }
  const int rows = (item.z + 31) / 32 * 32;
  if (ct >= rows) return;                       // whole warps: no row of this tile
  double* sums = v.seg_sums + (int64_t)slot * 32;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (k * NCW * 32 + ct < rows) sums[seg * rows + k * NCW * 32 + ct] = a.v[k];
  if (!(flags & kTaskEnd)) return;
  const int4 part = v.parts[task];
  const int nseg = part.w & 0xff, len = part.w >> 8;
  const int mine = (part.x + part.y + len - 1) / len - part.x / len;
  int32_t* count = v.arrived + slot + (ct >> 5);
  __threadfence();
  __syncwarp();
  int done = 0;
  if (lane == 0) done = atomicAdd(count, mine) + mine;
  if (__shfl_sync(0xffffffffu, done, 0) != nseg) return;
  __threadfence();
  for (int k = 0; k < K; ++k) {
    const int r = k * NCW * 32 + ct;
    if (r >= rows) break;
    double t = 0.0;
    for (int g = 0; g < nseg; ++g) t += __ldcg(sums + g * rows + r);
    store_output(v, item, r, t);
  }
  if (lane == 0) *count = 0;
}

// Out-of-line entries to the rare paths of the packed kernels, so that their
// registers do not burden the packed loop: they rebuild the targets' frame
// coordinates from the shared-memory split (the same rounding as the packed
// path) and return the K partial sums.
template <int K>
struct PartialSums {
  float v[K];
};
template <int K>
__device__ __forceinline__ void frame_targets(const TargetSplit& ts, const float* c, f2_t (&x2)[K][3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      float h, l;
      ts.get(k, d, h, l);
      const float x = frame_main(h, l, c[d]);
      x2[k][d] = f2_pack(x, x);
    }
  }
}
// The careful path's sums with the r = 0 guard, of the charges too if near has
// kWholePair set.  A call of its own: its registers must not crowd the plain loop's.
constexpr unsigned kWholePair = 0x80000000u;
template <int KERN, int K>
__device__ __noinline__ PartialSums<K> careful_sums(const float* sf, const float* res, int count,
                                                    const TargetSplit ts, const float* c, unsigned near,
                                                    const Param<KERN, float> prm) {
  f2_t x2[K][3];
  frame_targets<K>(ts, c, x2);
  const ulonglong2 *sb = reinterpret_cast<const ulonglong2*>(sf), *rb = reinterpret_cast<const ulonglong2*>(res);
  PartialSums<K> out;
  if (near & kWholePair)
    chunk_f32_careful<KERN, K, kGuardPair>(sb, rb, (count + 1) / 2, x2, ts, c, near, out.v, prm);
  else
    chunk_f32_careful<KERN, K, kGuardFactor>(sb, rb, (count + 1) / 2, x2, ts, c, near, out.v, prm);
  return out;
}
// One staged chunk in FP32 for K targets (partial sums in a[]).  ts holds
// the targets' FP32 splits and c the chunk's frame centre, x2 the targets' frame coordinates, ext the chunk's half-extents and
// near distance tau, res its staged frame residuals, and bit k of `slot` says
// that the producer found target slot k's group near the chunk.  A target
// with max_d (|x''_d| - e_d) < tau is near: the warp then takes the careful
// packed path, which adds the frame residuals for near targets only, and with
// the r = 0 guard if a target lies inside the chunk's box (or within a
// thousandth of tau of it).  Otherwise the plain packed path runs.  A sum that
// is not finite is redone with coincident pairs left out, charge and all.  The
// regularized kernel is finite at r = 0: where a target may lie at a source proxy
// (overlap), its proxy chunks take the guarded call too.
// The guard costs what its selects do: on all near chunks 512 problems of 16k
// (lists of about 30 chunks) take 75.5 ms in this kernel instead of 74.0, the
// unequal sets 83.2 instead of 82.6; and a tile's own chunk evaluated unguarded
// first and guarded after 77.7.
template <int KERN, int K>
__device__ __forceinline__ void eval_chunk_f32(const void* buf, const float4* rbuf, int count,
                                               const f2_t (&x2)[K][3], const TargetSplit& ts,
                                               const float* c, const float4* ext_p, unsigned slot, bool warp_full,
                                               bool overlap, const Param<KERN, float>& prm, float (&a)[K]) {
  const float* sf = reinterpret_cast<const float*>(buf);
  const float* res = reinterpret_cast<const float*>(rbuf);
  float xs[K][3];
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float hi;
      f2_unpack(x2[k][d], xs[k][d], hi);
    }
  unsigned near = 0;
  bool any_near = false, inside = false;
  if (slot) {                                   // warp-uniform
    const float4 ext = *ext_p;
    bool within = AlwaysGuarded<KERN>::value;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float m = fmaxf(fmaxf(fabsf(xs[k][0]) - ext.x, fabsf(xs[k][1]) - ext.y),
                            fabsf(xs[k][2]) - ext.z);
      if (((slot >> k) & 1u) && m < ext.w) near |= 1u << k;
      within = within || m < 0.001f * ext.w;
    }
    any_near = __any_sync(0xffffffffu, near != 0);
    inside = __any_sync(0xffffffffu, within);
  }
  if (KERN == BLDTT_TEST_POLY) {
    chunk_f32_slow<K>(sf, res, count, xs, ts, c, near, a);
    return;
  }
  const ulonglong2* sb = reinterpret_cast<const ulonglong2*>(buf);
  if (any_near && !inside) {
    chunk_f32_careful<KERN, K, kNoGuard>(sb, reinterpret_cast<const ulonglong2*>(rbuf), (count + 1) / 2, x2,
                                      ts, c, near, a, prm);
  } else if (any_near) {
    const PartialSums<K> r = careful_sums<KERN, K>(sf, res, count, ts, c, near, prm);
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = r.v[k];
  } else if (KERN == BLDTT_REG_COULOMB && overlap && !(ext_p->w >= 0.f)) {
    const PartialSums<K> r = careful_sums<KERN, K>(sf, sf, count, ts, c, 0u, prm);
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = r.v[k];
  } else if (K > 1 && !warp_full) {
    // the warp's last target row lies beyond a partial tile: evaluate the others only
    constexpr int K1 = K > 1 ? K - 1 : 1;
    float a1[K1];
    const f2_t(&x2s)[K1][3] = *reinterpret_cast<const f2_t(*)[K1][3]>(&x2);
    chunk_f32<KERN, K1>(sb, (count + 1) / 2, x2s, a1, prm);
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = k < K1 ? a1[k < K1 ? k : 0] : 0.f;
  } else {
    chunk_f32<KERN, K>(sb, (count + 1) / 2, x2, a, prm);
  }
  bool bad = false;
#pragma unroll
  for (int k = 0; k < K; ++k) bad = bad || not_finite(a[k]);
  if (__any_sync(0xffffffffu, bad)) {
    // residuals that were not staged are not read: any finite numbers do (their factor is 0)
    const PartialSums<K> r = careful_sums<KERN, K>(sf, slot ? res : sf, count, ts, c, near | kWholePair, prm);
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = r.v[k];
  }
}

// The parameter block is taken by value: device functions that read it by
// reference make each thread keep a private copy on its stack (0.5 KB; 70 MB
// of local writes per launch at 1E6, cached in L1).  Passing it as a
// __grid_constant__ parameter instead removes those writes but ran slower,
// 32.30 against 32.09 ms at 1E6 and 154-179 against 90 ms on the unequal-set
// Yukawa workload (1E7 targets, 5E6 Plummer sources), also when only the
// producer kept a private copy.  A pointer to per-segment blocks in device
// memory ran slower too: 32.3 against 32.1 ms and 143 against 90 ms.
template <bool F32, int KERN, int NCW, int K, int MINB, int STAGES, bool SKIP>
__global__ void __launch_bounds__((NCW + 1) * 32, MINB) k_interact(InteractView v) {
  static_assert(NCW * 32 * K == kTile, "a CTA covers exactly one work-item tile");
  constexpr int kConsumers = NCW * 32;
  using Vec = typename std::conditional<F32, float4, double4>::type;
  __shared__ __align__(128) Vec sbuf[STAGES][kChunk];
  constexpr int kRes = F32 ? kChunk : 1;     // frame residual records (FP32 only)
  __shared__ __align__(128) float4 sres[STAGES][kRes];
  __shared__ __align__(16) StageMeta smeta[STAGES];
  __shared__ __align__(8) uint64_t full[STAGES];
  __shared__ __align__(8) uint64_t empty[STAGES];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], NCW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp == NCW) {
    Producer<Vec, kRes, STAGES> prod(v, sbuf, sres, smeta, full, empty, lane);
    prod.run();
    return;
  }

  const int ct = threadIdx.x;   // consumer thread 0..kConsumers-1
  int4 item = make_int4(0, 0, 0, 0);
  double X[K][3];               // FP64 targets (FP64 path)
  // FP32 split of this thread's targets (FP32 path), in shared memory
  constexpr int kSplit = F32 ? K * 3 * kConsumers : 1;
  __shared__ __align__(16) f2_t s_hl[kSplit];
  const TargetSplit ts{s_hl + ct, kConsumers};
  double acc[K];                // the current segment's sums
  __shared__ double s_tot[K * kConsumers];   // the item's finished segments (in shared memory: no register)
  bool warp_full = true;
  bool warp_active = true;
  Param<KERN, float> prm{};     // its FP32 parameter
  Param64 prm64{};              // its FP64 parameter
  bool yukawa = KERN == BLDTT_YUKAWA;   // the fused Coulomb/Yukawa launch: this item's kernel
  for (uint32_t it = 0;; ++it) {
    const int s = (int)(it % STAGES);
    if (!mbar_wait(&full[s], (it / STAGES) & 1u, v.err)) return;
    if (smeta[s].item < 0) return;
    if (smeta[s].flags & kTaskStart) {
      item = v.items[smeta[s].item];
      const int pid = v.t_problem[item.x];
      if (F32) set_param(prm, v.prob_prm[pid], v.prob_kappa + pid);
      if (!F32) {
        prm64.kappa = v.prob_kappa[pid];
        if (KERN == BLDTT_YUKAWA || KERN == kKernCoulombYukawa) prm64.screen = fixed64::make_screen(prm64.kappa);
      }
      if (KERN == kKernCoulombYukawa) yukawa = v.prob_kernel[pid] == BLDTT_YUKAWA;
      // does any row of this warp's last target slot hold a real target?
      warp_full = (K - 1) * kConsumers + (warp * 32) < item.z;
      // does any row of its first slot?  (if not, the warp only keeps the ring
      // going; FP64, and layouts for plans with many small items, skip such
      // warps' work)
      if (SKIP || !F32) warp_active = warp * 32 < item.z;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        acc[k] = 0.0;
        s_tot[k * kConsumers + ct] = 0.0;
        target_coords(v, item, k * kConsumers + ct, X[k][0], X[k][1], X[k][2]);
        if (F32) {
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const float h = (float)X[k][d];
            const float l = (float)(X[k][d] - (double)h);
            s_hl[(3 * k + d) * kConsumers + ct] = f2_pack(h, l);
          }
        }
      }
    }
    const int count = smeta[s].count;
    if ((SKIP || !F32) && !warp_active) {
      // no real target in this warp's rows: nothing to evaluate
    } else if constexpr (F32) {
      f2_t x2[K][3];
      const float* c = smeta[s].c;
      frame_targets<K>(ts, c, x2);
      const float4* ext = &smeta[s].ext;
      const unsigned gm = smeta[s].near;
      unsigned slot = 0;
      if (gm) {
#pragma unroll
        for (int k = 0; k < K; ++k) slot |= ((gm >> (k * NCW + warp)) & 1u) << k;
      }
      float a[K];
      if constexpr (KERN != kKernCoulombYukawa)
        eval_chunk_f32<KERN, K>(sbuf[s], sres[s], count, x2, ts, c, ext, slot, warp_full, v.overlap, prm, a);
      else if (yukawa)
        eval_chunk_f32<BLDTT_YUKAWA, K>(sbuf[s], sres[s], count, x2, ts, c, ext, slot, warp_full, v.overlap, prm, a);
      else
        eval_chunk_f32<BLDTT_COULOMB, K>(sbuf[s], sres[s], count, x2, ts, c, ext, slot, warp_full, v.overlap, prm, a);
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] += (double)a[k];
    } else {
      double a[K];
      if (KERN != kKernCoulombYukawa)
        rows_f64<KERN, K>(reinterpret_cast<const double4*>(sbuf[s]), count, X, warp_full, a, prm64);
      else if (yukawa)
        rows_f64<BLDTT_YUKAWA, K>(reinterpret_cast<const double4*>(sbuf[s]), count, X, warp_full, a, prm64);
      else
        rows_f64<BLDTT_COULOMB, K>(reinterpret_cast<const double4*>(sbuf[s]), count, X, warp_full, a, prm64);
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] += a[k];
    }
    // read again (volatile): kept from the top, the flags would hold a register through the packed loop
    const unsigned flags = *static_cast<volatile unsigned*>(&smeta[s].flags);
    if (flags & kSegEnd) {
      const int slot = smeta[s].slot;
      if (slot < 0 && !(flags & kTaskEnd)) {       // a whole item's segment: into its totals
#pragma unroll
        for (int k = 0; k < K; ++k) {
          s_tot[k * kConsumers + ct] += acc[k];
          acc[k] = 0.0;
        }
      } else {
        SegSums<K> a;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          a.v[k] = acc[k];
          acc[k] = 0.0;
        }
        end_segment<NCW, K>(v, item, smeta[s].item, slot, smeta[s].seg, flags, a, s_tot);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
  }
}

// Consumer layouts the kernel is instantiated for: NCW warps x K targets, the
// CTAs per SM the register allocation is sized for, the depth of the
// shared-memory ring (3 stages let six CTAs share an SM; 4 stages at five
// CTAs hide the producer's list walks better on short items), and whether
// warps whose rows hold no real target skip their work (worth it when many
// items are smaller than a tile; a cost of about 1 % otherwise).  Layouts
// kLayoutSkip + i are layout i with skipping.
struct Layout {
  int ncw, k, minb, stages;
};
static const Layout kLayouts[kLayoutSkip] = {{4, 2, 6, 3}, {2, 4, 6, 3}, {4, 2, 5, 4}};

template <bool F32, int KERN, bool SKIP>
static const void* kernel_for_skip(int base) {
  if constexpr (KERN == BLDTT_COULOMB || KERN == kKernCoulombYukawa) {
    if (base == 1) return reinterpret_cast<const void*>(&k_interact<F32, KERN, 2, 4, 6, 3, SKIP>);
    if (base == 2) return reinterpret_cast<const void*>(&k_interact<F32, KERN, 4, 2, 5, 4, SKIP>);
  }
  // The oscillatory kernel's packed loop takes 90 registers; at six CTAs its
  // spills cost more than the two CTAs give (1E5 points of a Plummer sphere, n 6, leaves of
  // 1000, whole compute phase: 4.39 ms at six, 4.27 at five, 4.20 at four).
  if constexpr (F32 && KERN == BLDTT_OSCILLATORY)
    return reinterpret_cast<const void*>(&k_interact<F32, KERN, 4, 2, 4, 3, SKIP>);
  else
    return reinterpret_cast<const void*>(&k_interact<F32, KERN, 4, 2, 6, 3, SKIP>);
}

template <bool F32, int KERN>
static const void* kernel_for(int layout) {
  if constexpr (F32) {
    if (layout >= kLayoutSkip) return kernel_for_skip<F32, KERN, true>(layout - kLayoutSkip);
  }
  // FP64 leaves idle rows out in every layout (rows_f64); a skipping layout is
  // its base layout.
  return kernel_for_skip<F32, KERN, false>(layout % kLayoutSkip);
}

// Layouts instantiated for a kernel (the autotuner tries these).
int layouts_available(int kernel, int* out) {
  const int nbase = (kernel == BLDTT_COULOMB || kernel == kKernCoulombYukawa) ? kLayoutSkip : 1;
  int n = 0;
  for (int i = 0; i < nbase; ++i) out[n++] = i;
  for (int i = 0; i < nbase; ++i) out[n++] = kLayoutSkip + i;
  return n;
}

int layout_threads(int layout) { return (kLayouts[layout % kLayoutSkip].ncw + 1) * 32; }

static const void* select_kernel(int kernel, bool f32, int layout) {
  switch (kernel) {
    case BLDTT_COULOMB: return f32 ? kernel_for<true, BLDTT_COULOMB>(layout) : kernel_for<false, BLDTT_COULOMB>(layout);
    case BLDTT_YUKAWA: return f32 ? kernel_for<true, BLDTT_YUKAWA>(layout) : kernel_for<false, BLDTT_YUKAWA>(layout);
    case kKernCoulombYukawa:
      return f32 ? kernel_for<true, kKernCoulombYukawa>(layout) : kernel_for<false, kKernCoulombYukawa>(layout);
    case BLDTT_OSCILLATORY: return f32 ? kernel_for<true, BLDTT_OSCILLATORY>(layout) : kernel_for<false, BLDTT_OSCILLATORY>(layout);
    case BLDTT_REG_COULOMB: return f32 ? kernel_for<true, BLDTT_REG_COULOMB>(layout) : kernel_for<false, BLDTT_REG_COULOMB>(layout);
    default: return f32 ? kernel_for<true, BLDTT_TEST_POLY>(layout) : kernel_for<false, BLDTT_TEST_POLY>(layout);
  }
}

// Persistent grid of every segment: all CTAs that fit on the device at once
// (never more than the segment's items).
int interaction_grids(bldtt_plan* p) {
  int dev = 0, sms = 0;
  BL_CUDA(cudaGetDevice(&dev));
  BL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const bool f32 = p->precision == BLDTT_FP32_BULK;
  for (auto& seg : p->segments) {
    int per_sm = 0;
    seg.threads = layout_threads(seg.layout);
    // all of the SM's 228 KB as shared memory: at the default carveout five of the six CTAs fit
    BL_CUDA(cudaFuncSetAttribute(select_kernel(seg.kernel, f32, seg.layout),
                                 cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared));
    BL_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, select_kernel(seg.kernel, f32, seg.layout), seg.threads, 0));
    if (per_sm < 1) per_sm = 1;
    const int g = sms * per_sm;
    seg.grid = g > seg.count ? seg.count : g;
    if (seg.grid < 1) seg.grid = 1;
  }
  return BLDTT_OK;
}

// Whether a pair of overlapping or touching clusters may be approximated.  With
// (r_t + r_s) < theta R all points of the two are (1 - theta) R or more apart: far
// more than their rounding in FP32 (6e-8 R) up to theta = 0.999.  The learned
// selector may take any pair below 1 that lies in its box of features (the
// fifth is (r_t + r_s)/R).
static bool clusters_may_overlap(const bldtt_plan* p) {
  return p->theta > 0.999 || (p->learned && p->selector_net && p->sel_hi[4] > 0.999f);
}

static InteractView make_view(const bldtt_plan* p) {
  const Tree& tt = p->tt;
  const Tree& st = p->st;
  InteractView v;
  v.items = p->items;
  v.parts = p->parts;
  v.seg_sums = p->seg_sums;
  v.arrived = p->item_counter + kMaxSegmentsLaunch;
  v.nitems = p->nitems;
  v.counter = p->item_counter;
  v.list_ptr = p->list_ptr;
  v.list_src = p->list_src;
  v.nct = tt.nclusters;
  v.t_parent = tt.parent;
  v.s_leaf_first = st.leaf_first;
  v.s_leaf_last = st.leaf_last;
  v.pad_prefix = p->pad_prefix;
  v.chunk_frame = p->chunk_frame;
  v.pool_res = p->pool_res;
  v.item_box = p->item_box;
  v.deg = p->deg;
  v.pool = p->pool;
  v.tx = tt.x;
  v.ty = tt.y;
  v.tz = tt.z;
  for (int i = 0; i < kMaxDegrees; ++i) {
    v.t_nodes[i] = i < p->deg.n ? p->nodes_t[i] : nullptr;
    v.phit[i] = i < p->deg.n ? p->phit_d[i] : nullptr;
  }
  v.phi_near = p->phi_near;
  v.err = p->dev_err;
  v.t_problem = tt.problem;
  v.prob_prm = p->prob_prm;
  v.prob_kappa = p->prob_kappa;
  v.prob_kernel = p->prob_kernel;
  v.overlap = clusters_may_overlap(p);
  return v;
}

// One segment's persistent launch over items [first, first + count).
static int launch_segment(const bldtt_plan* p, const InteractView& base, int g, cudaStream_t s) {
  const auto& seg = p->segments[g];
  InteractView v = base;
  v.items = p->items + seg.first;
  v.parts = p->parts + seg.first;
  v.nitems = seg.count;
  v.counter = p->item_counter + g;
  if (v.item_box) v.item_box = p->item_box + (int64_t)seg.first * (2 * kItemGroups);
  void* args[] = {&v};
  BL_CUDA(cudaLaunchKernel(select_kernel(seg.kernel, p->precision == BLDTT_FP32_BULK, seg.layout),
                           dim3(seg.grid), dim3(seg.threads), args, 0, s));
  return BLDTT_OK;
}

int run_segment(bldtt_plan* p, int g, cudaStream_t s) {
  BL_CUDA(cudaMemsetAsync(p->item_counter + g, 0, sizeof(int32_t), s));
  BL_TRY(launch_segment(p, make_view(p), g, s));
  BL_LAUNCHED(p->compute_counter.launches);
  return BLDTT_OK;
}

int run_interactions(bldtt_plan* p, cudaStream_t s) {
  if (p->nitems == 0 || p->segments.empty()) return BLDTT_OK;
  const InteractView v = make_view(p);
  BL_CUDA(cudaMemsetAsync(p->item_counter, 0, p->counter_words * sizeof(int32_t), s));
  for (int g = 0; g < (int)p->segments.size(); ++g) {
    BL_TRY(launch_segment(p, v, g, s));
    BL_LAUNCHED(p->compute_counter.launches);
  }
  return BLDTT_OK;
}

}  // namespace bldtt
