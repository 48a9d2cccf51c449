// 1/r and exp(-kappa r)/r to FP64 accuracy in integer arithmetic.
//
// The FP64 pipe of this GPU issues 1.7 lanes per clock and SM, the integer pipe
// 64; an FP64 evaluation of 1/r takes 12 FP64 instructions (3 differences, 3
// for r^2, 5 around the reciprocal square root, 1 to accumulate), one of
// exp(-kappa r)/r about 40.  Here only the differences and the accumulation
// stay FP64 (4 instructions).  From the differences' bits on the value is
// carried in 64-bit fixed point with 58 or more significant bits, so the error of
// 1/r and 1/sqrt(r^2 + kappa^2) is below the final rounding to 53 bits; the FP64
// expressions they replace round r^2, the square root and the quotient or product
// one by one.
//
//   d      53-bit mantissas aligned to the largest exponent E of the three
//   S      sum of squares over 2^64 (the squares of the low words, below
//          2^-58 of S, are dropped):        r^2 = S 2^(2 (E - 1053))
//   Y      (S / 2^62)^-1/2 by one Householder step of order three from a float
//          seed, the residual 1 - S Y0^2 exact to 2^-62
//   exp2   2^-t, t = kappa log2(e) r: integer part, 8 table bits and a degree-5
//          Taylor polynomial of the rest (Tang's table-driven scheme, ACM TOMS
//          15, 1989, in fixed point)
//
// exp(-kappa r) turns r's relative error of about 2^-59 into kappa r times as
// much, so the screened value is off by up to kappa r 1.45 2^-58 beside the last
// rounding (9 units of 2^-53 at kappa r = 300; FP64 expressions, which round r and
// kappa r to 2^-53, up to some hundreds).
//
// Functions are plain C++ so that they can be checked on a host against
// extended precision.
#pragma once

#include <stdint.h>
#include <string.h>
#ifndef __CUDACC__
#include <math.h>
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace bldtt {
namespace fixed64 {

typedef unsigned long long u64;
typedef long long i64;

__host__ __device__ __forceinline__ u64 bits_of(double v) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(v);
#else
  u64 b;
  memcpy(&b, &v, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double of_bits(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double v;
  memcpy(&v, &b, 8);
  return v;
#endif
}
__host__ __device__ __forceinline__ u64 mul_hi(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ uint32_t mul_hi32(uint32_t a, uint32_t b) { return (uint32_t)(((u64)a * b) >> 32); }
__host__ __device__ __forceinline__ u64 wide(uint32_t a, uint32_t b) { return (u64)a * b; }
__host__ __device__ __forceinline__ int leading_zeros(u64 v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}
__host__ __device__ __forceinline__ int leading_zeros32(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return __builtin_clz(v);
#endif
}
// High word of the pair (hi, lo) shifted left by s, 0 <= s < 32.
__host__ __device__ __forceinline__ uint32_t shl_pair(uint32_t hi, uint32_t lo, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, (uint32_t)s);
#else
  return (uint32_t)((((u64)hi << 32 | lo) << s) >> 32);
#endif
}
// Right shifts of 32 bits and of the word pair (hi, lo) by s >= 0, the latter's
// low word; 0 (or, for the pair, of no use: its high word is 0) from s = 32 on.
__host__ __device__ __forceinline__ uint32_t shr(uint32_t v, int s) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
  return r;
#else
  return s > 31 ? 0u : v >> s;
#endif
}
__host__ __device__ __forceinline__ uint32_t shr_pair(uint32_t hi, uint32_t lo, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_rc(lo, hi, (uint32_t)s);
#else
  return s > 31 ? hi : (uint32_t)((((u64)hi << 32) | lo) >> s);
#endif
}
__host__ __device__ __forceinline__ int exponent_of(u64 b) { return (int)(b >> 52) & 0x7ff; }

// One coordinate difference aligned to the exponent E >= its own: h (31 bits)
// and l (the next 31); adds h^2 to S and h l to C.
__host__ __device__ __forceinline__ void add_square(u64 b, int E, u64& S, u64& C) {
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  const int s = E - exponent_of(b);
  const uint32_t m = (hi & 0xfffffu) | 0x100000u;
  const uint32_t H = (m << 10) | (lo >> 22);
  const uint32_t l = shr_pair(H, lo << 10, s) >> 1;
  const uint32_t h = shr(H, s);
  S += wide(h, h);
  C += wide(h, l);
}

// Exponents at which FP64's r^2 neither underflows to 0 nor overflows.
constexpr int kMinE = 485, kMaxE = 1534;

// (S / 2^62)^-1/2 in units of 2^-62, S in [2^60, 2^64).
__host__ __device__ __forceinline__ u64 inv_sqrt(u64 S) {
  const uint32_t Sh = (uint32_t)(S >> 32), Sl = (uint32_t)S;
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((float)Sh));
#else
  const float y = 1.0f / sqrtf((float)Sh);
#endif
  const uint32_t Y0 = (uint32_t)(y * 549755813888.f);          // 2^39: Y0 / 2^24, exact
  const u64 P = wide(Y0, Y0);
  const uint32_t Ph = (uint32_t)(P >> 32), Pl = (uint32_t)P;
  // S P / 2^48 modulo 2^64, and what is missing to 1 (2^62)
  const u64 T = (wide(Sh, Ph) << 16) + (wide(Sh, Pl) >> 16) + (wide(Sl, Ph) >> 16) + (mul_hi32(Sl, Pl) >> 16);
  const i64 e = (i64)((1ull << 62) - T);                        // |e| < 2^42
  const int32_t es = (int32_t)(e >> 20);
  const i64 c = (e >> 1) + (i64)(((u64)((i64)es * es) * 3) >> 25);   // e/2 + 3 e^2/8
  const i64 ch = c >> 32;
  return ((u64)Y0 << 38) + (u64)((ch * (i64)Y0) << 8) + (wide((uint32_t)c, Y0) >> 24);
}

// M 2^-62 2^X as a double (M > 0), rounded to nearest; 0 if !ok.
__host__ __device__ __forceinline__ double to_double(u64 M, int X, bool ok) {
  const int lz = leading_zeros(M);
  const int e = 1023 + X + 1 - lz;              // biased exponent, before a carry of the rounding
  const u64 n = M << lz;
  // the implicit bit of n >> 11 adds one to the exponent field
  u64 b = ((u64)(uint32_t)(e - 1) << 52) + (n >> 11) + ((n >> 10) & 1);
  if (!(ok && e >= 1)) {                        // one branch for both: rarely taken
    const int sh = 12 - e;                      // subnormal: units of 2^-1074
    b = !ok || sh > 64 ? 0ull : sh == 64 ? n >> 63 : (n >> sh) + ((n >> (sh - 1)) & 1);
  }
  return of_bits(b);
}

// Sum of squares of the three differences (and, for the regularized kernel, of
// a fourth term); E out of range: the pair contributes nothing.
__host__ __device__ __forceinline__ u64 sum_squares(double dx, double dy, double dz, int* E) {
  const u64 bx = bits_of(dx), by = bits_of(dy), bz = bits_of(dz);
  int e = exponent_of(bx), f = exponent_of(by), g = exponent_of(bz);
  e = e > f ? e : f;
  e = e > g ? e : g;
  *E = e;
  u64 S = 0, C = 0;
  add_square(bx, e, S, C);
  add_square(by, e, S, C);
  add_square(bz, e, S, C);
  return S + (C >> 30);
}

// Differences in 64-bit fixed point, units of 2^-k, |d| < 2^62: nothing is left
// to the FP64 pipe but the accumulation.  Each coordinate's rounding to whole
// units moves d by one unit at most, so pairs below 2^56 units (kFixedTop: the
// size of the largest high word) are left to FP64 differences: there the unit
// is 2^-56 of r, beyond it less, against 2^-54 of an FP64 result.
constexpr uint32_t kFixedTop = 1u << 24;
__host__ __device__ __forceinline__ int32_t high_ones(i64 d) {
  const int32_t h = (int32_t)(d >> 32);
  return h ^ (h >> 31);
}
__host__ __device__ __forceinline__ uint32_t fixed_top(i64 dx, i64 dy, i64 dz) {     // < 2^30
  return (uint32_t)(high_ones(dx) | high_ones(dy) | high_ones(dz));
}
// Sum of squares as sum_squares gives it, top >= kFixedTop.
__host__ __device__ __forceinline__ u64 sum_squares_fixed(i64 dx, i64 dy, i64 dz, uint32_t top, int k, int* E) {
  const int s = leading_zeros32(top) - 1;
  *E = 1085 - k - s;
  u64 S = 0;
  i64 C = 0;
  const i64 d[3] = {dx, dy, dz};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const u64 a = (u64)d[i];
    const int32_t h = (int32_t)shl_pair((uint32_t)(a >> 32), (uint32_t)a, s);
    const int32_t l = (int32_t)(((uint32_t)a << s) >> 2);
    S += (u64)((i64)h * h);
    C += (i64)h * l;
  }
  return S + (u64)(C >> 29);
}

// 1/r; 0 where FP64's r^2 is 0 (or overflows).
__host__ __device__ __forceinline__ double inv_r_of(u64 S, int E) {
  const u64 Y = inv_sqrt(S);
  // Y in (2^61.2, 2^63]: two cases instead of a count of leading zeros
  const bool big = (Y >> 62) != 0;
  const u64 b = ((u64)(uint32_t)((big ? 2044 : 2043) - E) << 52) + (big ? (Y + 512) >> 10 : (Y + 256) >> 9);
  return of_bits((unsigned)(E - kMinE) <= (unsigned)(kMaxE - kMinE) ? b : 0ull);
}
__host__ __device__ __forceinline__ double inv_r(double dx, double dy, double dz) {
  int E;
  const u64 S = sum_squares(dx, dy, dz, &E);
  return inv_r_of(S, E);
}

// 1/sqrt(r^2 + kappa^2), kappa >= 0; 0 where FP64's r^2 is 0 (or overflows).
__host__ __device__ __forceinline__ double inv_sqrt_r2_kappa2(double dx, double dy, double dz, double kappa) {
  const u64 bx = bits_of(dx), by = bits_of(dy), bz = bits_of(dz), bk = bits_of(kappa);
  int e = exponent_of(bx), f = exponent_of(by), g = exponent_of(bz);
  e = e > f ? e : f;
  e = e > g ? e : g;
  const int E3 = e;
  f = exponent_of(bk);
  e = e > f ? e : f;
  u64 S = 0, C = 0;
  add_square(bx, e, S, C);
  add_square(by, e, S, C);
  add_square(bz, e, S, C);
  add_square(bk, e, S, C);
  S += C >> 30;
  // four squares: S in [2^60, 2^64]; S just below 4 2^62 at most, as h < 2^31
  const u64 Y = inv_sqrt(S);
  const bool ok = (unsigned)(E3 - kMinE) <= (unsigned)(kMaxE - kMinE) && e <= kMaxE;
  return to_double(Y, 1022 - e, ok);
}

// kappa log2(e) = m 2^-64 2^x, m of 64 significant bits (m = 0: kappa = 0).
struct Screen {
  u64 m;
  int x;
};
__host__ __device__ __forceinline__ Screen make_screen(double kappa) {
  Screen k{0, 0};
  const u64 b = bits_of(kappa);
  if (exponent_of(b) == 0) return k;            // 0 (and subnormals: exp(-kappa r) is 1)
  const u64 m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 11;   // [2^63, 2^64)
  k.m = mul_hi(m, 0xb8aa3b295c17f0bcull);       // log2(e) 2^63: product over 2^64 in [2^62.5, 2^63.6)
  k.x = exponent_of(b) - 1023 + 2;
  if (!(k.m >> 63)) {
    k.m <<= 1;
    k.x -= 1;
  }
  return k;
}

// 2^(-j/256) in units of 2^-63.
#ifdef __CUDACC__
static __device__ const
#else
static const
#endif
u64 kExp2[256] = {
    0x8000000000000000ull, 0x7fa765aca88f6453ull, 0x7f4f08ae3dc7c426ull, 0x7ef6e8da4b544f9aull,
    0x7e9f06067a4360baull, 0x7e47600890f223deull, 0x7deff6b672f84e24ull, 0x7d98c9e62113e1faull,
    0x7d41d96db915019dull, 0x7ceb252375c9cf9bull, 0x7c94acddaeea5d3aull, 0x7c3e7072d904a6ceull,
    0x7be86fb985689ddcull, 0x7b92aa886214411cull, 0x7b3d20b6399fc237ull, 0x7ae7d219f329b948ull,
    0x7a92be8a92436616ull, 0x7a3de5df36dcfeefull, 0x79e947ef1d320d2dull, 0x7994e4919db5d74eull,
    0x7940bb9e2cffd89dull, 0x78ecccec5bb84661ull, 0x78991853d684a285ull, 0x78459dac65f45bb5ull,
    0x77f25ccdee6d7ae6ull, 0x779f559070195e36ull, 0x774c87cc06d1812eull, 0x76f9f358ea0c5249ull,
    0x76a7980f6cca15c2ull, 0x765575c7fd81d5a0ull, 0x76038c5b260e5eeeull, 0x75b1dba18b9b4c20ull,
    0x75606373ee921c97ull, 0x750f23ab2a87593eull, 0x74be1c203627c62bull, 0x746d4cac2325a155ull,
    0x741cb5281e25ee34ull, 0x73cc556d6eadce5full, 0x737c2d55770fe711ull, 0x732c3cb9b459d38bull,
    0x72dc8373be41a454ull, 0x728d015d47136b40ull, 0x723db6501b9ed447ull, 0x71eea2262324cb0cull,
    0x719fc4b95f452d29ull, 0x71511de3ebec8913ull, 0x7102ad7fff41e9b4ull, 0x70b47367e994ae92ull,
    0x70666f76154a7089ull, 0x7018a18506ccf314ull, 0x6fcb096f5c782210ull, 0x6f7da70fce881bf9ull,
    0x6f307a412f074892ull, 0x6ee382de69bc7bf8ull, 0x6e96c0c284192610ull, 0x6e4a33c89d278e49ull,
    0x6dfddbcbed791babull, 0x6db1b8a7c714a92bull, 0x6d65ca379564e639ull, 0x6d1a1056dd26c382ull,
    0x6cce8ae13c57ebdbull, 0x6c8339b26a25494eull, 0x6c381ca636d99642ull, 0x6bed33988bcbfab5ull,
    0x6ba27e656b4eb57aull, 0x6b57fce8f09dd17full, 0x6b0daeff4fcde703ull, 0x6ac39484d5bae8c5ull,
    0x6a79ad55e7f6fd10ull, 0x6a2ff94f04b962b0ull, 0x69e6784cc2cd61bdull, 0x699d2a2bd181482aull,
    0x69540ec8f895722dull, 0x690b2601182b5e56ull, 0x68c26fb128b4cd63ull, 0x6879ebb63ae2edc6ull,
    0x683199ed779592caull, 0x67e97a341fca775bull, 0x67a18c678c8c8c61ull, 0x6759d0652ee352afull,
    0x6712460a8fc24072ull, 0x66caed354ff83222ull, 0x6683c5c3281ee6e9ull, 0x663ccf91e88a8873ull,
    0x65f60a7f79393e2eull, 0x65af7669d9c2cbe4ull, 0x6569132f21483ba7ull, 0x6522e0ad7e639312ull,
    0x64dcdec3371793d1ull, 0x64970d4ea8bf8766ull, 0x64516c2e47ff1623ull, 0x640bfb40a0b22959ull,
    0x63c6ba6455dcd8aeull, 0x6381a978219b628full, 0x633cc85ad5122fbdull, 0x62f816eb585de1edull,
    0x62b39508aa836d6full, 0x626f4291e1603dd5ull, 0x622b1f66299a6599ull, 0x61e72b64c690d8afull,
    0x61a3666d124bb204ull, 0x615fd05e7d6c83e4ull, 0x611c69188f1eb339ull, 0x60d9307ae507dd9aull,
    0x6096266533384a2bull, 0x60534ab7441b6546ull, 0x60109d50f86846d8ull, 0x5fce1e124712437cull,
    0x5f8bccdb3d398841ull, 0x5f49a98bfe1bc11cull, 0x5f07b404c304c9f1ull, 0x5ec5ec25db3f6a41ull,
    0x5e8451cfac061b5full, 0x5e42e4e2b073d935ull, 0x5e01a53f7974fd86ull, 0x5dc092c6adb825b8ull,
    0x5d7fad59099f22feull, 0x5d3ef4d75f2ff504ull, 0x5cfe69229605cef5ull, 0x5cbe0a1bab4226dfull,
    0x5c7dd7a3b17dcf75ull, 0x5c3dd19bd0ba1c1aull, 0x5bfdf7e546520f3eull, 0x5bbe4a6164eb92f4ull,
    0x5b7ec8f19468bbc9ull, 0x5b3f737751d915c8ull, 0x5b0049d42f6afbb6ull, 0x5ac14be9d45cf869ull,
    0x5a827999fcef3242ull, 0x5a43d2c67a54e0c0ull, 0x5a05575132a5cc20ull, 0x59c7071c20cfd70cull,
    0x5988e20954889245ull, 0x594ae7faf23eda52ull, 0x590d18d3330c7f1eull, 0x58cf747464a7f584ull,
    0x5891fac0e95612c8ull, 0x5854ab9b37dbd1e5ull, 0x581786e5db7022c2ull, 0x57da8c8373adc331ull,
    0x579dbc56b48521baull, 0x57611642662e4a33ull, 0x57249a29651adc07ull, 0x56e847eea1e80a49ull,
    0x56ac1f752150a563ull, 0x5670209ffc1f2e82ull, 0x56344b525f1ff495ull, 0x55f89f6f8b133af4ull,
    0x55bd1cdad49f699cull, 0x5581c377a44346f0ull, 0x5546932976483b15ull, 0x550b8bd3dab49cbdull,
    0x54d0ad5a753e077cull, 0x5495f7a0fd3bbb8eull, 0x545b6a8b3d990704ull, 0x542105fd14c7b869ull,
    0x53e6c9da74b29ab5ull, 0x53acb60762affaaeull, 0x5372ca67f774358full, 0x533906e05f045106ull,
    0x52ff6b54d8a89c75ull, 0x52c5f7a9b6df5b77ull, 0x528cabc35f4f799dull, 0x525387864abb4762ull,
    0x521a8ad704f3404full, 0x51e1b59a2cc8da3eull, 0x51a907b474015dc9ull, 0x5170810a9f48c7cfull,
    0x513821818624b40cull, 0x50ffe8fe12e750c4ull, 0x50c7d76542a25b72ull, 0x508fec9c251a267cull,
    0x50582887dcb8a7e1ull, 0x50208b0d9e8090dfull, 0x4fe91412b2006e83ull, 0x4fb1c37c7145d328ull,
    0x4f7a993048d088d7ull, 0x4f439513b785cc80ull, 0x4f0cb70c4ea39210ull, 0x4ed5feffb1b3d155ull,
    0x4e9f6cd3967fdba8ull, 0x4e69006dc503ba65ull, 0x4e32b9b417619617ull, 0x4dfc988c79d52661ull,
    0x4dc69cdceaa72a9cull, 0x4d90c68b7a20eb1eull, 0x4d5b157e4a7fc325ull, 0x4d25899b8fe8b365ull,
    0x4cf022c9905bfd32ull, 0x4cbae0eea3a8c63cull, 0x4c85c3f13360c4d5ull, 0x4c50cbb7bacbf4cbull,
    0x4c1bf828c6dc54b8ull, 0x4be7492af621abd6ull, 0x4bb2bea4f8bd5847ull, 0x4b7e587d905625d1ull,
    0x4b4a169b900c2d00ull, 0x4b15f8e5dc6cbab0ull, 0x4ae1ff436b663ff7ull, 0x4aae299b443c4a6bull,
    0x4a7a77d47f7b84b1ull, 0x4a46e9d646edbf6aull, 0x4a137f87d58e025bull, 0x49e038d0777ca5e0ull,
    0x49ad159789f37496ull, 0x497a15c47b39d53eull, 0x4947393eca98fcd6ull, 0x49147fee085028d6ull,
    0x48e1e9b9d588e19bull, 0x48af7689e44b44eaull, 0x487d2645f7725895ull, 0x484af8d5e2a06536ull,
    0x4818ee218a3358eeull, 0x47e70610e3393241ull, 0x47b5408bf36472e2ull, 0x47839d7ad1009a90ull,
    0x47521cc5a2e6a9e0ull, 0x4720be54a071ad01ull, 0x46ef821011734e6bull, 0x46be67e04e28717cull,
    0x468d6fadbf2dd4f3ull, 0x465c9960dd74bd4bull, 0x462be4e23237a6efull, 0x45fb521a56ef0042ull,
    0x45cae0f1f545eb73ull, 0x459a9151c70f0819ull, 0x456a632296394492ull, 0x453a564d3cc4b723ull,
    0x450a6abaa4b77ecdull, 0x44daa053c812abd2ull, 0x44aaf701b0c72feeull, 0x447b6ead78aad636ull,
    0x444c0740496d4294ull, 0x441cc0a35c8cf8eaull, 0x43ed9abffb4c6bc9ull, 0x43be957f7ea712b6ull,
    0x438fb0cb4f468808ull, 0x4360ec8ce577ae44ull, 0x433248adc91fdd02ull, 0x4303c51791b21550ull,
    0x42d561b3e6243d8aull, 0x42a71e6c7ce464afull, 0x4278fb2b1bce0d15ull, 0x424af7d9981f7e98ull,
    0x421d1461d66f2023ull, 0x41ef50adcaa0d899ull, 0x41c1aca777db771bull, 0x41942838f07e22a3ull,
    0x4166c34c5615d0ecull, 0x41397dcbd952c4a6ull, 0x410c57a1b9fe12f6ull, 0x40df50b846ef302bull,
    0x40b268f9de0183baull, 0x4085a050ec0a036aull, 0x4058f6a7ecccd5b6ull, 0x402c6be96af2fb58ull,
};

// exp(-kappa r)/r; 0 where FP64's r^2 is 0 (or overflows), and where t = kappa
// log2(e) r is 2^11 or more (1/r is below 2^538).
__host__ __device__ __forceinline__ double screened_inv_r_of(u64 S, int E, const Screen& k) {
  const u64 Y = inv_sqrt(S);
  const u64 R = mul_hi(S, Y) << 3;              // r = R 2^-63 2^(E - 1022)
  const u64 Z = mul_hi(R, k.m);                 // t = kappa log2(e) r = Z 2^-w
  const int w = 1085 - k.x - E;
  const int sh = w > 56 ? w - 56 : 0, F = w > 56 ? 56 : w;
  const u64 U = sh > 63 ? 0ull : Z >> sh;       // t in units of 2^-F
  const bool ok = (unsigned)(E - kMinE) <= (unsigned)(kMaxE - kMinE) && (w >= 51 || k.m == 0);   // below: t >= 2^11
  const int Fs = F < 51 ? 51 : F;
  const u64 V = k.m == 0 ? 0ull : U;
  const int n = (int)(V >> Fs);
  const u64 G = V << (64 - Fs);                 // fraction, units of 2^-64
  const u64 W = G & 0x00ffffffffffffffull;      // below the 8 table bits
  const uint32_t Wh = (uint32_t)(W >> 32), Wl = (uint32_t)W;
  // 2^-w = 1 - w (c1 - w (c2 - w (c3 - w (c4 - w c5)))), c_i = ln(2)^i / i!
  const uint32_t h4 = 0x0276556eu - mul_hi32(Wh, 0x00576200u);
  const uint32_t h3 = 0x0e35846cu - mul_hi32(Wh, h4);
  const u64 h2 = 0x3d7f7bff058b1d51ull - (wide(Wh, h3) + mul_hi32(Wl, h3));
  const u64 h1 = 0xb17217f7d1cf79acull - mul_hi(W, h2);
  const u64 D = mul_hi(W, h1);
  const u64 T = kExp2[G >> 56];
  const u64 X = T - mul_hi(T, D);               // 2^-t 2^n in units of 2^-63, in (2^62, 2^63]
  const u64 M = mul_hi(Y, X) << 1;              // units of 2^-62
  return to_double(M, 1022 - E - n, ok);
}
__host__ __device__ __forceinline__ double screened_inv_r(double dx, double dy, double dz, const Screen& k) {
  int E;
  const u64 S = sum_squares(dx, dy, dz, &E);
  return screened_inv_r_of(S, E, k);
}

// v in units of 2^-k, rounded to nearest, modulo 2^64 (differences of values
// less than 2^62 units apart are right); k so that |v| 2^k < 2^1000.
__host__ __device__ __forceinline__ i64 to_fixed(double v, int k) {
  const u64 b = bits_of(v);
  const int e = exponent_of(b);
  const u64 m = e ? (b & 0xfffffffffffffull) | 0x10000000000000ull : b & 0xfffffffffffffull;
  const int sh = (e ? e : 1) - 1075 + k;          // v = m 2^(sh - k)
  u64 f;
  if (sh >= 0)
    f = sh > 63 ? 0ull : m << sh;
  else
    f = sh < -54 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1;
  return (i64)((b >> 63) ? 0ull - f : f);
}

}  // namespace fixed64
}  // namespace bldtt
