// The FP64 exponential of the FP64 sweeps, on the integer pipes.
//
// This GPU's FP64 pipe retires two lanes per SM and clock, its integer pipes 32
// (multiply-high, wide multiply) to 128 (add): measured 1.99 DFMA, 1.68 DADD, 24.7
// IMAD.WIDE, 31.8 IMAD.HI, 63 shifts and logic, 125 adds. A plan entry of the FP64
// sweeps needs three FP64 operations besides its exponential (a_i + b_j, the FMA
// with the cost, the FMA into the sum); CUDA's exp adds about twenty more, which
// made it six sevenths of the FP64 sweeps' time. exp64 takes none: the argument's
// bits become a 96-bit fixed-point t log2(e), whose top fraction bits index a
// table of 2^(j / 2048) and whose rest goes through a cubic in fixed point (the
// table-driven scheme of P. T. P. Tang, ACM TOMS 15, 1989, with the Taylor
// polynomial of 2^x). About 55 integer instructions, 14 of them multiplies.
// Errors (4e5 arguments per range, extended precision): at most 0.70 ulp for |t| < 300
// and 0.74 up to |t| = 708, mean below 0.015, rms 0.29 (perfect rounding: 0.289; CUDA's
// exp: 0.87, 0.01, 0.30).
// Measured (FP64, CUDA's exp -> this one): solve of the 28 x 28 grid 75.1 -> 29.9 ms,
// its marginals 267 -> 153 us, the Hessian-vector product at 1501 x 1999 763 -> 379 us,
// Round of the 64 x 64 grid 2.54 -> 0.71 ms. (With subnormal results left to CUDA's
// exp, which most warps of a wide cost then call: 50.9 ms, 190, 570 us and 1.21 ms.)
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace eot {

constexpr int kExpBits = 11;
constexpr int kExpSize = 1 << kExpBits;

struct ExpTable {
  unsigned long long v[kExpSize];
};
namespace exp64_detail {
// floor(a b / 2^126) for a, b in Q2.126
constexpr unsigned __int128 mul_q126(unsigned __int128 a, unsigned __int128 b) {
  const unsigned __int128 lo64 = ~0ull;
  const unsigned __int128 ah = a >> 64, al = a & lo64, bh = b >> 64, bl = b & lo64;
  const unsigned __int128 mid1 = ah * bl, mid2 = al * bh;
  const unsigned __int128 mid = (mid1 & lo64) + (mid2 & lo64) + ((al * bl) >> 64);
  const unsigned __int128 hi = ah * bh + (mid1 >> 64) + (mid2 >> 64) + (mid >> 64);
  return (hi << 2) | ((mid & lo64) >> 62);
}
// 2^(j / 2048) in Q2.62, plus half a unit of the FP64 result (exp64 cuts 10 bits)
constexpr ExpTable make_table() {
  ExpTable t{};
  const unsigned __int128 root = ((unsigned __int128)0x40058bce410147e8ull << 64) | 0x4a2f2a71570c7978ull;
  unsigned __int128 p = (unsigned __int128)1 << 126;
  for (int j = 0; j < kExpSize; ++j) {
    t.v[j] = (unsigned long long)((p + ((unsigned __int128)1 << 63)) >> 64) + 512ull;
    p = mul_q126(p, root);
  }
  return t;
}
}  // namespace exp64_detail
static __device__ const ExpTable kExpTable = exp64_detail::make_table();

// Copies the table to shared memory (all threads of the CTA; a barrier before use).
__device__ __forceinline__ void exp_fill(ExpTable& s) {
  for (int k = threadIdx.x; k < kExpSize / 2; k += blockDim.x)
    reinterpret_cast<ulonglong2*>(s.v)[k] = __ldg(reinterpret_cast<const ulonglong2*>(kExpTable.v) + k);
}

static __device__ __noinline__ double exp_rare(double t) { return exp(t); }

// high 64 bits of a b (+ the mean of what the dropped low products carry)
__device__ __forceinline__ uint64_t mulhi_approx(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl) {
  return (uint64_t)ah * bh + ((uint64_t)__umulhi(ah, bl) + __umulhi(al, bh) + 1u);
}

// exp(t) for every t; `tab` in shared memory
__device__ __forceinline__ double exp64(double t, const ExpTable& tab) {
  const uint32_t hi = (uint32_t)__double2hiint(t), lo = (uint32_t)__double2loint(t);
  const uint32_t ax = hi & 0x7fffffffu;
  // 2^-20 <= |t| < 708.39 (normal results). Below, results are subnormal down to -745.5:
  // they take the same way with 2^-64 put aside, since a sweep over a wide cost meets
  // them in most warps; the rest (tiny, overflowing, NaN) is rare.
  bool sub = false;
  if (ax - 0x3eb00000u >= 0x4086232bu - 0x3eb00000u) {
    if (hi >= 0xc0874c00u && hi < 0xfff00000u) return 0.0;  // t < -745.5
    if (ax < 0x3c900000u) return 1.0;                       // |t| < 2^-54
    sub = hi >= 0xc086232bu && hi < 0xc0874c00u;
    if (!sub) return exp_rare(t);
  }
  // H + L = |t| log2(e) as mantissa x 2^-63 / 2^64 (96 bits, without the product of the
  // low words), then W = t log2(e) 2^85 (96 bits, two's complement)
  const uint32_t mh = __funnelshift_l(lo, ax, 11) | 0x80000000u, ml = lo << 11;
  const uint64_t A = (uint64_t)mh * 0x5c17f0bcu, B = (uint64_t)ml * 0xb8aa3b29u;
  const uint64_t H0 = (uint64_t)mh * 0xb8aa3b29u + (A >> 32);
  uint32_t L, hl, hh;
  asm("add.cc.u32 %0, %3, %4;\n\taddc.cc.u32 %1, %5, %6;\n\taddc.u32 %2, %7, 0;"
      : "=&r"(L), "=&r"(hl), "=r"(hh)
      : "r"((uint32_t)A), "r"((uint32_t)B), "r"((uint32_t)H0), "r"((uint32_t)(B >> 32)), "r"((uint32_t)(H0 >> 32)));
  const uint32_t sh = 1032u - (ax >> 20);  // 0 .. 29
  const uint32_t sgn = (uint32_t)((int32_t)hi >> 31);
  const uint32_t w2 = ((hh >> sh) - (sub ? 64u << 21 : 0u)) ^ sgn;
  const uint32_t w1 = __funnelshift_r(hl, hh, sh) ^ sgn;
  const uint32_t w0 = __funnelshift_r(L, hl, sh) ^ sgn;
  // 11 bits of exponent, 11 of table index, 64 of x2 = 2048 x (x < 2^-11)
  const uint64_t T = tab.v[(w2 >> 10) & (kExpSize - 1)];
  const uint32_t rh = __funnelshift_l(w1, w2, 22), rl = __funnelshift_l(w0, w1, 22);
  // (2^x - 1) / x2 = s: ln2^k / k! scaled by 2048^(1-k), in units of 2^-45, then 2^-64;
  // the constants after a multiplication hold half a unit more, for what its floor drops
  const uint32_t q3 = __umulhi(rh, 39u) + 465603u;
  const uint32_t q2 = __umulhi(rh, q3) + 4127059965u;
  const uint64_t s = (uint64_t)__umulhi(rh, q2) * (1u << 19) + (0xb17217f7d1cf79acull + (1ull << 18));
  const uint64_t p = mulhi_approx(rh, rl, (uint32_t)(s >> 32), (uint32_t)s);  // (2^x - 1) 2^75
  const uint64_t tp = mulhi_approx((uint32_t)(T >> 32), (uint32_t)T, (uint32_t)(p >> 32), (uint32_t)p);
  const uint64_t m = T + (tp >> 11);  // 2^(j / 2048 + x) in Q2.62
  const uint32_t rlo = __funnelshift_r((uint32_t)m, (uint32_t)(m >> 32), 10);
  const uint32_t rhi = ((uint32_t)(m >> 32) >> 10) + ((uint32_t)((int32_t)w2 >> 1) & 0xfff00000u) + (1022u << 20);
  const double r = __hiloint2double((int)rhi, (int)rlo);
  return sub ? r * 5.42101086242752217e-20 : r;
}

// (double)x on the integer pipes (exact; zeros, subnormals and non-finite values
// take the conversion instruction, which runs at the FP64 pipe's rate)
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x), e = b & 0x7f800000u;
  if (e - 0x00800000u >= 0x7f000000u) return (double)x;
  return __hiloint2double((int)((((b & 0x7fffffffu) >> 3) + 0x38000000u) | (b & 0x80000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

constexpr float kCutMax = 1.0e30f;  // callers fall back to FP64 where |cut_f32(x)| reaches this
// x cut (towards 0) to FP32 on the integer pipes (a conversion instruction would
// run at the FP64 pipe's rate); |x| < 2^-126 gives 0, |x| >= 2^128 +-inf, NaN NaN
__device__ __forceinline__ float cut_f32(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t a = hi & 0x7fffffffu;
  uint32_t r = __funnelshift_l(lo, a - (896u << 20), 3);
  if (a < (897u << 20)) r = 0u;
  if (a >= (1151u << 20)) r = a > 0x7ff00000u || (a == 0x7ff00000u && lo) ? 0x7fc00000u : 0x7f800000u;
  return __uint_as_float(r | (hi & 0x80000000u));
}
__device__ __forceinline__ float cut_f32(float x) { return x; }

}  // namespace eot
