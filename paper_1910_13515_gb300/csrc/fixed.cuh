// fixed.cuh -- 53-bit arithmetic of the constraint solve on the integer and
// FP32 pipes.
//
// The GB300 issues one FP64 operation for every 60 FP32 ones or 27 64-bit
// integer adds (1.88 against 113 and 51 per clock and SM, measured), so the
// solve keeps its quantities in 64-bit fixed point: the exponents and the
// residual are sums with small integer coefficients, which integers form
// exactly; the exponential is a table value times 1 + p with p in two floats;
// and the Newton direction is an FP32 factorisation refined with the residual
// of the exact Jacobian-vector product.
//
//   L     multipliers times log2(e), units 2^-55 (range +-256)
//   X     exponents sum_k L_k phi_k(xi_i), units 2^-55: F_i = 2^X
//   F     doubles (the cell's state keeps them); read as integers in units 2^-58
//   m, G  targets and residuals, units 2^-58 (range +-32)
//
// The ranges are checked (multipliers_in_range, the sums in newton_fx); a cell outside them is solved
// in FP64, by a kernel of its own.
#pragma once
#include "d3q39_gen.cuh"

namespace lbm39 {
namespace fx {

typedef unsigned long long u64;
typedef long long s64;

// The exponential's table in shared memory; a kernel that solves first runs
// load_table() with the whole block.
__device__ __forceinline__ u64* table() {
  __shared__ u64 t[1024];
  return t;
}

// Table entries carry the constants of exp2_fixed: half of the 8 units of 2^-55
// that the final rounding drops (4 and 3 in turn, so that ties go either way), plus
// the exponent bits of its second float.
constexpr u64 TABLE_BIAS = 4ull + 0x81800000ull;

__device__ __forceinline__ void load_table() {
  u64* t = table();
  for (int j = threadIdx.x; j < 1024; j += blockDim.x) t[j] = gen::kExp2Fixed[j] + TABLE_BIAS - (j & 1);
  __syncthreads();
}

// Integer types whose sums the generated exponent code forms.
struct I64 {
  s64 v;
  __device__ __forceinline__ I64() {}
  __device__ __forceinline__ explicit I64(s64 x) : v(x) {}
  __device__ __forceinline__ explicit I64(int x) : v(x) {}
  friend __device__ __forceinline__ I64 operator+(I64 a, I64 b) { return I64((s64)((u64)a.v + (u64)b.v)); }
  friend __device__ __forceinline__ I64 operator-(I64 a, I64 b) { return I64((s64)((u64)a.v - (u64)b.v)); }
  friend __device__ __forceinline__ I64 mul_rn(I64 a, I64 b) { return I64((s64)((u64)a.v * (u64)b.v)); }
  friend __device__ __forceinline__ I64 fma(I64 a, I64 b, I64 c) { return I64((s64)((u64)a.v * (u64)b.v + (u64)c.v)); }
};

// 2^X as a double, X in units 2^-55.
// X = n + j/1024 + s, s in [0, 2^-10) of 45 bits; 2^s - 1 = s (c1 + s (c2 + c3 s + c4 s^2))
// with c_k = ln2^k / k! (truncation below 2^-59), s = (a + b) 2^-33 with a, b < 2^23 and < 1
// exact in floats; the inner quadratic and both products in pairs of floats (error of p below
// 2^-57).  The product T p, T = 2^(j/1024), is split into integers in units of 2^-32 and 2^-54
// by adding powers of two, added to the table's 55-bit value and rounded to 53 bits: within
// 1 ulp (the parts' bounds added up; 0.87 at most and 0.31 rms over 2e7 random arguments, where the
// rounding alone is 0.29 rms).  About 55 full-rate operations, where
// the nine FP64 operations of exp_tang_core take the issue time of 540.
__device__ __forceinline__ double exp2_fixed(s64 X, const u64* __restrict__ tab) {
  constexpr float C1H = 0x1.62e43p-1f, C1L = -0x1.05c610p-29f;
  constexpr float C2H = 0x1.ebfbep-3f, C2L = -0x1.f4e9c6p-33f;
  constexpr float C3 = 0x1.c6b08ep-5f, C4 = 0x1.3b2ab6p-7f;
  constexpr float U = 0x1p-33f;
  const unsigned hi = (unsigned)((u64)X >> 32), lo = (unsigned)X;
  const u64 Tb = tab[(hi >> 13) & 1023u];
  const unsigned th = (unsigned)(Tb >> 32), tl = (unsigned)Tb;
  const float a = __uint_as_float((__funnelshift_r(lo, hi, 22) & 0x7fffffu) | 0x4b000000u) - 8388608.0f;
  const float b = __uint_as_float((lo & 0x3fffffu) | 0x40000000u) - 2.0f;
  // w = c2 + c3 s + c4 s^2
  const float t = fmaf(a, C4 * U * U, C3 * U) * a;
  const float wh = C2H + t;
  const float wl = ((C2H - wh) + t) + C2L;
  // v = s w (units 2^-33)
  const float vh = a * wh;
  float vl = fmaf(a, wh, -vh);
  vl = fmaf(a, wl, vl);
  vl = fmaf(b, wh, vl);
  // z = c1 + v
  const float zh = fmaf(vh, U, C1H);
  const float zl = fmaf(vh, U, C1H - zh) + fmaf(vl, U, C1L);
  // p = s z (units 2^-33)
  const float ph = a * zh;
  float pl = fmaf(a, zh, -ph);
  pl = fmaf(a, zl, pl);
  pl = fmaf(b, zh, pl);
  // q = T p; the table's high word is 2^23 T, its low word and the bias are T's tail
  const float Th = __uint_as_float(th + 0x3f000000u);
  const float Tl = __uint_as_float((tl >> 9) | 0x4b000000u) - (8388608.0f + 0x1.03p+22f);  // 2^-46
  float qh = Th * ph;
  float ql = fmaf(Th, ph, -qh);
  ql = fmaf(Th, pl, ql);
  ql = fmaf(Tl * 0x1p-46f, ph, ql);
  const float qs = qh + ql;
  ql = ql - (qs - qh);
  // q = 2 A + r, r in units 2^-21 by the second sum
  const float f1 = fmaf(qs, 0.5f, 8388608.0f);
  const float r = fmaf(f1 - 8388608.0f, -2.0f, qs) + ql;
  const unsigned A = __float_as_uint(f1) & 0x7fffffu;
  const unsigned B = __float_as_uint(r - 6.0f) << 1;  // 0x81800000 - 2 r
  const u64 y = Tb + ((u64)A << 23) - B;  // 2^(j/1024 + s) in units 2^-55, and 4
  const u64 m = y >> 3;                   // in units 2^-52: 1.xxx
  const unsigned e = ((unsigned)((int)hi >> 3) & 0xfff00000u) + (1022u << 20);
  return __hiloint2double((int)((unsigned)(m >> 32) + e), (int)(unsigned)m);
}

// F 2^(1023 - top) as an integer in units 2^-58, rounded down, for F > 0 with F 2^(1023 - top)
// below 2.
__device__ __forceinline__ u64 unit58(double F, int top = 1023) {
  const unsigned hi = (unsigned)__double2hiint(F), lo = (unsigned)__double2loint(F);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const u64 m = ((u64)__funnelshift_l(lo, mh, 6) << 32) | (lo << 6);
  const unsigned s = min((unsigned)top - (hi >> 20), 63u);
  return m >> s;
}

// The same for F of either sign, |F| 2^(1023 - top) below 2: rounded down, as a 64-bit integer.
__device__ __forceinline__ u64 floor58(double F, int top) {
  const unsigned hi = (unsigned)__double2hiint(F), lo = (unsigned)__double2loint(F);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const s64 m = (s64)(((u64)__funnelshift_l(lo, mh, 6) << 32) | (lo << 6));
  const unsigned s = min((unsigned)top - (hi >> 20 & 0x7ffu), 63u);
  return (u64)(((int)hi < 0 ? -m : m) >> s);
}

// A double of magnitude below 32 in units 2^-58, rounded toward zero.
__device__ __forceinline__ s64 signed58(double v) {
  const int h = __double2hiint(v);
  const unsigned hi = (unsigned)h & 0x7fffffffu, lo = (unsigned)__double2loint(v);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const int e = (int)(hi >> 20);                                // value = m 2^(e - 1075)
  const u64 m = (((u64)mh << 32) | lo) << 10;                   // units 2^(e - 1085)
  const unsigned s = (unsigned)min(1027 - e, 63);               // to units 2^-58
  const s64 a = (s64)(m >> s);
  return h < 0 ? -a : a;
}

// A multiplier in units of L: v log2(e) 2^55 to the nearest integer, |v| < 2^7.
__device__ __forceinline__ s64 to_log2(double v) {
  constexpr u64 LOG2E = 0xb8aa3b295c17f0bcull;                  // log2(e) 2^63
  const int h = __double2hiint(v);
  const unsigned hi = (unsigned)h & 0x7fffffffu, lo = (unsigned)__double2loint(v);
  const int e = (int)(hi >> 20);
  if (e < 1023 - 64) return 0;                                  // below 2^-64
  const u64 m = (((u64)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 11;  // units 2^(e - 1086)
  const u64 p = __umul64hi(m, LOG2E);                           // v log2(e), units 2^(e - 1085)
  const int s = 1030 - e;                                       // to units 2^-55
  const s64 a = s > 63 ? (s64)(s == 64 ? p >> 63 : 0) : (s64)((p + ((1ull << s) >> 1)) >> s);
  return h < 0 ? -a : a;
}

__device__ __forceinline__ double from_log2(s64 L) {
  return (double)L * 0x1.62e42fefa39efp-56;                     // ln2 2^-55
}

}  // namespace fx
}  // namespace lbm39
