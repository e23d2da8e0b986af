// solve_fx.cuh -- the constraint solve of a cell on the integer and FP32 pipes
// (fixed.cuh): the iteration of newton() -- same starting point, stopping rule,
// polishing step, line search and failure rule -- with its residuals in 64-bit
// fixed point and its direction from an FP32 factorisation.
//
// REFINE (the FP64 path's Newton-Raphson): the direction is refined with the
// residual b - J d of the exact Jacobian-vector product, formed in integers, so
// that it has the FP64 solve's accuracy as far as the iteration can tell: its
// error (about 1e-11 of the step) moves the next residual by less than the
// rounding of a residual in FP64 does, and the updates a cell takes stay the
// same.  Without it the direction is the FP32 one of root finders 2 and 3.
//
// What bounds it: instruction supply and the latency of dependent integer and FP32
// instructions at 12 warps an SM (an IPC of 1.8 of 4; a fifth of the stalls wait for
// instructions, and code that grows by a few thousand instructions costs more than
// it saves; two blocks an SM at 255 registers without spills, and blocks of 64, 192,
// 256 and 384 threads, with and without a barrier in each iteration, measured 2 to
// 15 % slower).  On the 128^3 box at rms Ma 0.5 ten steps with the initialisation take 44.5 ms where the
// FP64 solve took 259.4, on the 256^3 box at rms Ma 0.8 five take 213 where it took 1137.
#pragma once
#include "cell.cuh"
#include "fixed.cuh"

namespace lbm39 {

// v / 2^s to the nearest integer, s > 0.
__device__ __forceinline__ fx::s64 shift_round(fx::s64 v, int s) {
  return s > 62 ? 0 : (v + (fx::s64)((1ull << s) >> 1)) >> s;
}

// log2(e) 2^30 = LOG2E_HI + LOG2E_LO 2^-31
constexpr int LOG2E_HI = 1549082004, LOG2E_LO = 1460010030;

__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }

// Exponent of a normal positive float.
__device__ __forceinline__ int exponent_of(float x) { return (int)(__float_as_uint(x) >> 23) - 127; }

template <int N>
__device__ __forceinline__ fx::u64 max_abs64(const fx::s64 (&v)[N]) {
  fx::u64 r = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const fx::u64 a = (fx::u64)(v[k] < 0 ? -v[k] : v[k]);
    r = a > r ? a : r;
  }
  return r;
}

// v as floats in units of 2^(32 - c), c = clz(max|v|) - 2 (largest magnitude below 2^30),
// each truncated to 24 significant bits.
template <int N>
__device__ __forceinline__ void truncated_floats(const fx::s64 (&v)[N], int c, float (&b)[N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const fx::u64 a = (fx::u64)(v[k] < 0 ? -v[k] : v[k]);
    const int z = __clzll((fx::s64)(a | 1));
    const float f = (float)(int)((a << z) >> 40) * pow2f(8 + c - z);
    b[k] = v[k] < 0 ? -f : f;
  }
}

// The same, truncated to a multiple of the unit.
template <int N>
__device__ __forceinline__ void scaled_floats(const fx::s64 (&v)[N], int c, float (&b)[N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) b[k] = (float)(int)(((fx::u64)v[k] << c) >> 32);
}

// A workspace array whose slots hold 64-bit integers.
template <int BLK>
struct IntView {
  WS<BLK> w;
  __device__ __forceinline__ fx::s64 operator[](int k) const { return __double_as_longlong(w[k]); }
  __device__ __forceinline__ void set(int k, fx::s64 v) const { w[k] = __longlong_as_double(v); }
};

// F as floats truncated to 24 bits (F in [2^-126, 0.75)).
template <int BLK>
struct FloatView {
  WS<BLK> F;
  __device__ __forceinline__ float operator[](int i) const { return view_float(F[i]); }
};

// The direction of J d = G (J = sum_i F_i phi phi^T at the workspace's F, G in units 2^-58 with
// its scaled floats b and their shift c) in units of L.  False where FP32 cannot factor J, or
// where the refinement does not contract.
template <int BLK, bool REFINE, bool D2>
__device__ __forceinline__ bool direction_fx(WS<BLK> F, const fx::s64 (&G)[Sys<D2>::N],
                                             const float (&b)[Sys<D2>::N], int c,
                                             fx::s64 (&dl)[Sys<D2>::N]) {
  constexpr int N = Sys<D2>::N;
  float J[N * (N + 1) / 2], rd[N], d[N];
  {
    float s[N];
    const FloatView<BLK> Ff{F};
    if constexpr (D2) gen::moments2d<float>(Ff, s, J);
    else gen::moments<float>(Ff, s, J);
  }
  if (!ldlt_factor<float, N>(J, rd)) return false;
#pragma unroll
  for (int k = 0; k < N; ++k) d[k] = b[k];
  ldlt_apply<float, N>(J, rd, d);
  const float mx = max_abs(d);
  if (mx == 0.0f) {
#pragma unroll
    for (int k = 0; k < N; ++k) dl[k] = 0;
    return true;
  }
  if (!(mx > 0x1p16f && mx < 0x1p80f)) return false;
  const int eb = exponent_of(mx);
  if constexpr (!REFINE) {
    // each component exactly: d = D 2^(e - 23), dl = D log2(e) 2^(e - 23 + 32 - c - 58 + 55)
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const unsigned u = __float_as_uint(d[k]);
      const int D = (int)((u & 0x7fffffu) | 0x800000u);
      const int s = c + 32 - ((int)(u >> 23 & 0xff) - 127);
      const fx::s64 v = shift_round((fx::s64)D * LOG2E_HI * 256 + (((fx::s64)D * LOG2E_LO) >> 23), max(s, 1));
      dl[k] = (int)u < 0 ? -v : v;
      if (s < 1) return false;
    }
    return true;
  } else {
    // the FP32 direction rounded to integers D of 21 bits: d = D 2^g
    const float scale = pow2f(20 - eb);
    const int g = eb - 46 - c;
    const int s = -(g + 17);
    if (s <= 0) return false;
    int Dk[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
      Dk[k] = (int)(__float_as_uint(fmaf(d[k], scale, 12582912.0f)) - 0x4b400000u);
    // J d by y_i = phi(xi_i) . D (exact) and sum_i F_i y_i phi, in units 2^(g - 26)
    fx::u64 Jd[N];
    const auto prod = [&](auto I, int y) -> fx::u64 {
      constexpr int i = decltype(I)::value;
      const fx::u64 q = fx::unit58(F[i]);
      const int qh = (int)(q >> 32), ql = (int)((unsigned)q >> 1);
      return (fx::u64)((fx::s64)qh * y + (((fx::s64)ql * y) >> 31));
    };
    if constexpr (D2) gen::jvec_fx2d(Dk, prod, Jd);
    else gen::jvec_fx(Dk, prod, Jd);
    fx::s64 r[N];
    const int q = -32 - g;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const fx::s64 Gs = q >= 0 ? (fx::s64)((fx::u64)G[k] << q) : G[k] >> min(-q, 63);
      r[k] = (fx::s64)((fx::u64)Gs - Jd[k]);
      // D log2(e) 2^38, then in units of L
      dl[k] = shift_round((fx::s64)Dk[k] * LOG2E_HI * 256 + (((fx::s64)Dk[k] * LOG2E_LO) >> 23), s);
    }
    const fx::u64 rq = max_abs64(r);
    if (rq == 0) return true;
    const int c1 = __clzll((fx::s64)rq) - 2;
    if (c1 < 0) return false;
    scaled_floats(r, c1, d);
    ldlt_apply<float, N>(J, rd, d);
    const float m1 = max_abs(d);
    if (m1 == 0.0f) return true;
    if (!(m1 > 0x1p-40f && m1 < 0x1p80f)) return false;
    const int e1 = exponent_of(m1);
    if (e1 + 6 - c1 > 20 - 8) return false;  // the correction is over 2^-8 of the step
    const int s1 = -(e1 + 11 - c1 + g);
    if (s1 <= 0) return false;
    const float scale1 = pow2f(20 - e1);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int D1 = (int)(__float_as_uint(fmaf(d[k], scale1, 12582912.0f)) - 0x4b400000u);
      dl[k] += shift_round((fx::s64)D1 * LOG2E_HI, s1);
    }
    return true;
  }
}

// True where every |L_k| is below 64, 16, 4 and 1 (as numbers) for the multipliers of order 0 to
// 3: no exponent then reaches 208.
template <class A>
__device__ __forceinline__ bool multipliers_in_range(const A& l) {
  unsigned bad = 0;
#pragma unroll
  for (int k = 0; k < NM; ++k) {
    const int bits = k == 0 ? 61 : k < 4 ? 59 : k < 10 ? 57 : 55;
    const unsigned h = (unsigned)((fx::u64)l[k].v >> 32) + (1u << (bits - 32));
    bad |= h >> (bits - 31);
  }
  return bad == 0;
}

// The multipliers at src (doubles, `stride` apart) into units of L in the workspace; false outside
// its range.
template <int BLK>
__device__ __forceinline__ bool multipliers_to_log2(const double* src, long long stride,
                                                    WS<BLK> lam) {
  const IntView<BLK> L{lam};
#pragma unroll
  for (int k = 0; k < NM; ++k) lam[k] = src[k * stride];
  int top = 0;
#pragma unroll 1
  for (int k = 0; k < NM; ++k) {
    const double v = lam[k];
    top = max(top, __double2hiint(v) & 0x7fffffff);
    L.set(k, fx::to_log2(v));
  }
  return top < ((1023 + 6) << 20);
}

// The solve (see newton() for the iteration).  In: the multipliers at src (`stride` apart: the
// workspace's, or the stored state, which a solve that takes no update then does not read), w's
// targets, and with cached its F at the multipliers.  Out: true with the result, w's F (the targets
// are overwritten) and, where `moved`, its multipliers, else neither has changed; false where a
// value leaves the fixed-point ranges or FP32 cannot give a direction: the caller restores the
// workspace and solves in FP64.
template <int BLK, bool REFINE, bool D2>
__device__ __forceinline__ bool newton_fx(WS<BLK> w, const double* src, long long stride,
                                          const Phys& ph, int maxit, bool cached,
                                          NewtonResult& out, bool& moved) {
  using S = Sys<D2>;
  constexpr int N = S::N;
  WS<BLK> F = w.at(WS_E), lam = w.at(WS_LAM), m = w.at(WS_M);
  const IntView<BLK> X{F}, L{lam}, M{m};
  int top = 0;
#pragma unroll
  for (int k = 0; k < NM; ++k) {
    const double v = m[k];
    top = max(top, __double2hiint(v) & 0x7fffffff);
    // rounding the 24 populations with |xi|^2 >= 4 down takes half a unit from each on average
    const int half = k == 0 ? 12 : k >= 4 && k <= 6 ? 29 : 0;
    M.set(k, fx::signed58(v) - half);
  }
  if (top >= (1023 + 4) << 20) return false;  // |m| >= 16, inf, NaN
  bool have_L = false;
  if (!cached) {
    if (!multipliers_to_log2<BLK>(src, stride, lam)) return false;
    have_L = true;
  }
  int n = 0, failed = 0, ls = 0, c0 = 0;
  int sh = -1;  // trial point L - dl 2^-sh (negative: L itself)
  bool first = true, polished = false, restore = false;
  float s0 = 0.0f;
  fx::s64 dl[N];
  for (;;) {
    unsigned fmax = 0, fmin = ~0u;
    if (first && cached) {
#pragma unroll 1
      for (int i = 0; i < Q; ++i) {
        if (!D2 || ((kZOwn >> i) & 1ull)) {
          const double v = F[i];
          fmax = max(fmax, (unsigned)__double2hiint(v));
          fmin = min(fmin, (unsigned)__double2hiint(v));
        }
      }
    } else {
      fx::I64 l[NM], x[Q];
#pragma unroll
      for (int k = 0; k < NM; ++k) l[k] = fx::I64(L[k]);
      if (sh >= 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) l[S::idx(k)] = l[S::idx(k)] - fx::I64(dl[k] >> sh);
      }
      if (!multipliers_in_range(l)) return false;
      if constexpr (D2) gen::exponents2d(l, x);
      else gen::exponents(l, x);
#pragma unroll
      for (int i = 0; i < Q; ++i) X.set(i, x[i].v);
      const fx::u64* tab = fx::table();
      // three exponentials at a time from the workspace: a loop that the nearest instruction cache
      // holds, in a kernel whose straight-line code does not fit (one at a time: 1 % slower)
#pragma unroll 3
      for (int i = 0; i < Q; ++i) {
        if (!D2 || ((kZOwn >> i) & 1ull)) {
          const double v = fx::exp2_fixed(X[i], tab);
          F[i] = v;
          fmax = max(fmax, (unsigned)__double2hiint(v));
          fmin = min(fmin, (unsigned)__double2hiint(v));
        }
      }
      if constexpr (D2) {
        static_for<0, Q>([&](auto I) {
          constexpr int i = decltype(I)::value;
          if constexpr (zmirror(i) < i) F[i] = F[zmirror(i)];
        });
      }
    }
    fx::s64 G[N];
    bool reject = false;
    {
      fx::u64 s[N];
      const auto val = [&](auto I) { return fx::unit58(F[decltype(I)::value]); };
      if constexpr (D2) gen::sums_fx2d(val, s);
      else gen::sums_fx(val, s);
      // F_i in [2^-126, 0.75): sum F_i is below 30 and has not wrapped; below 3.5, sum F_i |xi|^2
      // has not either; and that below 10.6, no sum reaches 32
      constexpr int E = D2 ? 3 : 4;  // the sums of xi_x^2, xi_y^2, xi_z^2 are E, E + 1, E + 2
      constexpr unsigned E2MAX = (unsigned)(10.6 * (1 << 25));
      const unsigned e2 = ((unsigned)(s[E] >> 32) >> 1) + ((unsigned)(s[E + 1] >> 32) >> 1) +
                          ((unsigned)(s[E + 2] >> 32) >> 1);
      const bool mass = (unsigned)(s[0] >> 32) > (7u << 25);
      if (fmax >= 0x3fe80000u || fmin < (897u << 20) || mass || e2 > E2MAX) {
        // a trial point far out is rejected where its residual, from the sums of F_i and
        // F_i |xi_i|^2 in FP32, is surely above that of the last accepted one
        if (first || polished || restore) return false;
        float s0f = -1.0f, s2f = -0x1p-58f * ((float)M[4] + (float)M[5] + (float)M[6]);
#pragma unroll 1
        for (int i = 0; i < Q; ++i) {
          const float f = trunc_float(F[i]);
          s0f += f;
          s2f = fmaf((float)(kCX[i] * kCX[i] + kCY[i] * kCY[i] + kCZ[i] * kCZ[i]), f, s2f);
        }
        if (!(s0 * pow2f(max(-52 - 2 * c0, -126)) < 0.9f * (s0f * s0f + s2f * s2f * (1.0f / 3.0f))))
          return false;
        reject = true;
      }
#pragma unroll
      for (int k = 0; k < N; ++k) G[k] = (fx::s64)s[k] - M[S::idx(k)];
    }
    if (restore) break;  // F is back at the last accepted L after a failed line search
    fx::u64 rq = 0;
    int c = 0;
    float b[N], ssq = 0.0f;
    if (!reject) {
      rq = max_abs64(G);
      c = __clzll((fx::s64)(rq | 1)) - 2;
      if (c < 0) return false;
      // root finders 2 and 3 take their right-hand side in single precision
      if constexpr (REFINE) scaled_floats(G, c, b);
      else truncated_floats(G, c, b);
#pragma unroll
      for (int k = 0; k < N; ++k) ssq = fmaf(b[k], b[k], ssq);
      if (!first && !polished) {
        const float thr = s0 * pow2f(min(max(2 * (c - c0), -126), 60));
        if (fabsf(ssq - thr) <= 1e-5f * thr) return false;  // undecided in FP32
        reject = !(ssq < thr);
      }
    }
    if (reject) {  // halve the step
      if (++ls > LS_MAX) {
        failed = 1;
        restore = true;
        sh = -1;
        continue;
      }
      ++sh;
      continue;
    }
    // accept the trial point
    if (sh >= 0) {
#pragma unroll
      for (int k = 0; k < N; ++k) L.set(S::idx(k), L[S::idx(k)] - (dl[k] >> sh));
    }
    if (!first) ++n;
    first = false;
    if (n >= ph.min_upd && rq < ph.tol_fx && (rq < ph.tol_fx100 || polished)) break;
    if (n >= maxit) { failed = 1; break; }
    s0 = ssq;
    c0 = c;
    if (!have_L) {
      if (!multipliers_to_log2<BLK>(src, stride, lam)) return false;
      have_L = true;
    }
    if (!direction_fx<BLK, REFINE, D2>(F, G, b, c, dl)) return false;
    polished = rq < ph.tol_fx;
    sh = 0;
    ls = 0;
  }
  if (have_L) {
#pragma unroll 1
    for (int k = 0; k < NM; ++k) lam[k] = fx::from_log2(L[k]);
  }
  moved = have_L;
  out = NewtonResult{n, failed};
  return true;
}

// The Gaussian start of gaussian_guess, its normalising sum with the fixed-point exponential: CUDA's
// FP64 exp, 39 times a cell, was a third of an initialisation (a 128^3 box's pass of ten steps went
// from 48.8 to 45.9 ms).  False outside the range.
template <int BLK>
__device__ __forceinline__ bool gaussian_guess_fx(double ux, double uy, double uz, double T,
                                                  WS<BLK> w) {
  WS<BLK> F = w.at(WS_E), lam = w.at(WS_LAM);
  const IntView<BLK> X{F};
  const double it = 1.0 / T;
  double top = fmax(fabs(it), fmax(fabs(ux * it), fmax(fabs(uy * it), fabs(uz * it))));
  if (!(top < 16.0)) return false;
  lam[1] = ux * it; lam[2] = uy * it; lam[3] = uz * it;
  lam[4] = lam[5] = lam[6] = -0.5 * it;
#pragma unroll
  for (int k = 7; k < NM; ++k) lam[k] = 0.0;
  fx::I64 l[NM], x[Q];
#pragma unroll
  for (int k = 0; k < NM; ++k) l[k] = fx::I64(k >= 1 && k <= 6 ? fx::to_log2(lam[k]) : 0);
  if (!multipliers_in_range(l)) return false;
  gen::exponents(l, x);
#pragma unroll
  for (int i = 0; i < Q; ++i) X.set(i, x[i].v);
  const fx::u64* tab = fx::table();
  double s = 0.0;
#pragma unroll 3
  for (int i = 0; i < Q; ++i) s += fx::exp2_fixed(X[i], tab);
  lam[0] = -log(s);
  return true;
}

}  // namespace lbm39
