// The solver's device arithmetic compiled for the host: CUDA's keywords and
// the intrinsics it uses, then the headers, then C entry points for ctypes.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __constant__
#define __shared__ static
#define __forceinline__ inline
#define __noinline__
#define __restrict__
#define __syncthreads()
using std::exp;
using std::fabs;
using std::fma;
using std::log;
using std::max;
using std::min;
template <class A, class B>
static inline A bits(B b) {
  static_assert(sizeof(A) == sizeof(B), "size");
  A a;
  std::memcpy(&a, &b, sizeof a);
  return a;
}
typedef unsigned long long ull;
static struct { int x; } threadIdx = {0}, blockDim = {1};
static inline float __uint_as_float(unsigned u) { return bits<float>(u); }
static inline unsigned __float_as_uint(float f) { return bits<unsigned>(f); }
static inline int __double2hiint(double d) { return (int)(bits<ull>(d) >> 32); }
static inline int __double2loint(double d) { return (int)bits<ull>(d); }
static inline double __hiloint2double(int h, int l) {
  return bits<double>(((ull)(unsigned)h << 32) | (unsigned)l);
}
static inline long long __double_as_longlong(double d) { return bits<long long>(d); }
static inline double __longlong_as_double(long long v) { return bits<double>(v); }
static inline float __double2float_rn(double d) { return (float)d; }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, int s) {
  return (unsigned)(((((ull)hi << 32) | lo) << (s & 31)) >> 32);
}
static inline unsigned __funnelshift_r(unsigned lo, unsigned hi, int s) {
  return (unsigned)((((ull)hi << 32) | lo) >> (s & 31));
}
static inline ull __umul64hi(ull a, ull b) { return (ull)(((unsigned __int128)a * b) >> 64); }
static inline int __float2int_rn(float f) { return (int)std::lrint(f); }
static inline int __clzll(long long x) { return x ? __builtin_clzll((ull)x) : 64; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline float __fmul_rn(float a, float b) { return a * b; }

#include "../paper_1910_13515_gb300/csrc/solve_fx.cuh"

using namespace lbm39;

template <bool REFINE, bool D2>
static int solve(double* ws, const Phys& ph, int maxit, int cached, int fixed, int* out) {
  WS<1> w{ws};
  NewtonResult r{-1, -1};
  if (fixed) {
    bool moved;
    if (!newton_fx<1, REFINE, D2>(w, ws + WS_LAM, 1, ph, maxit, cached != 0, r, moved)) return 0;
    out[2] = moved;
  } else {
    r = newton<1, !REFINE, D2>(w, ph.tol, ph.min_upd, maxit, cached != 0);
  }
  out[0] = r.n_upd;
  out[1] = r.failed;
  return 1;
}

extern "C" {

void fx_exp2(const long long* X, double* y, long long n) {
  fx::load_table();
  for (long long i = 0; i < n; ++i) y[i] = fx::exp2_fixed(X[i], fx::table());
}

void fx_convert(const double* F, ull* u58, const double* v, long long* s58, const double* l,
                long long* L, double* back, long long n) {
  for (long long i = 0; i < n; ++i) {
    u58[i] = fx::unit58(F[i]);
    s58[i] = fx::signed58(v[i]);
    L[i] = fx::to_log2(l[i]);
    back[i] = fx::from_log2(L[i]);
  }
}

// One cell: ws (WS_DOUBLES_FX) = F (39, library order), lam (13), m (13) in; F, lam out.  Returns 0 where the
// fixed-point solve gives the cell up.
int fx_solve(double* ws, int refine, int d2, int fixed, int cached, double tol, int maxit,
             int* out) {
  fx::load_table();
  Phys ph{};
  ph.tol = tol;
  ph.tol_fx = (ull)std::ceil(tol * 0x1p58);
  ph.tol_fx100 = (ull)std::ceil(1e-2 * tol * 0x1p58);
  if (refine) return d2 ? solve<true, true>(ws, ph, maxit, cached, fixed, out)
                        : solve<true, false>(ws, ph, maxit, cached, fixed, out);
  return d2 ? solve<false, true>(ws, ph, maxit, cached, fixed, out)
            : solve<false, false>(ws, ph, maxit, cached, fixed, out);
}

void velocities(int* v) {
  for (int i = 0; i < Q; ++i) v[3 * i] = CX[i], v[3 * i + 1] = CY[i], v[3 * i + 2] = CZ[i];
}

}  // extern "C"
