// kernels.cuh -- CUDA kernels of the D3Q39 DDF step: initial equilibrium, the
// fused collide-and-stream passes (AA pattern), boundary fills, macroscopic
// read-out and conserved sums.
//
// Storage: 78 planes of Np elements (f_0..f_38 then g_0..g_38), x fastest,
// of type P: double (FP64 path) or float (precision form: each population
// stored as its deviation from a reference population h_ref, Desc::href).
// AA pattern over one buffer.  At even time the buffer holds the
// pre-collision populations h_i(x) in slot (x, i).  The even pass reads its
// own slots, collides and writes h*_i(x) into slot (x, opp i).  The odd pass
// gathers h_i(x) = h*_i(x - xi_i) from slot (x - xi_i, opp i), collides and
// pushes h*_i(x) into slot (x + xi_i, i), which is the pre-collision h_i of
// the next time step.  Every slot is read and written by one thread only (the
// slot pushed for direction i is the one gathered for opp(i)).  Solid,
// freestream and outflow cells never collide.  After each pass the fill
// kernels write into the slots of those cells (and, after an odd pass, of
// their fluid neighbours) what the fluid cells read next: the half-way
// bounce-back copies of solid cells and what freestream and outflow cells
// would have streamed (Sec. 4 boundary kinds), so the step kernels treat
// every neighbour alike.
//
// A fluid cell's step runs in three phases: gather and moments; targets and
// Newton (F, lam, m in shared memory); gather again, sensor, BGK and push.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "cell.cuh"
#include "launch.cuh"
#include "plane.cuh"
#include "solve_fx.cuh"

namespace lbm39 {

// Cells of one warp: 32 w + the bits that are set.
struct Rest {
  unsigned w, bits;
};

struct Desc {
  void* pop;                          // 78 planes of P
  double* lam;                        // 13 planes of multipliers kept between steps, then
                                      // 39 planes of F_i = exp(Phi lam) at them
  Rest* rest;                         // the cells that a fixed-point kernel leaves to its FP64
                                      // kernel (k_step_fp64, k_init_fp64)
  const uint8_t* mask;                // nullptr: every cell fluid, all axes periodic
  unsigned long long* ctr;            // counters (CTR_*)
  const void* free_store;             // 78 stored values (P) of a freestream cell
  const double* heq_inf;              // 78 far-field equilibrium populations (FP64)
  const double* href;                 // 78 reference populations (precision form)
  double mref[5];                     // sum of href: rho, j, sum f|xi|^2 + sum g
  long long N, Np;                    // cells, plane stride in elements
  long long t;                        // time step being taken (schedules fallback retries)
  int d2;                             // one cell thick in z, z-mirror-symmetric populations
  int nx, ny, nz;
  int per[3];                         // periodic axes
  Phys ph;
};

// CTR_UPD32: float steps of single-precision starts; CTR_START32: solves that took one.
enum {
  CTR_FAILED = 0, CTR_UPDATES = 1, CTR_HIST = 2, CTR_EPS = 34, CTR_UPD32 = 38, CTR_START32 = 39,
  CTR_N = 40
};
// Set by lbm39_init when some fluid cell starts with u_z != 0 (outside the
// block counters: not reported by lbm39_stats).
constexpr int CTR_ASYM = 42;
// Lengths of the lists of cells left to the FP64 kernels, also outside the block counters: steps at
// even and odd times, then alternate ranges of an initialisation.  A list's length is zero before
// its fixed-point kernel, since the FP64 kernel that follows one list clears the other of its pair.
// CTR_TAKEN: the entries of each that the FP64 kernel's warps took beyond their first.
constexpr int CTR_REST = 44, CTR_TAKEN = 48;

struct Coord {
  int x, y, z;
};

// (cell < 2^31: lattices are limited to 2^31 - 1 cells)
__device__ __forceinline__ Coord coord_of(const Desc& d, long long cell) {
  const int c = (int)cell;
  const int yz = c / d.nx;
  return Coord{c - yz * d.nx, yz % d.ny, yz / d.ny};
}

// a mod n for a in [-3, n + 2]: one conditional correction when n >= 3, the last bit or 0 below.
// (Written with the remainder operator, the 21 wraps of a neighbour table were 2000 instructions
// in each of the odd pass's two tables, a third of the kernel.)
__device__ __forceinline__ int wrap(int a, int n) {
  const int add = n >= 3 ? n : 0, mask = n >= 3 ? -1 : n - 1;
  return (a + (a < 0 ? add : 0) - (a >= n ? add : 0)) & mask;
}

// Index of the cell at x + (dx, dy, dz) with periodic wrap of every axis
// (non-periodic axes carry boundary layers, so fluid cells never wrap there).
// Every index is below 2^31, so the 21 terms are 32-bit.
struct Nbr {
  int xs[7], ys[7], zs[7];
  __device__ __forceinline__ Nbr() {}
  __device__ __forceinline__ Nbr(const Desc& d, Coord c) {
#pragma unroll
    for (int s = 0; s < 7; ++s) {
      xs[s] = wrap(c.x + s - 3, d.nx);
      ys[s] = wrap(c.y + s - 3, d.ny) * d.nx;
      zs[s] = wrap(c.z + s - 3, d.nz) * d.nx * d.ny;
    }
  }
  __device__ __forceinline__ int at(int dx, int dy, int dz) const {
    return xs[dx + 3] + ys[dy + 3] + zs[dz + 3];
  }
};

// The neighbour table of the cell at c, built from a copy of the coordinates
// that the compiler cannot see through: a table built before the constraint
// solve is then not kept in registers across it (the odd pass builds it twice).
template <bool ODD>
__device__ __forceinline__ Nbr fresh_nbr(const Desc& d, Coord c) {
  Nbr nb;
  if constexpr (ODD) {
    asm volatile("" : "+r"(c.x), "+r"(c.y), "+r"(c.z));
    nb = Nbr(d, c);
  }
  return nb;
}

// Pre-collision populations of one distribution (base 0: f, Q: g) of fluid
// cell `cell` at the lattice's current time: own slots at even time, the odd
// gather from (x - xi_i, slot opp i) at odd time.  Where x - xi_i is solid,
// that slot holds the bounced population (bounce_even_cell), so the gather
// has no per-direction branch.
// D2 (the z-mirror-symmetric lattices): one of each mirror pair is read; they
// are equal bit for bit.
template <bool ODD, class P, bool D2 = false>
__device__ __forceinline__ void gather(const Desc& d, long long cell, const Nbr& nb, int base,
                                       P (&h)[Q]) {
  const P* __restrict__ pop = static_cast<const P*>(d.pop);
  static_for<0, Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (D2 && zmirror(i) < i) {
      h[i] = h[zmirror(i)];
    } else if constexpr (!ODD) {
      h[i] = at(pop + (long long)(base + i) * d.Np, (int)cell);
    } else {
      constexpr int cx = CX[i], cy = CY[i], cz = CZ[i];
      h[i] = at(pop + (long long)(base + opp(i)) * d.Np, nb.at(-cx, -cy, -cz));
    }
  });
}

// Post-collision population h*_i of fluid cell `cell` into its AA slot: own
// slot opp i at even time, (x + xi_i, slot i) at odd time (a solid x + xi_i
// hands it back to x afterwards: bounce_odd_cell).
template <bool ODD, class P, int i>
__device__ __forceinline__ void push(const Desc& d, long long cell, const Nbr& nb, int base,
                                     P v) {
  P* __restrict__ pop = static_cast<P*>(d.pop);
  if constexpr (!ODD) {
    at(pop + (long long)(base + opp(i)) * d.Np, (int)cell) = v;
  } else {
    constexpr int cx = CX[i], cy = CY[i], cz = CZ[i];
    at(pop + (long long)(base + i) * d.Np, nb.at(cx, cy, cz)) = v;
  }
}

// push() of v and, on a z-mirror-symmetric lattice (D2), of the mirrored population, which has
// the same value; i is the first of its pair.
template <bool ODD, class P, int i, bool D2>
__device__ __forceinline__ void push_pair(const Desc& d, long long cell, const Nbr& nb, int base,
                                          P v) {
  push<ODD, P, i>(d, cell, nb, base, v);
  if constexpr (D2 && zmirror(i) != i) push<ODD, P, zmirror(i)>(d, cell, nb, base, v);
}

// The smallest j >= 0 with c_g <= 2.5 2^j: g_i = c_g T f_i divided by 2^j stays in the range that the
// integer sums give the g_i up to T = 0.8 (in most cells beyond), and at c_g = 2 (gamma = 1.4) has the
// unit of the f_i.
inline int g_shift(double cg) {
  return cg > 2.5 ? std::ilogb(std::nextafter(cg / 2.5, 0.0)) + 1 : 0;
}

// Raw moments of a cell: rho, j = rho u, e2 = sum f|xi|^2 + sum g = 2 rho E.
struct Raw {
  double rho, jx, jy, jz, e2;
};

// Phase A: gather each distribution in turn and take the moments (FP64).
template <bool ODD, class P, bool D2 = false>
__device__ __forceinline__ Raw gather_raw(const Desc& d, long long cell, const Nbr& nb) {
  Raw r;
  double gs;
  if constexpr (sizeof(P) == 8) {
    P h[Q];
    gather<ODD, P, D2>(d, cell, nb, 0, h);
    gen::f_moments<double>(h, r.rho, r.jx, r.jy, r.jz, r.e2);
    gather<ODD, P, D2>(d, cell, nb, Q, h);
    gs = gen::g_sum<double>(h);
  } else {  // deviations: moments of h_ref (precomputed) plus those of the deviations
    P h[Q];
    double hd[Q];
    gather<ODD, P>(d, cell, nb, 0, h);
#pragma unroll
    for (int i = 0; i < Q; ++i) hd[i] = (double)h[i];
    gen::f_moments<double>(hd, r.rho, r.jx, r.jy, r.jz, r.e2);
    gather<ODD, P>(d, cell, nb, Q, h);
#pragma unroll
    for (int i = 0; i < Q; ++i) hd[i] = (double)h[i];
    gs = gen::g_sum<double>(hd);
    r.rho += d.mref[0]; r.jx += d.mref[1]; r.jy += d.mref[2]; r.jz += d.mref[3];
    gs += d.mref[4];
  }
  r.e2 += gs;
  return r;
}

template <bool ODD, class P>
__device__ __forceinline__ Macro gather_moments(const Desc& d, long long cell, const Nbr& nb) {
  const Raw r = gather_raw<ODD, P>(d, cell, nb);
  return macro_from_moments(r.rho, r.jx, r.jy, r.jz, r.e2, d.ph.inv_2cv);
}

// gather_moments out of line.
template <bool ODD, bool D2>
__device__ __noinline__ void gather_moments_fp64(const void* pop, long long Np, long long cell,
                                                 const Nbr* nb, double inv_2cv, Macro* M) {
  Desc d;
  d.pop = const_cast<void*>(pop);
  d.Np = Np;
  const Raw r = gather_raw<ODD, double, D2>(d, cell, *nb);
  *M = macro_from_moments(r.rho, r.jx, r.jy, r.jz, r.e2, inv_2cv);
}

// The sum of the g_i of a cell in units 2^(-58 - kg), with the scale kg at which the largest |g_i| is
// in [0.25, 0.5), or k if that is smaller; out of line.  False for infinities and NaN.
template <bool ODD, bool D2>
__device__ __noinline__ bool g_sum_again(const void* pop, long long Np, long long cell,
                                         const Nbr* nb, int k, fx::u64* gs, int* kg) {
  Desc d;
  d.pop = const_cast<void*>(pop);
  d.Np = Np;
  double g[Q];
  gather<ODD, double, D2>(d, cell, *nb, Q, g);
  unsigned gmax = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i)
    gmax = max(gmax, (unsigned)__double2hiint(g[i]) & 0x7fffffffu);
  if (gmax > (2000u << 20)) return false;
  const int scale = min(1021 - (int)(gmax >> 20), k);
  fx::u64 sum = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) sum += fx::floor58(g[i], 1023 - scale);
  *gs = sum;
  *kg = scale;
  return true;
}

// The macroscopic variables of a cell with the sums formed in 64-bit integers, for the lattices one
// cell thick in z and for the comparison model: 158 FP64 additions less, each of which takes the
// issue time of 60 FP32 operations.  D2: of a z-mirror-symmetric lattice, with one of each mirror
// pair read (28 % less) and the same values.
// The f_i are scaled by the power of two that brings the largest into [0.25, 0.5) and rounded down
// to units of 2^-58 (about 2^-56 of the density; the largest are exact); the sums are exact.
// Rounding down takes half a unit from each of the 24 populations with |xi_i|^2 >= 4 on average,
// which is given back.  The g_i = c_g T f_i have the scale of the f_i divided by the power of two of
// c_g.  SIGNED (the comparison model): with populations of either sign, which its polynomials give
// from Ma 0.6 on; where there is a negative one, two bits fewer leave room for the sums; and where a
// g_i is beyond the scale, the g_i are read again with that of their largest.  Else such a cell is
// summed in FP64 (the reduced kernel grew by 1.5 % in time with the second reading), as is one whose
// sums leave the ranges.
// (With FP64 sums for the cells that have negative f_i, or g_i above the scale of the f_i, 20 steps of
// the comparison model on 1024 x 1024 took 19.6 ms at gamma 1.2 and 19.4 at rms Ma 1; now 14.8, as at
// gamma 1.4 and Ma 0.3, and 18.6 with FP64 sums for all cells.)
// On the 1024 x 512 airfoil (few solver updates) a step takes 261 us with these sums and 318 with
// FP64 ones.  The other 3-D lattices keep FP64 sums: their kernel, with the 13-multiplier solve, is
// bound by instruction fetches, and the longer code took a step of a 128^3 box from 4.2 to 4.5 ms.
// f: the gathered f_i, for the caller.
template <bool ODD, bool D2, bool SIGNED = false>
__device__ __forceinline__ Macro gather_moments_fx(const Desc& d, long long cell, const Nbr& nb,
                                                   double (&f)[Q]) {
  constexpr int NS = D2 ? 4 : 5;
  constexpr unsigned ABS = SIGNED ? 0x7fffffffu : 0xffffffffu;
  const auto units = [](double v, int k) {
    if constexpr (SIGNED) return fx::floor58(v, 1023 - k);
    else return fx::unit58(v, 1023 - k);
  };
  fx::u64 s[NS], gs = 0;
  unsigned fmax = 0, fneg = 0;
  gather<ODD, double, D2>(d, cell, nb, 0, f);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    fmax = max(fmax, (unsigned)__double2hiint(f[i]) & ABS);
    fneg |= (unsigned)__double2hiint(f[i]);
  }
  const bool neg = SIGNED && (int)fneg < 0;
  // neg: |f_i| < 1/8, so that sum |f_i| |xi_i|^2 <= 204/8 < 32
  const int k = 1021 - (int)(fmax >> 20) - (neg ? 2 : 0);
  const auto val = [&](auto I) { return units(f[decltype(I)::value], k); };
  if constexpr (D2) gen::macro_fx2d(val, s);
  else gen::macro_fx(val, s);
  int kg = k - d.ph.g_shift;
  bool again, out = false;
  {
    double g[Q];
    unsigned gmax = 0, gneg = 0;
    gather<ODD, double, D2>(d, cell, nb, Q, g);
    static_for<0, Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      if constexpr (!D2 || zmirror(i) >= i) {
        gmax = max(gmax, (unsigned)__double2hiint(g[i]) & ABS);
        gneg |= (unsigned)__double2hiint(g[i]);
        const fx::u64 u = units(g[i], kg);
        gs += D2 && zmirror(i) != i ? 2 * u : u;
      }
    });
    // beyond the scale (neg: |g_i| < 1/4, else g_i < 1), NaN, or negative on its own
    again = gmax >= (unsigned)((neg ? 1021 : 1023) - kg) << 20 || (SIGNED && !neg && (int)gneg < 0);
  }
  if constexpr (SIGNED) {
    if (again) {
      const Nbr here = nb;
      out = !g_sum_again<ODD, D2>(d.pop, d.Np, cell, &here, k, &gs, &kg);
    }
  } else {
    out = again;
  }
  constexpr int E = NS - 1;
  // without neg: f_i < 0.5 and sum f < 7, so sum f |xi|^2 < 63; g_i < 1, so sum g < 39.  With neg or
  // again |sum g| < 20
  const bool one = !neg && !again && kg == k;  // the energy is one sum
  if (fmax - (100u << 20) > (1900u << 20) || out ||
      (!neg && (unsigned)(s[0] >> 32) > (7u << 26)) ||
      (one && ((unsigned)(s[E] >> 32) >> 1) + ((unsigned)(gs >> 32) >> 1) > (60u << 25))) {
    const Nbr here = nb;
    Macro M;
    gather_moments_fp64<ODD, D2>(d.pop, d.Np, cell, &here, d.ph.inv_2cv, &M);
    return M;
  }
  // products that are not contracted into the sums that follow: both systems round alike
  const double sc = __hiloint2double((1023 - 58 - k) << 20, 0);
  const auto value = [&](fx::u64 v) { return gen::mul_rn((double)(fx::s64)v, sc); };
  double jz = 0.0, e2;
  if constexpr (!D2) jz = value(s[3]);
  if (one) {
    e2 = gen::mul_rn((double)(s[E] + gs + 87 + 12), sc);
  } else {
    const fx::u64 e = s[E] + 87, g = gs + 12;
    e2 = gen::mul_rn(neg ? (double)(fx::s64)e : (double)e, sc) +
         gen::mul_rn(neg || again ? (double)(fx::s64)g : (double)g,
                     __hiloint2double((1023 - 58 - kg) << 20, 0));
  }
  return macro_from_moments(value(s[0] + 12), value(s[1]), value(s[2]), jz, e2, d.ph.inv_2cv);
}

// The same out of line, for the full system on such lattices.
template <bool ODD>
__device__ __noinline__ void gather_moments_thin(const void* pop, long long Np, long long cell,
                                                 const Nbr* nb, double inv_2cv, int g_shift,
                                                 Macro* M) {
  Desc d;
  d.pop = const_cast<void*>(pop);
  d.Np = Np;
  d.ph.inv_2cv = inv_2cv;
  d.ph.g_shift = g_shift;
  double f[Q];
  *M = gather_moments_fx<ODD, false>(d, cell, *nb, f);
}

// The macroscopic variables as the step of a fixed-point kernel forms them.
template <bool ODD, bool D2>
__device__ __forceinline__ Macro step_moments(const Desc& d, long long cell, const Nbr& nb) {
  if constexpr (D2) {
    double f[Q];
    return gather_moments_fx<ODD, true>(d, cell, nb, f);
  }
  if (d.nz != 1) return gather_moments<ODD, double>(d, cell, nb);
  const Nbr here = nb;
  Macro M;
  gather_moments_thin<ODD>(d.pop, d.Np, cell, &here, d.ph.inv_2cv, d.ph.g_shift, &M);
  return M;
}

// 39 eps in FP64 from the populations at f, where the FP32 screen cannot decide: not inlined, as
// few cells take it (its divisions are a seventh of the step kernel's code otherwise).
template <int BLK>
__device__ __noinline__ double sensor_sum_fp64(const double* f, double rho, WS<BLK> F) {
  double s = 0.0;
#pragma unroll 1
  for (int i = 0; i < Q; ++i) {
    const double feq = rho * F[i];
    s += fabs(f[i] - feq) / feq;
  }
  return s;
}

// Phase C: gather again, Knudsen sensor (Eq. DeltaAvg, f only), tau_eff =
// tau alpha(eps) (Eq. alpha) for f and g, BGK and push.  F holds the final
// normalised equilibrium; f^eq = rho F, g^eq = (2C_v - D) T rho F.
// PR: with the Prandtl-number adjustment (the quasi-equilibrium correction of g;
// a separate instantiation, so the paper's Pr = 1 collision carries none of it).
template <bool ODD, class P, int BLK, bool PR = false, bool D2 = false>
__device__ __forceinline__ int relax_push(const Desc& d, long long cell, const Nbr& nb,
                                          const Macro& M, WS<BLK> F) {
  const Phys& ph = d.ph;
  const double rho = M.rho;
  const float rho32 = trunc_float(rho);
  const double cgr = ph.cg * M.T * rho;
  double eps;
  if constexpr (sizeof(P) == 8) {
    P f[Q];
    gather<ODD, P, D2>(d, cell, nb, 0, f);
    // FP32 screen of 39 eps from float views (error bound: screen_undecided);
    // the FP64 value where the screen cannot decide the branch of Eq. (alpha)
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    int emin = SCREEN_EMAX, emax = SCREEN_EMIN;
    static_for<0, Q>([&](auto I) {  // one of each mirror pair, counted twice
      constexpr int i = decltype(I)::value;
      if constexpr (!D2 || zmirror(i) >= i) {
        const double Fd = F[i];
        const int eF = exp_field(Fd), ef = exp_field(f[i]);
        emin = min(emin, min(eF, ef));
        emax = max(emax, max(eF, ef));
        const float feq = rho32 * view_float(Fd);
        const float t = fabsf(view_float(f[i]) - feq) * rcp32(feq);
        acc[i & 3] += D2 && zmirror(i) != i ? 2.0f * t : t;
      }
    });
    const float s32 = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    eps = (double)s32 * (1.0 / Q);
    if (screen_undecided(s32, emin, emax, rho32)) {
      double fs[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) fs[i] = f[i];
      eps = sensor_sum_fp64<BLK>(fs, rho, F) * (1.0 / Q);
    }
    const int branch = alpha_branch(eps);
    const double omega = omega_of(ph, branch);
    static_for<0, Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      if constexpr (!D2 || zmirror(i) >= i)
        push_pair<ODD, P, i, D2>(d, cell, nb, 0, fma(-omega, fma(-rho, F[i], f[i]), f[i]));
    });
    double s13[NM];
    if constexpr (PR) gen::moments_s<double>(f, s13);  // sum_i f_i phi_k(xi_i)
    P g[Q];
    gather<ODD, P, D2>(d, cell, nb, Q, g);
    if constexpr (!PR) {
      static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if constexpr (!D2 || zmirror(i) >= i)
          push_pair<ODD, P, i, D2>(d, cell, nb, Q, fma(-omega, fma(-cgr, F[i], g[i]), g[i]));
      });
    } else {
      // heat flux q = (1/2) sum_i c_i (|c_i|^2 f_i + g_i), c_i = xi_i - u, from the raw
      // sums: sum_i f_i c_i |c_i|^2 = S3 - 2 S2 u - u sum_i f_i |xi_i|^2 + 2 rho u |u|^2
      const double ux = M.ux, uy = M.uy, uz = M.uz, u2 = ux * ux + uy * uy + uz * uz;
      const double e2f = s13[4] + s13[5] + s13[6];
      double g0 = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
      static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int cx = CX[i], cy = CY[i], cz = CZ[i];
        g0 += g[i];
        if constexpr (cx != 0) gx = fma((double)cx, g[i], gx);
        if constexpr (cy != 0) gy = fma((double)cy, g[i], gy);
        if constexpr (cz != 0) gz = fma((double)cz, g[i], gz);
      });
      const double r2u2 = 2.0 * s13[0] * u2;
      const double qx = 0.5 * (s13[10] - 2.0 * (s13[4] * ux + s13[7] * uy + s13[8] * uz) -
                               ux * e2f + r2u2 * ux + gx - ux * g0);
      const double qy = 0.5 * (s13[11] - 2.0 * (s13[7] * ux + s13[5] * uy + s13[9] * uz) -
                               uy * e2f + r2u2 * uy + gy - uy * g0);
      const double qz = 0.5 * (s13[12] - 2.0 * (s13[8] * ux + s13[9] * uy + s13[6] * uz) -
                               uz * e2f + r2u2 * uz + gz - uz * g0);
      // (1/tau - 1/tau2) g^eq_i (c_i . b), b = 2 q / ((2 C_v - D) rho T^2),
      // = F_i (beta0 + xi_i . beta) with beta = 2 (1/tau - 1/tau2) q / T, beta0 = -u . beta
      const double k = 2.0 * domega_of(ph, branch) / M.T;
      const double bx = k * qx, by = k * qy, bz = k * qz;
      const double b0 = -(ux * bx + uy * by + uz * bz);
      static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int cx = CX[i], cy = CY[i], cz = CZ[i];
        const double cb = fma((double)cx, bx, fma((double)cy, by, fma((double)cz, bz, b0)));
        push<ODD, P, i>(d, cell, nb, Q,
                        fma(F[i], cb, fma(-omega, fma(-cgr, F[i], g[i]), g[i])));
      });
    }
  } else {
    // precision form: h~ = h - h_ref stored in FP32; equilibrium deviation
    // h^eq - h_ref formed in FP64 and rounded; sensor and BGK in FP32.
    // The sensor compares each stored deviation with the equilibrium in the same storage,
    // rf_i = (f^eq_i - f_ref_i) rounded to float: s = 39 eps = sum_i |f~_i - rf_i| / f^eq_i.
    // FP32 screen, and the FP64 value of the same sum where the screen cannot decide the
    // branch of Eq. (alpha) (screen_undecided_dev), so alpha is an FP64 decision.
    const double* __restrict__ href = d.href;
    P f[Q];
    gather<ODD, P>(d, cell, nb, 0, f);
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const double Fi = F[i];
      f[i] -= __double2float_rn(fma(rho, Fi, -__ldg(href + i)));  // f~ - (f^eq - f_ref)
      acc[i & 3] += fabsf(f[i]) * rcp32(rho32 * trunc_float(Fi));
    }
    const float s32 = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    eps = (double)s32 * (1.0 / Q);
    if (screen_undecided_dev(s32)) {
      P fs[Q];
      gather<ODD, P>(d, cell, nb, 0, fs);  // the stored values (cached)
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const double feq = rho * F[i];
        const float rf = __double2float_rn(fma(rho, F[i], -__ldg(href + i)));
        s += fabs((double)fs[i] - (double)rf) / feq;  // the difference is exact
      }
      eps = s * (1.0 / Q);
    }
    const float omega = (float)omega_of(ph, alpha_branch(eps));
    P f2[Q];
    gather<ODD, P>(d, cell, nb, 0, f2);  // the stored values again (cached)
    static_for<0, Q>([&](auto I) {
      constexpr int i = decltype(I)::value;
      push<ODD, P, i>(d, cell, nb, 0, fmaf(-omega, f[i], f2[i]));
    });
    P g[Q];
    gather<ODD, P>(d, cell, nb, Q, g);
    if constexpr (!PR) {
      static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        const float qg = __double2float_rn(fma(cgr, F[i], -__ldg(href + Q + i)));
        push<ODD, P, i>(d, cell, nb, Q, fmaf(-omega, g[i] - qg, g[i]));
      });
    } else {
      // heat flux from the non-equilibrium parts (the 13-moment equilibrium has none):
      // q = (1/2) sum_i c_i (|c_i|^2 (f_i - f^eq_i) + (g_i - g^eq_i)), in FP32
      const float ux = (float)M.ux, uy = (float)M.uy, uz = (float)M.uz;
      float e[Q], qx = 0.0f, qy = 0.0f, qz = 0.0f;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        e[i] = g[i] - __double2float_rn(fma(cgr, F[i], -__ldg(href + Q + i)));  // g - g^eq
        const float cx = (float)kCX[i] - ux, cy = (float)kCY[i] - uy, cz = (float)kCZ[i] - uz;
        const float w = 0.5f * fmaf(cx * cx + cy * cy + cz * cz, f[i], e[i]);
        qx = fmaf(cx, w, qx);
        qy = fmaf(cy, w, qy);
        qz = fmaf(cz, w, qz);
      }
      const float k = (float)(2.0 * domega_of(ph, alpha_branch(eps)) / M.T);
      const float bx = k * qx, by = k * qy, bz = k * qz;
      const float b0 = -(ux * bx + uy * by + uz * bz);
      static_for<0, Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int cx = CX[i], cy = CY[i], cz = CZ[i];
        const float cb = fmaf((float)cx, bx, fmaf((float)cy, by, fmaf((float)cz, bz, b0)));
        push<ODD, P, i>(d, cell, nb, Q, fmaf(trunc_float(F[i]), cb, fmaf(-omega, e[i], g[i])));
      });
    }
  }
  return alpha_branch(eps);
}

template <int BLK>
__device__ __forceinline__ void flush_stats(unsigned int* s_ctr, unsigned long long* ctr) {
  __syncthreads();
  for (int k = threadIdx.x; k < CTR_N; k += BLK)
    if (s_ctr[k]) atomicAdd(ctr + k, (unsigned long long)s_ctr[k]);
}

// Per-cell solver state between steps: lam (13 planes) and F = exp(Phi lam)
// (39 planes), in that order from Desc::lam.
constexpr int SOLVER_PLANES = NM + Q;

template <int BLK>
__device__ __forceinline__ void load_multipliers(const Desc& d, long long cell, WS<BLK> w) {
  const double* __restrict__ st = d.lam;
#pragma unroll
  for (int k = 0; k < NM; ++k) w[WS_LAM + k] = at(st + k * d.Np, (int)cell);
}

template <int BLK, bool D2 = false>
__device__ __forceinline__ void load_cached_F(const Desc& d, long long cell, WS<BLK> w) {
  const double* __restrict__ st = d.lam;
  static_for<0, Q>([&](auto I) {  // D2: one of each mirror pair is read
    constexpr int i = decltype(I)::value;
    if constexpr (!D2 || zmirror(i) >= i) {
      const double v = at(st + (NM + i) * d.Np, (int)cell);
      w[WS_E + i] = v;
      if constexpr (D2 && zmirror(i) != i) w[WS_E + zmirror(i)] = v;
    }
  });
}

template <int BLK>
__device__ __forceinline__ void load_solver_state(const Desc& d, long long cell, WS<BLK> w) {
  load_multipliers<BLK>(d, cell, w);
  load_cached_F<BLK>(d, cell, w);
}

template <int BLK>
__device__ __forceinline__ void store_solver_state(const Desc& d, long long cell, WS<BLK> w) {
  double* __restrict__ st = d.lam + cell;
#pragma unroll 4
  for (int k = 0; k < NM; ++k) st[k * d.Np] = w[WS_LAM + k];
  st += NM * d.Np;
#pragma unroll 4
  for (int i = 0; i < Q; ++i) st[i * d.Np] = w[WS_E + i];
}

// F = exp(Phi lam) at the workspace multipliers.
template <int BLK>
__device__ __forceinline__ void eval_at_lam(WS<BLK> w) {
  double G[NM];
  const WS<1> none{nullptr};
  eval_equilibrium<BLK>(w.at(WS_LAM), none, 0.0, w.at(WS_E), w.at(WS_M), G, false,
                        gen::kExp2Table);
}

// Where the 13-moment solve failed or took no update: the fallback's
// multipliers embedded in lam and marked (lam unchanged but unmarked if the
// fallback fails too), and F = exp(Phi lam) exactly as the full solve
// evaluates it (the fallback evaluates the embedding with the same exponents
// and exponential), so the cached F stays exact.  retry:
// the cell came in with a fallback embedding, whose five multipliers (still in
// the stored state) start the fallback.
// state, Np: the solver-state planes (Desc::lam) and their stride.
template <int BLK>
__device__ __noinline__ void fallback_cell(const double* state, long long Np, long long cell,
                                           WS<BLK> w, double T, bool retry) {
  double warm[N5];
  if (retry) {
#pragma unroll
    for (int k = 0; k < N5; ++k) warm[k] = state[k * Np + cell];
  }
  WS<BLK> lam = w.at(WS_LAM);
  if (fallback_equilibrium<BLK>(w, T, retry ? warm : nullptr) == 0) {
    WS<BLK> mu = w.at(WS_M);
#pragma unroll
    for (int k = 0; k < 4; ++k) lam[k] = mu[k];
    lam[4] = lam[5] = lam[6] = mu[4];
#pragma unroll
    for (int k = 7; k < NM; ++k) lam[k] = 0.0;
    lam[9] = -0.0;  // the embedding mark: on the fallback
    // F already holds exp(Phi lam): the fallback's last evaluation was at this
    // embedding, with the full solve's exponents and exponential
  } else {
    lam[9] = lam[9] + 0.0;  // the fallback failed too: not on the fallback
    eval_at_lam<BLK>(w);    // F = exp(Phi lam), the cached value the next solve starts from
  }
}

// Newton budget of a cell on the fallback at time step t: the full budget
// maxit on the steps that are multiples of RETRY_PERIOD, else none.
__device__ __forceinline__ int retry_budget(long long t, int maxit) {
  return (t & (RETRY_PERIOD - 1)) == 0 ? maxit : 0;
}

// Whether a kernel solves in fixed point.  The chord-Newton hybrid does not: its factor fills the
// registers.  Nor does the precision form: its stores round F to FP32 deviations, and a last bit
// of F that falls the other way there changes the stored state by 1e-9 and grows with the flow.
template <class P, int SOLVER>
constexpr bool in_fixed_point = sizeof(P) == 8 && SOLVER != 1;

// Threads per block of the kernels that solve, and their workspace (the FP64 solves keep their
// direction there too).
constexpr int solve_blk(bool fixed) { return fixed ? 128 : 64; }
constexpr int solve_min_blocks(bool fixed) { return fixed ? 3 : 4; }
// The FP64 kernels beside the fixed-point ones: one block an SM, as many warps as four blocks of 64
// (a step's launch that finds nothing to do is over sooner with 152 blocks than with 608).
constexpr int FP64_BLK = 256;
constexpr size_t FP64_WS_BYTES = (size_t)FP64_BLK * WS_DOUBLES * sizeof(double);
constexpr size_t ws_bytes(bool fixed) {
  return (size_t)solve_blk(fixed) * (fixed ? WS_DOUBLES_FX : WS_DOUBLES) * sizeof(double);
}

// The table of the exponential that the solver reads, for the whole block.
template <bool FIXED>
__device__ __forceinline__ void load_solver_table() {
  if constexpr (FIXED) fx::load_table();
  else load_exp_table();
}

// The constraint solve of a cell from the warm start in the workspace (F cached
// at lam) with the lattice's root finder SOLVER (FP64 path): 0 Newton-Raphson;
// 1 the chord-Newton hybrid (newton_chord); 2 Newton with a single-precision
// direction; 3 that after a single-precision start (start32).  The precision
// form (P = float) always takes 3.  n32: the float steps of the start.
// FIXED: in fixed point (newton_fx); false for a cell that it cannot represent,
// whose stored state has not changed: it is solved in FP64.  There the
// workspace's multipliers are read from the stored state when the first update
// needs them, and moved says whether the workspace's state has changed (its
// multipliers are loaded then).  Else in FP64, always true.
template <class P, int BLK, bool D2, int SOLVER, bool FIXED>
__device__ __forceinline__ bool solve_cell(const Desc& d, long long cell, WS<BLK> w, int maxit,
                                           NewtonResult& nr, int& n32, bool& moved) {
  constexpr bool MIXED = sizeof(P) == 4 || SOLVER >= 2, START = sizeof(P) == 4 || SOLVER == 3;
  n32 = 0;
  moved = true;
  bool cached = true;
  [[maybe_unused]] const unsigned lanes = __activemask();
  if constexpr (START) {
    if (FIXED) load_multipliers<BLK>(d, cell, w);
    if (maxit > 0) {  // a cell on the fallback off a retry step takes no step at all
      n32 = start32<BLK, D2>(w);
      cached = n32 == 0;
    }
    if constexpr (FIXED) __syncwarp(lanes);  // see step_cell
  }
  if constexpr (FIXED) {
    const double* src = START ? w.p + WS_LAM * BLK : d.lam + cell;
    if (!newton_fx<BLK, !MIXED, D2>(w, src, START ? BLK : d.Np, d.ph, maxit, cached, nr, moved))
      return false;
    if constexpr (START) moved = moved || n32 > 0;
  } else if constexpr (SOLVER == 1 && sizeof(P) == 8) {
    nr = newton_chord<BLK, D2>(w, d.ph, maxit, true);
  } else {
    nr = newton_in<BLK, MIXED, D2>(w, w.at(WS_DL), exp_table(), d.ph.tol, d.ph.min_upd, maxit,
                                   cached);
  }
  return true;
}

// One fluid cell's time step (even or odd AA pass): phases A, B and C, with
// the Newton statistics added to the block's counters.  w: the cell's workspace.
// D2: the nine-function constraint system of a z-mirror-symmetric lattice one
// cell thick in z (Sys<true>; the same values as the full system wherever both solve).
// SOLVER: the root finder of the constraint equations (solve_cell).
// FIXED: solved in fixed point; true, with nothing done, for a cell that is left
// to the FP64 step.
template <bool ODD, class P, int BLK, bool D2 = false, bool PR = false, int SOLVER = 0,
          bool FIXED = in_fixed_point<P, SOLVER>>
__device__ __forceinline__ bool step_cell(const Desc& d, long long cell, WS<BLK> w,
                                          unsigned int* s_ctr) {
  WS<BLK> F = w.at(WS_E), lam = w.at(WS_LAM), m = w.at(WS_M);
  Coord c{0, 0, 0};
  if constexpr (ODD) c = coord_of(d, cell);
  constexpr bool INTEGER = in_fixed_point<P, SOLVER>;  // also in the FP64 step of such a lattice
  constexpr bool HALF = D2 && INTEGER;                 // one of each mirror pair is read
  Macro M;
  if constexpr (INTEGER) M = step_moments<ODD, D2>(d, cell, fresh_nbr<ODD>(d, c));
  else M = gather_moments<ODD, P>(d, cell, fresh_nbr<ODD>(d, c));
  targets<BLK>(M.ux, M.uy, M.uz, M.T, m);
  bool marked;
  if constexpr (FIXED) {
    load_cached_F<BLK, D2>(d, cell, w);
    // lam_9 = -0 is the mark's first sign; the other multipliers are read only then
    marked = __double_as_longlong(d.lam[9 * d.Np + cell]) == (long long)0x8000000000000000ull;
    if (marked) {
      load_multipliers<BLK>(d, cell, w);
      marked = is_fallback_embedding<BLK>(lam);
    }
  } else {
    load_solver_state<BLK>(d, cell, w);
    marked = is_fallback_embedding<BLK>(lam);
  }
  // a marked cell off a retry step gets no update (it stays on the fallback
  // unless its embedding already meets the 13 constraints)
  const int maxit = !marked ? d.ph.maxit : retry_budget(d.t, d.ph.maxit);
  int n32;
  bool moved;
  NewtonResult nr;
  const unsigned lanes = __activemask();
  const bool solved = solve_cell<P, BLK, D2, SOLVER, FIXED>(d, cell, w, maxit, nr, n32, moved);
  if constexpr (FIXED) {
    // the lanes go on together: with the return below, the compiler otherwise left a warp as its
    // solves had diverged, and phase C ran 1.7 times for each (a 128^3 box 54 ms, not 44.5).  With
    // root finder 3 they come together after its start, where that matters more (2 % on boxes)
    if constexpr (SOLVER != 3) __syncwarp(lanes);
    if (!solved) return true;
  }
  if (nr.failed) {
    if (!moved) load_multipliers<BLK>(d, cell, w);
    if constexpr (FIXED) targets<BLK>(M.ux, M.uy, M.uz, M.T, m);  // newton_fx overwrites them
    fallback_cell<BLK>(d.lam, d.Np, cell, w, M.T, marked);
    store_solver_state<BLK>(d, cell, w);
  } else if (moved) {
    lam[9] = lam[9] + 0.0;  // a solved state carries no embedding mark
    store_solver_state<BLK>(d, cell, w);
  } else if (marked) {
    d.lam[9 * d.Np + cell] = 0.0;
  }
  const int branch = relax_push<ODD, P, BLK, PR, HALF>(d, cell, fresh_nbr<ODD>(d, c), M, F);
  atomicAdd(&s_ctr[CTR_FAILED], (unsigned)nr.failed);
  atomicAdd(&s_ctr[CTR_UPDATES], (unsigned)nr.n_upd);
  atomicAdd(&s_ctr[CTR_HIST + min(nr.n_upd, 31)], 1u);
  atomicAdd(&s_ctr[CTR_EPS + branch], 1u);
  if (n32) {
    atomicAdd(&s_ctr[CTR_UPD32], (unsigned)n32);
    atomicAdd(&s_ctr[CTR_START32], 1u);
  }
  return false;
}

// The cells that a fixed-point kernel leaves to the FP64 solve.  They are few, but one of them can
// take hundreds of evaluations, and the slowest ends the step; they come in clusters, and the four
// warps of a block, solving in FP64 where they are, share one SM's FP64 pipe.  So the whole step of
// such a cell is put off to a launch of its own (its slots of the AA buffer are its own), whose
// warps take the list's entries one by one and which has the 255 registers of an FP64 solve.
// A 64^3 box at rms Ma 1.3 takes 136 ms for 8 steps; with these cells solved in place, at the
// fixed-point kernel's 168 registers, 196, and with FP64 solves for all cells 161.
// leave: by whole warps; appends the cells of the lanes with left set to list k.
__device__ __forceinline__ void leave(const Desc& d, int k, long long cell, bool left) {
  const unsigned bits = __ballot_sync(0xffffffffu, left);
  if (bits != 0 && (threadIdx.x & 31) == 0)
    d.rest[atomicAdd(d.ctr + CTR_REST + k, 1ull)] = Rest{(unsigned)(cell >> 5), bits};
}

// The entry that this warp takes after entry e, of lists shared by `warps` warps.
__device__ __forceinline__ long long next_entry(unsigned long long* taken, long long warps) {
  unsigned long long e = 0;
  if ((threadIdx.x & 31) == 0) e = atomicAdd(taken, 1ull);
  return warps + (long long)__shfl_sync(0xffffffffu, e, 0);
}

// This warp's first entry: neighbouring entries go to different SMs.
__device__ __forceinline__ long long first_entry() {
  return (long long)(threadIdx.x / 32) * gridDim.x + blockIdx.x;
}

// Calls f(cell) for each cell of list k, or with all for each of n cells; a warp takes the 32 cells
// of an entry together, as the fixed-point kernel had them.
template <class F>
__device__ __forceinline__ void for_rest(const Desc& d, int k, bool all, long long n, F&& f) {
  const long long warps = (long long)gridDim.x * (blockDim.x / 32);
  const long long count = all ? (n + 31) / 32 : (long long)d.ctr[CTR_REST + k];
  long long e = first_entry();
  while (e < count) {
    const Rest r = all ? Rest{(unsigned)e, 0xffffffffu} : d.rest[e];
    const long long cell = (long long)r.w * 32 + (threadIdx.x & 31);
    if ((r.bits >> (threadIdx.x & 31) & 1) && cell < n) f(cell);
    __syncwarp();
    e = next_entry(d.ctr + CTR_TAKEN + k, warps);
  }
}

// Empties list k before its next use.
__device__ __forceinline__ void clear_rest(const Desc& d, int k) {
  d.ctr[CTR_REST + k] = 0;
  d.ctr[CTR_TAKEN + k] = 0;
}

// One time step over every fluid cell (even or odd AA pass).
template <bool ODD, class P, int BLK, bool D2, bool PR = false, int SOLVER = 0>
__global__ void __launch_bounds__(BLK, solve_min_blocks(in_fixed_point<P, SOLVER>)) k_step(Desc d) {
  extern __shared__ double smem[];
  __shared__ unsigned int s_ctr[CTR_N];
  for (int k = threadIdx.x; k < CTR_N; k += BLK) s_ctr[k] = 0;
  load_solver_table<in_fixed_point<P, SOLVER>>();
  cudaGridDependencySynchronize();  // launch_step
  const long long cell = (long long)blockIdx.x * BLK + threadIdx.x;
  bool left = false;
  if (cell < d.N && (d.mask == nullptr || d.mask[cell] == MASK_FLUID))
    left = step_cell<ODD, P, BLK, D2, PR, SOLVER>(d, cell, WS<BLK>{smem + threadIdx.x}, s_ctr);
  if constexpr (in_fixed_point<P, SOLVER>) leave(d, ODD, cell, left);
  flush_stats<BLK>(s_ctr, d.ctr);
}

// The step of the cells left by k_step, or with all of every fluid cell, solved in FP64.  All: the
// lattices whose tolerance is below the fixed-point resolution (at 1e-13 a 64^3 box's 8 steps take
// 24.6 ms; 25.4 where the fixed-point kernel called the FP64 solve for each cell).
template <bool ODD, bool D2, bool PR, int SOLVER>
__global__ void __launch_bounds__(FP64_BLK, 1) k_step_fp64(Desc d, bool all) {
  constexpr int BLK = FP64_BLK;
  extern __shared__ double smem[];
  __shared__ unsigned int s_ctr[CTR_N];
  cudaGridDependencySynchronize();
  if (blockIdx.x == 0 && threadIdx.x == 0) clear_rest(d, !ODD);
  if (!all && d.ctr[CTR_REST + ODD] == 0) return;
  for (int k = threadIdx.x; k < CTR_N; k += BLK) s_ctr[k] = 0;
  load_exp_table();
  for_rest(d, ODD, all, d.N, [&](long long cell) {
    if (d.mask == nullptr || d.mask[cell] == MASK_FLUID)
      step_cell<ODD, double, BLK, D2, PR, SOLVER, false>(d, cell, WS<BLK>{smem + threadIdx.x},
                                                         s_ctr);
  });
  flush_stats<BLK>(s_ctr, d.ctr);
}

// Stored value of population j (0..77) whose FP64 value is v.
template <class P>
__device__ __forceinline__ P to_store(const Desc& d, int j, double v) {
  if constexpr (sizeof(P) == 8) return v;
  else return __double2float_rn(v - __ldg(d.href + j));
}

// gaussian_guess out of line (39 FP64 exponentials).
template <int BLK>
__device__ __noinline__ void gaussian_guess_out(double ux, double uy, double uz, double T,
                                                WS<BLK> lam) {
  gaussian_guess<BLK>(ux, uy, uz, T, lam);
}

// Equilibrium initial condition of a cell, its inputs at index r; returns whether it is left to
// the FP64 kernel (FIXED; nothing is written then).  asym: whether it starts with u_z != 0.
template <class P, int BLK, bool FIXED>
__device__ __forceinline__ bool init_cell(const Desc& d, const double* rho, const double* u,
                                          long long us, const double* T, long long cell,
                                          long long r, int maxit, WS<BLK> w, unsigned int* s_ctr,
                                          bool& asym) {
  P* pop = static_cast<P*>(d.pop);
  if (d.mask != nullptr && d.mask[cell] != MASK_FLUID) {
    for (int j = 0; j < 2 * Q; ++j) pop[(long long)j * d.Np + cell] = P(0);
    for (int k = 0; k < SOLVER_PLANES; ++k) d.lam[k * d.Np + cell] = 0.0;
    return false;
  }
  const double rr = rho[r], ux = u[r], uy = u[us + r], uz = u[2 * us + r], TT = T[r];
  asym = uz != 0.0;
  WS<BLK> lam = w.at(WS_LAM), F = w.at(WS_E), m = w.at(WS_M);
  targets<BLK>(ux, uy, uz, TT, m);
  NewtonResult nr;
  if constexpr (FIXED) {
    bool moved;
    const unsigned lanes = __activemask();
    const bool solved = gaussian_guess_fx<BLK>(ux, uy, uz, TT, w) &&
                        newton_fx<BLK, true, false>(w, lam.p, BLK, d.ph, maxit, false, nr, moved);
    __syncwarp(lanes);  // as in step_cell
    if (!solved) return true;
    if (nr.failed) targets<BLK>(ux, uy, uz, TT, m);  // newton_fx overwrites them
  } else {
    gaussian_guess_out<BLK>(ux, uy, uz, TT, lam);
    nr = newton_in<BLK, false, false>(w, w.at(WS_DL), exp_table(), d.ph.tol, d.ph.min_upd, maxit,
                                      false);
  }
  if (nr.failed) fallback_cell<BLK>(d.lam, d.Np, cell, w, TT, false);
  store_solver_state<BLK>(d, cell, w);
  const double cgr = d.ph.cg * TT * rr;
  for (int i = 0; i < Q; ++i) {
    pop[(long long)i * d.Np + cell] = to_store<P>(d, i, rr * F[i]);
    pop[(long long)(Q + i) * d.Np + cell] = to_store<P>(d, Q + i, cgr * F[i]);
  }
  atomicAdd(&s_ctr[CTR_FAILED], (unsigned)nr.failed);
  return false;
}

// Equilibrium initial condition of the cells in [c0, c0 + len): inputs are
// indexed by cell - c0; u planes are `us` elements apart.  Non-fluid cells in
// the range get zero populations and multipliers.  list: where the cells left
// to the FP64 kernel go.
template <class P, int BLK>
__global__ void __launch_bounds__(BLK, solve_min_blocks(in_fixed_point<P, 0>)) k_init(Desc d, const double* rho, const double* u,
                                              long long us, const double* T, long long c0,
                                              long long len, int maxit, int list) {
  constexpr bool FIXED = in_fixed_point<P, 0>;
  extern __shared__ double smem[];
  __shared__ unsigned int s_ctr[CTR_N];
  for (int k = threadIdx.x; k < CTR_N; k += BLK) s_ctr[k] = 0;
  load_solver_table<FIXED>();
  const long long r = (long long)blockIdx.x * BLK + threadIdx.x;
  bool asym = false, left = false;
  if (r < len && c0 + r < d.N)
    left = init_cell<P, BLK, FIXED>(d, rho, u, us, T, c0 + r, r, maxit, WS<BLK>{smem + threadIdx.x},
                                    s_ctr, asym);
  if constexpr (FIXED) leave(d, list, r, left);
  if (__syncthreads_or(asym) && threadIdx.x == 0) atomicAdd(d.ctr + CTR_ASYM, 1ull);
  flush_stats<BLK>(s_ctr, d.ctr);
}

// The initial condition of the cells of the range left by k_init, or with all of every cell,
// solved in FP64 (FP64 storage).
template <int BLK>
__global__ void __launch_bounds__(BLK, 1)
    k_init_fp64(Desc d, const double* rho, const double* u, long long us, const double* T,
                long long c0, long long len, int maxit, int list, bool all) {
  extern __shared__ double smem[];
  __shared__ unsigned int s_ctr[CTR_N];
  cudaGridDependencySynchronize();
  if (blockIdx.x == 0 && threadIdx.x == 0) clear_rest(d, list ^ 1);
  if (!all && d.ctr[CTR_REST + list] == 0) return;
  for (int k = threadIdx.x; k < CTR_N; k += BLK) s_ctr[k] = 0;
  load_exp_table();
  bool any = false;
  for_rest(d, list, all, min(len, d.N - c0), [&](long long r) {
    bool asym = false;
    init_cell<double, BLK, false>(d, rho, u, us, T, c0 + r, r, maxit, WS<BLK>{smem + threadIdx.x},
                                  s_ctr, asym);
    any = any || asym;
  });
  if (__syncthreads_or(any) && threadIdx.x == 0) atomicAdd(d.ctr + CTR_ASYM, 1ull);
  flush_stats<BLK>(s_ctr, d.ctr);
}

// Equilibrium populations (f then g, 78 values) and multipliers of one state
// (rho, u, T), from a cold start; one thread.  Used for the far-field state
// and for the reference state of the precision form.
template <int BLK>
__global__ void __launch_bounds__(BLK) k_state_equilibrium(Phys ph, double rho, double ux,
                                                           double uy, double uz, double T,
                                                           double* out78, int maxit,
                                                           unsigned long long* failed) {
  extern __shared__ double smem[];
  if (threadIdx.x != 0) return;
  WS<BLK> w{smem};
  WS<BLK> lam = w.at(WS_LAM), F = w.at(WS_E), m = w.at(WS_M);
  targets<BLK>(ux, uy, uz, T, m);
  gaussian_guess<BLK>(ux, uy, uz, T, lam);
  const NewtonResult nr = newton<BLK, false>(w, ph.tol, ph.min_upd, maxit, false);
  for (int i = 0; i < Q; ++i) {
    out78[i] = rho * F[i];
    out78[Q + i] = ph.cg * T * rho * F[i];
  }
  if (nr.failed) atomicAdd(failed, 1ull);
}

// A population reversed by the bounce-back: the stored value v of population
// `from` becomes population `to`.  FP64 storage holds the populations
// themselves; the precision form holds deviations from the reference
// populations, which differ between the two directions unless the reference
// is at rest, so the value is re-referenced: (v + h_ref,from) - h_ref,to.
template <class P>
__device__ __forceinline__ P reversed(const Desc& d, P v, int from, int to) {
  if constexpr (sizeof(P) == 8) return v;
  else return __double2float_rn((double)v + (__ldg(d.href + from) - __ldg(d.href + to)));
}

// The fill functions take their 39 directions in batches: the masks of a batch, then its
// populations, are read before the first is stored, and the neighbours are computed where the
// table of them would lie in local memory.  Few cells have work, and each waits for memory: what
// counts is that many blocks are resident (40 registers, six blocks of 256, with about 250 bytes of
// spills) and that a cell waits less often.  On the 1024 x 512 airfoil a fill takes 16 us (even) and
// 24 us (odd) where the direction-by-direction loops took 40 and 30; batches of 13 took 19 and 37
// (128 registers).
constexpr int FILL_BATCH = 3;
static_assert(Q % FILL_BATCH == 0, "whole batches");

// Index of the cell at c + (dx, dy, dz), as Nbr gives it.
__device__ __forceinline__ int neighbour(const Desc& d, Coord c, int dx, int dy, int dz) {
  return wrap(c.x + dx, d.nx) + (wrap(c.y + dy, d.ny) + wrap(c.z + dz, d.nz) * d.ny) * d.nx;
}

// Half-way bounce-back (Sec. 4) after an even pass.  The even pass leaves
// f*_opp(i)(x) of a fluid cell x in its slot i; the odd pass gathers f_i(x)
// from (x - xi_i, slot opp i), which for x = s + xi_i is (s, slot opp i): the
// solid cell s copies the value there.  Each of these slots has one writer.
template <class P>
__device__ __forceinline__ void bounce_even_cell(const Desc& d, long long s) {
  P* pop = static_cast<P*>(d.pop);
  const Coord c = coord_of(d, s);
#pragma unroll 1
  for (int i0 = 0; i0 < Q; i0 += FILL_BATCH) {
    int x[FILL_BATCH];
    bool fluid[FILL_BATCH];
    P f[FILL_BATCH], g[FILL_BATCH];
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      x[j] = neighbour(d, c, kCX[i], kCY[i], kCZ[i]);
      fluid[j] = d.mask[x[j]] == MASK_FLUID;
    }
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      if (fluid[j]) {
        f[j] = pop[(long long)i * d.Np + x[j]];
        g[j] = pop[(long long)(Q + i) * d.Np + x[j]];
      }
    }
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j, o = opp(i);  // population o of x is in its slot i; it returns as population i
      if (fluid[j]) {
        pop[(long long)o * d.Np + s] = reversed<P>(d, f[j], o, i);
        pop[(long long)(Q + o) * d.Np + s] = reversed<P>(d, g[j], Q + o, Q + i);
      }
    }
  }
}

// Half-way bounce-back after an odd pass: fluid cell x = s - xi_i pushed
// f*_i(x) into (s, slot i); it returns as f_opp(i)(x), which the even pass
// reads from (x, slot opp i) -- a slot no push writes, since its source
// x - xi_opp(i) = s is solid.
template <class P>
__device__ __forceinline__ void bounce_odd_cell(const Desc& d, long long s) {
  P* pop = static_cast<P*>(d.pop);
  const Coord c = coord_of(d, s);
#pragma unroll 1
  for (int i0 = 0; i0 < Q; i0 += FILL_BATCH) {
    int x[FILL_BATCH];
    bool fluid[FILL_BATCH];
    P f[FILL_BATCH], g[FILL_BATCH];
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      x[j] = neighbour(d, c, -kCX[i], -kCY[i], -kCZ[i]);
      fluid[j] = d.mask[x[j]] == MASK_FLUID;
    }
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      if (fluid[j]) {
        f[j] = pop[(long long)i * d.Np + s];
        g[j] = pop[(long long)(Q + i) * d.Np + s];
      }
    }
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j, o = opp(i);  // population i of x returns as its population o
      if (fluid[j]) {
        pop[(long long)o * d.Np + x[j]] = reversed<P>(d, f[j], i, o);
        pop[(long long)(Q + o) * d.Np + x[j]] = reversed<P>(d, g[j], Q + i, Q + o);
      }
    }
  }
}

// After an even pass: freestream cells hold the far-field post-collision
// populations and outflow cells a copy of the cell with x clamped into
// [3, nx-4], both in the reversed (post-collision) layout the odd pass reads;
// solid cells do their bounce-back copies.
template <class P>
__device__ __forceinline__ void fill_even_cell(const Desc& d, long long cell) {
  const uint8_t mk = d.mask[cell];
  if (mk == MASK_SOLID) {
    bounce_even_cell<P>(d, cell);
    return;
  }
  if (mk != MASK_FREE && mk != MASK_OUT) return;
  P* pop = static_cast<P*>(d.pop);
  const P* fs = static_cast<const P*>(d.free_store);
  long long src = -1;
  if (mk == MASK_OUT) {
    const Coord c = coord_of(d, cell);
    const int xc = min(max(c.x, 3), d.nx - 4);
    src = cell + (xc - c.x);
    if (d.mask[src] == MASK_FREE) src = -1;
  }
#pragma unroll 1
  for (int i0 = 0; i0 < Q; i0 += FILL_BATCH) {
    P f[FILL_BATCH], g[FILL_BATCH];
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      const long long jf = (long long)opp(i) * d.Np, jg = (long long)(Q + opp(i)) * d.Np;
      f[j] = src < 0 ? fs[i] : pop[jf + src];
      g[j] = src < 0 ? fs[Q + i] : pop[jg + src];
    }
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      pop[(long long)opp(i) * d.Np + cell] = f[j];
      pop[(long long)(Q + opp(i)) * d.Np + cell] = g[j];
    }
  }
}

// After an odd pass: fluid slots whose source is a freestream or outflow cell
// receive what that cell streamed: the far-field equilibrium, or the
// post-collision population of the clamped cell c, which c pushed into slot
// (c + xi_i, i) (also when c + xi_i is solid: bounce_odd_cell only copies it
// on; that slot's source is c, a fluid cell, so no fill writes it).  Solid
// cells do their bounce-back copies.
template <class P>
__device__ __forceinline__ void fill_odd_cell(const Desc& d, long long cell) {
  const uint8_t mk = d.mask[cell];
  if (mk == MASK_SOLID) {
    bounce_odd_cell<P>(d, cell);
    return;
  }
  if (mk != MASK_FLUID) return;
  const Coord c = coord_of(d, cell);
  const bool near = (!d.per[0] && (c.x < 6 || c.x >= d.nx - 6)) ||
                    (!d.per[1] && (c.y < 6 || c.y >= d.ny - 6)) ||
                    (!d.per[2] && (c.z < 6 || c.z >= d.nz - 6));
  if (!near) return;
  P* pop = static_cast<P*>(d.pop);
  const P* fs = static_cast<const P*>(d.free_store);
#pragma unroll 1
  for (int i0 = 0; i0 < Q; i0 += FILL_BATCH) {
    uint8_t ms[FILL_BATCH], mc[FILL_BATCH];  // masks of the source and of its clamped cell
    P f[FILL_BATCH], g[FILL_BATCH];
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      const int sx = wrap(c.x - kCX[i], d.nx);
      const int s = neighbour(d, c, -kCX[i], -kCY[i], -kCZ[i]);
      ms[j] = d.mask[s];
      mc[j] = MASK_FREE;
      if (!d.per[0]) mc[j] = d.mask[s + (min(max(sx, 3), d.nx - 4) - sx)];
    }
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      if (ms[j] != MASK_FREE && ms[j] != MASK_OUT) continue;
      f[j] = fs[i];
      g[j] = fs[Q + i];
      if (ms[j] == MASK_OUT && mc[j] != MASK_FREE) {
        const Coord cc{min(max(wrap(c.x - kCX[i], d.nx), 3), d.nx - 4),
                       wrap(c.y - kCY[i], d.ny), wrap(c.z - kCZ[i], d.nz)};
        const long long t = (long long)i * d.Np + neighbour(d, cc, kCX[i], kCY[i], kCZ[i]);
        f[j] = pop[t];
        g[j] = pop[t + Q * d.Np];
      }
    }
#pragma unroll
    for (int j = 0; j < FILL_BATCH; ++j) {
      const int i = i0 + j;
      if (ms[j] != MASK_FREE && ms[j] != MASK_OUT) continue;
      pop[(long long)i * d.Np + cell] = f[j];
      pop[(long long)(Q + i) * d.Np + cell] = g[j];
    }
  }
}

constexpr int FILL_BLK = 256;

template <class P>
__global__ void __launch_bounds__(FILL_BLK, 6) k_fill_even(Desc d) {
  const long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell < d.N) fill_even_cell<P>(d, cell);
}

template <class P>
__global__ void __launch_bounds__(FILL_BLK, 6) k_fill_odd(Desc d) {
  const long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell < d.N) fill_odd_cell<P>(d, cell);
}

// rho, u, T, p = rho T of cells [c0, c0 + len) into out arrays indexed by
// cell - c0 (u planes `us` apart; any pointer may be null); non-fluid cells 0.
template <bool ODD, class P>
__global__ void k_macros(Desc d, double* rho, double* u, long long us, double* T, double* p,
                         long long c0, long long len) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long cell = c0 + r;
  if (r >= len || cell >= d.N) return;
  Macro M{0, 0, 0, 0, 0};
  if (d.mask == nullptr || d.mask[cell] == MASK_FLUID) {
    Nbr nb;
    if constexpr (ODD) nb = Nbr(d, coord_of(d, cell));
    M = gather_moments<ODD, P>(d, cell, nb);
  }
  if (rho) rho[r] = M.rho;
  if (u) { u[r] = M.ux; u[us + r] = M.uy; u[2 * us + r] = M.uz; }
  if (T) T[r] = M.T;
  if (p) p[r] = M.rho * M.T;
}

// Conserved sums over fluid cells (mass, momentum, total energy): fixed
// grid-stride assignment and fixed-order tree reductions, so the result is
// deterministic.  partials: gridDim.x * 5 doubles.  Three blocks an SM: the loads wait for memory,
// and at the 246 registers that the odd gather otherwise takes lbm39_stats of a 64^3 box took 190 us
// instead of 179.
template <bool ODD, class P, int BLK>
__global__ void __launch_bounds__(BLK, 3) k_conserved(Desc d, double* partials) {
  __shared__ double red[5][BLK];
  double acc[5] = {0, 0, 0, 0, 0};
  for (long long cell = (long long)blockIdx.x * BLK + threadIdx.x; cell < d.N;
       cell += (long long)gridDim.x * BLK) {
    if (d.mask != nullptr && d.mask[cell] != MASK_FLUID) continue;
    Nbr nb;
    if constexpr (ODD) nb = Nbr(d, coord_of(d, cell));
    const Raw r = gather_raw<ODD, P>(d, cell, nb);
    acc[0] += r.rho;
    acc[1] += r.jx;
    acc[2] += r.jy;
    acc[3] += r.jz;
    acc[4] += 0.5 * r.e2;
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) red[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int s = BLK / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
#pragma unroll
      for (int k = 0; k < 5; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 5) partials[blockIdx.x * 5 + threadIdx.x] = red[threadIdx.x][0];
}

// Library reciprocals and CUDA's IEEE divisions side by side (diagnostic).
static __global__ void k_selftest_rcp(const double* x, double* y, double* ref, float* y32,
                                      float* ref32, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    y[i] = rcp64(x[i]);
    ref[i] = 1.0 / x[i];
    const float xf = (float)x[i];
    y32[i] = rcp32(xf);
    ref32[i] = 1.0f / xf;
  }
}

// Library exponential and CUDA's exp side by side (diagnostic).
static __global__ void k_selftest_exp(const double* x, double* y, double* ref, long long n) {
  load_exp_table();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    y[i] = exp_tang(x[i]);
    ref[i] = exp(x[i]);
  }
}

// FP64 FMA throughput probe: 8 independent chains per thread (diagnostic).
static __global__ void k_selftest_dfma(double* out, int iters, double a, double b) {
  double x0 = threadIdx.x * 1e-9, x1 = x0 + 1e-9, x2 = x0 + 2e-9, x3 = x0 + 3e-9;
  double x4 = x0 + 4e-9, x5 = x0 + 5e-9, x6 = x0 + 6e-9, x7 = x0 + 7e-9;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x0 = fma(x0, a, b); x1 = fma(x1, a, b); x2 = fma(x2, a, b); x3 = fma(x3, a, b);
      x4 = fma(x4, a, b); x5 = fma(x5, a, b); x6 = fma(x6, a, b); x7 = fma(x7, a, b);
    }
  }
  out[blockIdx.x * blockDim.x + threadIdx.x] = x0 + x1 + x2 + x3 + x4 + x5 + x6 + x7;
}

static __global__ void k_sum_partials(const double* partials, int nblocks, double* out5) {
  const int k = threadIdx.x;
  if (k >= 5) return;
  double s = 0.0;
  for (int b = 0; b < nblocks; ++b) s += partials[b * 5 + k];
  out5[k] = s;
}

// Blocks of the FP64 kernel of n cells: one an SM, or a warp for each 32 cells.
inline unsigned fp64_blocks(long long n) {
  return (unsigned)std::min((n + 31) / 32, 152LL);
}

// One time step over every fluid cell, without the boundary fills.
template <class P, bool D2, bool PR, int SOLVER>
void launch_step(const Desc& d, bool odd, cudaStream_t stream) {
  constexpr bool FIXED = in_fixed_point<P, SOLVER>;
  constexpr int BLK = solve_blk(FIXED);
  const unsigned grid = (unsigned)((d.N + BLK - 1) / BLK);
  if (!FIXED || d.ph.fx) {
    // where all blocks are resident at once the set-up is worth hiding; with more waves the blocks
    // set up early land unevenly on the SMs (shear layers of 300^2 and 330^2 took 4 and 5 % longer)
    constexpr size_t WSB = ws_bytes(FIXED);
    constexpr auto even = k_step<false, P, BLK, D2, PR, SOLVER>;
    constexpr auto odd_ = k_step<true, P, BLK, D2, PR, SOLVER>;
    if (grid <= 152u * solve_min_blocks(FIXED)) {
      if (odd) launch_ws_early<odd_>(grid, BLK, WSB, stream, d);
      else launch_ws_early<even>(grid, BLK, WSB, stream, d);
    } else {
      if (odd) launch_ws<odd_>(grid, BLK, WSB, stream, d);
      else launch_ws<even>(grid, BLK, WSB, stream, d);
    }
  }
  const bool all = !d.ph.fx;
  if constexpr (FIXED) {
    const unsigned grid64 = fp64_blocks(d.N);
    constexpr int B = FP64_BLK;
    constexpr size_t WSB = FP64_WS_BYTES;
    if (odd) launch_ws_early<k_step_fp64<true, D2, PR, SOLVER>>(grid64, B, WSB, stream, d, all);
    else launch_ws_early<k_step_fp64<false, D2, PR, SOLVER>>(grid64, B, WSB, stream, d, all);
  }
}

}  // namespace lbm39
