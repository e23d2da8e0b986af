// diag.cu -- per-cell diagnostic fields of a 13-moment lattice's current state:
// the Knudsen sensor eps (Eq. DeltaAvg) and the number of Newton updates the
// next step's solve takes, the two quantities the paper maps over the airfoil
// flow (Sec. 4).  Each cell does the next step's work up to its collision
// (moments, targets, the warm-started solve from the stored multipliers with
// the same retry schedule and root finder, the fallback equilibrium where the
// solve fails) and
// writes the two values; no population, multiplier or counter changes.
#include <cuda_runtime.h>

#include "../../include/lbm39.h"
#include "kernels.cuh"
#include "lattice_view.h"

namespace lbm39 {
namespace {


// f_i of the current state in FP64 (the stored deviation plus h_ref in the
// precision form; exact).
template <bool ODD, class P>
__device__ __forceinline__ void gather_f(const Desc& d, long long cell, double (&f)[Q]) {
  Nbr nb;
  if constexpr (ODD) nb = Nbr(d, coord_of(d, cell));
  P h[Q];
  gather<ODD, P>(d, cell, nb, 0, h);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if constexpr (sizeof(P) == 8) f[i] = h[i];
    else f[i] = (double)h[i] + d.href[i];
  }
}

// The step's own macroscopic variables (the same arithmetic, so the same updates).
template <bool ODD, class P, bool D2, bool FIXED>
__device__ __forceinline__ Macro moments_of(const Desc& d, long long cell) {
  Nbr nb;
  if constexpr (ODD) nb = Nbr(d, coord_of(d, cell));
  if constexpr (FIXED) return step_moments<ODD, D2>(d, cell, nb);
  else return gather_moments<ODD, P>(d, cell, nb);
}

// The FP64 solve of a cell that newton_fx gave up, from the stored state.
template <int BLK, bool D2, int SOLVER>
__device__ __forceinline__ NewtonResult solve_again(const Desc& d, long long cell, WS<BLK> w,
                                                    const Macro& M, int maxit, int& n32) {
  targets<BLK>(M.ux, M.uy, M.uz, M.T, w.at(WS_M));
  load_solver_state<BLK>(d, cell, w);
  n32 = 0;
  if constexpr (SOLVER == 3) {
    if (maxit > 0) n32 = start32<BLK, D2>(w);
  }
  return newton<BLK, (SOLVER >= 2), D2>(w, d.ph.tol, d.ph.min_upd, maxit, n32 == 0);
}

// eps: FP64 (1/Q) sum_i |f_i - f_i^eq| / f_i^eq of the state against the
// equilibrium the next step relaxes to; n_upd: its Newton updates, -1 where
// the solve fails (the cell takes the fallback equilibrium).  Non-fluid cells
// read 0.  odd: the AA parity of the lattice's time.
template <class P, bool D2, int SOLVER = 0>
__global__ void __launch_bounds__(solve_blk(in_fixed_point<P, SOLVER>))
    k_diag_fields(Desc d, int odd, double* eps_out, int* nupd_out) {
  constexpr bool FIXED = in_fixed_point<P, SOLVER>;
  constexpr int BLK = solve_blk(FIXED);
  extern __shared__ double smem[];
  load_solver_table<FIXED>();
  const long long cell = (long long)blockIdx.x * BLK + threadIdx.x;
  if (cell >= d.N) return;
  if (d.mask != nullptr && d.mask[cell] != MASK_FLUID) {
    eps_out[cell] = 0.0;
    nupd_out[cell] = 0;
    return;
  }
  WS<BLK> w{smem + threadIdx.x};
  WS<BLK> F = w.at(WS_E), lam = w.at(WS_LAM), m = w.at(WS_M);
  const Macro M = odd ? moments_of<true, P, D2, FIXED>(d, cell)
                      : moments_of<false, P, D2, FIXED>(d, cell);
  targets<BLK>(M.ux, M.uy, M.uz, M.T, m);
  load_solver_state<BLK>(d, cell, w);
  const bool marked = is_fallback_embedding<BLK>(lam);
  const int maxit = !marked ? d.ph.maxit : retry_budget(d.t, d.ph.maxit);
  int n32;
  bool moved;
  NewtonResult nr;
  bool solved = false;
  if (!FIXED || d.ph.fx) solved = solve_cell<P, BLK, D2, SOLVER, FIXED>(d, cell, w, maxit, nr, n32, moved);
  if constexpr (FIXED) {
    if (!solved) nr = solve_again<BLK, D2, SOLVER>(d, cell, w, M, maxit, n32);
  }
  if (nr.failed) {
    targets<BLK>(M.ux, M.uy, M.uz, M.T, m);  // the solve may have overwritten them
    fallback_cell<BLK>(d.lam, d.Np, cell, w, M.T, marked);
  }
  double f[Q];
  if (odd) gather_f<true, P>(d, cell, f);
  else gather_f<false, P>(d, cell, f);
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const double feq = M.rho * F[i];
    s += fabs(f[i] - feq) / feq;
  }
  eps_out[cell] = s * (1.0 / Q);
  nupd_out[cell] = nr.failed ? -1 : nr.n_upd;
}

template <class P, bool D2, int SOLVER = 0>
void launch_diag(const LatticeView& v, int odd, double* eps, int* n_upd) {
  constexpr bool FIXED = in_fixed_point<P, SOLVER>;
  constexpr int BLK = solve_blk(FIXED);
  launch_ws<k_diag_fields<P, D2, SOLVER>>((unsigned)((v.N + BLK - 1) / BLK), BLK,
                                          ws_bytes(FIXED), v.stream, v.desc, odd, eps, n_upd);
}

}  // namespace
}  // namespace lbm39

extern "C" int lbm39_diag_fields(lbm39_lattice* L, double* eps, int32_t* n_upd) {
  using namespace lbm39;
  LatticeView v;
  if (!lattice_view(L, &v) || !eps || !n_upd) return LBM39_ERR_ARG;
  if (!v.initialized) return LBM39_ERR_STATE;
  const int odd = (int)(v.desc.t & 1);
  if (v.mixed)
    launch_diag<float, false>(v, odd, eps, n_upd);
  else if (v.solver == 1 && v.desc.d2)
    launch_diag<double, true, 1>(v, odd, eps, n_upd);
  else if (v.solver == 1)
    launch_diag<double, false, 1>(v, odd, eps, n_upd);
  else if (v.solver == 2 && v.desc.d2)
    launch_diag<double, true, 2>(v, odd, eps, n_upd);
  else if (v.solver == 2)
    launch_diag<double, false, 2>(v, odd, eps, n_upd);
  else if (v.solver == 3 && v.desc.d2)
    launch_diag<double, true, 3>(v, odd, eps, n_upd);
  else if (v.solver == 3)
    launch_diag<double, false, 3>(v, odd, eps, n_upd);
  else if (v.desc.d2)
    launch_diag<double, true>(v, odd, eps, n_upd);
  else
    launch_diag<double, false>(v, odd, eps, n_upd);
  return cudaGetLastError() == cudaSuccess ? LBM39_OK : LBM39_ERR_CUDA;
}
