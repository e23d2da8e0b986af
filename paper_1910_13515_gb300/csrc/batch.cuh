// batch.cuh -- kernels of the serving form: many resident lattices advanced
// by one packed launch per time step.  A tile is one block of one lattice;
// each lattice keeps its own time (and therefore its own AA parity) and stops
// at its own end time, so a packed run gives every lattice exactly the
// arithmetic of stepping it alone.
#pragma once

#include "kernels.cuh"

namespace lbm39 {

struct BatchEntry {
  Desc d;
  long long t0;     // the lattice's time at step index 0 of the current launch sequence
  long long t_end;  // the lattice does not step past this time
};

struct Tile {
  int lat;          // index into the batch entries
  int pad;
  long long cell0;  // first cell of the tile
};

// D2: every lattice of these tiles takes the nine-constraint (z-mirror) solve
// (FP64 lattices one cell thick in z with u_z = 0); the host sorts the tiles by
// constraint system and launches one instantiation for each.
template <class P, int BLK, bool D2>
__global__ void __launch_bounds__(BLK, solve_min_blocks(in_fixed_point<P, 0>)) k_batch_step(const BatchEntry* __restrict__ E,
                                                    const Tile* __restrict__ tiles, int s) {
  extern __shared__ double smem[];
  __shared__ unsigned int s_ctr[CTR_N];
  __shared__ Desc sd;
  __shared__ long long st;
  const Tile tl = tiles[blockIdx.x];
  if (threadIdx.x == 0) {
    sd = E[tl.lat].d;
    st = E[tl.lat].t0 + s < E[tl.lat].t_end ? E[tl.lat].t0 + s : -1;
    sd.t = st;
  }
  for (int k = threadIdx.x; k < CTR_N; k += BLK) s_ctr[k] = 0;
  load_solver_table<in_fixed_point<P, 0>>();  // also publishes sd and st
  const long long t = st;
  if (t < 0) return;  // this lattice has reached its end time (uniform over the block)
  const long long cell = tl.cell0 + threadIdx.x;
  bool left = false;
  if (cell < sd.N && (sd.mask == nullptr || sd.mask[cell] == MASK_FLUID)) {
    WS<BLK> w{smem + threadIdx.x};
    if (in_fixed_point<P, 0> && !sd.ph.fx) left = true;
    else if (t & 1) left = step_cell<true, P, BLK, D2>(sd, cell, w, s_ctr);
    else left = step_cell<false, P, BLK, D2>(sd, cell, w, s_ctr);
  }
  if constexpr (in_fixed_point<P, 0>) leave(sd, t & 1, cell, left);
  flush_stats<BLK>(s_ctr, sd.ctr);
}

// The cells that k_batch_step left to the FP64 solve, over the lists of the lattices of its
// constraint system that have not reached their end time.
template <bool D2>
__global__ void __launch_bounds__(FP64_BLK, 1)
    k_batch_step_fp64(const BatchEntry* __restrict__ E, int nlat, int s) {
  constexpr int BLK = FP64_BLK;
  extern __shared__ double smem[];
  __shared__ unsigned int s_ctr[BLK / 32][CTR_N];  // a warp's, for one lattice at a time
  __shared__ Desc s_desc[BLK / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
  load_exp_table();
  cudaGridDependencySynchronize();
  const long long warps = (long long)gridDim.x * (BLK / 32);
  long long next = first_entry();  // this warp's next entry
  long long base = 0;              // entries of the lattices before j0
  for (int j0 = 0; j0 < nlat; j0 += 32) {
    const int j = j0 + lane;
    long long n = 0;
    if (j < nlat && (E[j].d.d2 != 0) == D2 && E[j].t0 + s < E[j].t_end) {
      const int odd = (E[j].t0 + s) & 1;
      n = (long long)E[j].d.ctr[CTR_REST + odd];
      if (blockIdx.x == 0 && warp == 0) clear_rest(E[j].d, !odd);
    }
    long long upto = n;  // entries of lattices j0 ... j
    for (int k = 1; k < 32; k *= 2) {
      const long long v = __shfl_up_sync(0xffffffffu, upto, k);
      if (lane >= k) upto += v;
    }
    const long long total = __shfl_sync(0xffffffffu, upto, 31);
    for (; next < base + total; next += warps) {
      const long long e = next - base;
      const int k = __ffs(__ballot_sync(0xffffffffu, upto > e)) - 1;
      const BatchEntry& b = E[j0 + k];
      const Rest r = b.d.rest[e - __shfl_sync(0xffffffffu, upto - n, k)];
      Desc& d = s_desc[warp];
      if (lane == 0) {
        d = b.d;
        d.t = b.t0 + s;
      }
      for (int i = lane; i < CTR_N; i += 32) s_ctr[warp][i] = 0;
      __syncwarp();
      if (r.bits >> lane & 1) {
        const long long cell = (long long)r.w * 32 + lane;
        WS<BLK> w{smem + threadIdx.x};
        if (d.t & 1) step_cell<true, double, BLK, D2, false, 0, false>(d, cell, w, s_ctr[warp]);
        else step_cell<false, double, BLK, D2, false, 0, false>(d, cell, w, s_ctr[warp]);
      }
      __syncwarp();
      for (int i = lane; i < CTR_N; i += 32)
        if (s_ctr[warp][i]) atomicAdd(d.ctr + i, (unsigned long long)s_ctr[warp][i]);
      __syncwarp();
    }
    base += total;
  }
}

// Boundary fills of the lattices that have freestream or outflow cells.
template <class P>
__global__ void __launch_bounds__(FILL_BLK, 6) k_batch_fill(const BatchEntry* __restrict__ E, const Tile* __restrict__ tiles,
                             int s) {
  const Tile tl = tiles[blockIdx.x];
  const BatchEntry& e = E[tl.lat];
  const long long t = e.t0 + s;
  if (t >= e.t_end) return;
  const long long cell = tl.cell0 + threadIdx.x;
  if (cell >= e.d.N) return;
  if (t & 1) fill_odd_cell<P>(e.d, cell);
  else fill_even_cell<P>(e.d, cell);
}

// After a launch sequence of n steps: every lattice's t0 moves on by n.
__global__ void k_batch_advance(BatchEntry* E, int nlat, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < nlat) E[j].t0 += n;
}

}  // namespace lbm39
