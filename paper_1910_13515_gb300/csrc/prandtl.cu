// prandtl.cu -- the step kernels with the Prandtl-number adjustment
// (lbm39_params.prandtl != 1): the same fused step as the paper's Pr = 1
// collision, with the quasi-equilibrium correction of g (kernels.cuh,
// relax_push<..., PR = true>), instantiated in a translation unit of their own
// so that the Pr = 1 kernels carry none of it and the library compiles in
// parallel.  These lattices always solve all 13 constraints (no z-mirror
// reduction).
#include <cuda_runtime.h>

#include "kernels.cuh"
#include "prandtl.h"

namespace lbm39 {

bool launch_step_prandtl(const Desc& d, bool odd, bool mixed, cudaStream_t stream) {
  if (mixed) launch_step<float, false, true, 0>(d, odd, stream);
  else launch_step<double, false, true, 0>(d, odd, stream);
  return cudaGetLastError() == cudaSuccess;
}

}  // namespace lbm39
