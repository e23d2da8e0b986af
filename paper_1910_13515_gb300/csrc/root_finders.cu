// root_finders.cu -- the FP64 step kernels with the other root finders of the
// constraint equations (lbm39_params.root_finder): 1, the chord-Newton hybrid
// (cell.cuh newton_chord); 2, Newton with a single-precision direction
// (cell.cuh newton<BLK, true>); 3, that after a single-precision start
// (cell.cuh start32).  The same fused step with another solver,
// instantiated in a translation unit of its own so that the Newton kernels are
// untouched and the library compiles in parallel.
#include <cuda_runtime.h>

#include "kernels.cuh"
#include "root_finders.h"

namespace lbm39 {

namespace {
template <int SOLVER>
void launch(const Desc& d, bool odd, cudaStream_t stream) {
  if (d.d2) launch_step<double, true, false, SOLVER>(d, odd, stream);
  else launch_step<double, false, false, SOLVER>(d, odd, stream);
}
}  // namespace

bool launch_step_root_finder(const Desc& d, bool odd, int solver, cudaStream_t stream) {
  if (solver == 1) launch<1>(d, odd, stream);
  else if (solver == 2) launch<2>(d, odd, stream);
  else if (solver == 3) launch<3>(d, odd, stream);
  else return false;
  return cudaGetLastError() == cudaSuccess;
}

}  // namespace lbm39
