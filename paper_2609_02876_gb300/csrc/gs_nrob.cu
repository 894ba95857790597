// Rodas5P instantiations for the neural Robertson (FP64): the per-lane form and,
// for small ensembles, the lane-group form.
#include "gs_kernels.cuh"

namespace gs {

// Up to this many trajectories the neural Robertson takes its lane-group form
// (16 lanes per trajectory, gs_nrob.cuh). gs_solve_grad, record + reverse,
// measured at rtol 1e-6: the group form takes 44 ms up to 1216 trajectories
// (one warp per FP64 unit), then 34 ms per 1000 (280 ms at 8192); the per-lane
// form takes 263 ms from 1 to 19456 trajectories (its warp count).
constexpr int64_t NR_GROUP_MAX = 7168;

cudaError_t launch_nrob_forward(const FwdArgs& a, cudaStream_t s) {
  if (a.n <= NR_GROUP_MAX) return fwd_dispatch<Rodas5PMethod, NeuralRobertsonGroup, double>(a, s);
  return fwd_dispatch<Rodas5PMethod, NeuralRobertson, double>(a, s);
}

cudaError_t launch_nrob_reverse(const RevArgs& a, cudaStream_t s) {
  if (a.n <= NR_GROUP_MAX) return rev_dispatch<Rodas5PMethod, NeuralRobertsonGroup, double>(a, s);
  return rev_dispatch<Rodas5PMethod, NeuralRobertson, double>(a, s);
}

cudaError_t launch_nrob_refresh(const RevArgs& a, double* arena, double* y_final, const double* y0, cudaStream_t s) {
  return refresh_dispatch<Rodas5PMethod, NeuralRobertson, double>(a, arena, y_final, y0, s);
}

}  // namespace gs
