// FP32-mixed Tsit5 over packed segments (gs_packed.cuh): Lorenz, Van der Pol and
// the linear test problem.
#include "gs_packed.cuh"

namespace gs {
namespace {

// Lanes a warp lets wait before it runs its per-trajectory code. Lorenz 2^24,
// record / sweep in ms: 12.3 / 17.8 with 1, 10.4 / 16.4 with 2, 9.6 / 15.8 with 3,
// 9.3 / 15.5 with 4, 9.3 / 15.5 with 8.
constexpr int BATCH = 4;

template <class Pb>
cudaError_t forward(const FwdArgs& a_in, cudaStream_t s) {
  FwdArgs a = a_in;
  cudaError_t e = cudaSuccess;
  a.h0_pre = 0;
  if (a.control)
    init_step_pass<Tsit5Method, Pb, float, true>(a, s, &e);
  else
    init_step_pass<Tsit5Method, Pb, float, false>(a, s, &e);
  if (e != cudaSuccess) return e;
  if (a.control) return persistent_launch(record_packed_kernel<Pb, true, BATCH>, TPB_FWD, 0, a.n, s, &a);
  return persistent_launch(record_packed_kernel<Pb, false, BATCH>, TPB_FWD, 0, a.n, s, &a);
}

template <class Pb>
cudaError_t reverse(const RevArgs& a, cudaStream_t s) {
  const size_t smem = (size_t)((a.n_save + 1) & ~1) * sizeof(double);
  return persistent_launch(reverse_packed_kernel<Pb, BATCH>, TPB_REV, smem, a.n, s, &a);
}

}  // namespace

bool packed_supports(int problem) { return problem == 0 || problem == 1 || problem == 4; }

cudaError_t launch_packed_forward(int problem, const FwdArgs& a, cudaStream_t s) {
  if (a.segw != PACKED_SEGW || a.k != 1 || a.y_save) return cudaErrorInvalidValue;
  switch (problem) {
    case 0: return forward<Lorenz>(a, s);
    case 1: return forward<VanDerPol>(a, s);
    case 4: return forward<Linear2>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_packed_reverse(int problem, const RevArgs& a, cudaStream_t s) {
  if (a.segw != PACKED_SEGW || a.k != 1 || a.y_save_bar) return cudaErrorInvalidValue;
  switch (problem) {
    case 0: return reverse<Lorenz>(a, s);
    case 1: return reverse<VanDerPol>(a, s);
    case 4: return reverse<Linear2>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gs
