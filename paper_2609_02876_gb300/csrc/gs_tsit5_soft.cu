// FP64 Tsit5 instantiations in soft arithmetic (SoftD in gs_device.cuh).
#include "gs_kernels.cuh"

namespace gs {

cudaError_t launch_tsit5_soft_forward(int problem, const FwdArgs& a, cudaStream_t s) {
  switch (problem) {
    case 0: return fwd_dispatch<Tsit5Method, Lorenz, double, true>(a, s);
    case 1: return fwd_dispatch<Tsit5Method, VanDerPol, double, true>(a, s);
    case 4: return fwd_dispatch<Tsit5Method, Linear2, double, true>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_tsit5_soft_reverse(int problem, const RevArgs& a, cudaStream_t s) {
  switch (problem) {
    case 0: return rev_dispatch<Tsit5Method, Lorenz, double, true>(a, s);
    case 1: return rev_dispatch<Tsit5Method, VanDerPol, double, true>(a, s);
    case 4: return rev_dispatch<Tsit5Method, Linear2, double, true>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gs
