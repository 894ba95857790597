// FP64 Tsit5 instantiations with a lane per state component (gs_group.cuh).
#include "gs_group.cuh"

namespace gs {

cudaError_t launch_tsit5_group_forward(int problem, const FwdArgs& a, cudaStream_t s) {
  switch (problem) {
    case 0: return fwd_dispatch<Tsit5GroupMethod, LorenzGroup, double>(a, s);
    case 1: return fwd_dispatch<Tsit5GroupMethod, VanDerPolGroup, double>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_tsit5_group_reverse(int problem, const RevArgs& a, cudaStream_t s) {
  switch (problem) {
    case 0: return rev_dispatch<Tsit5GroupMethod, LorenzGroup, double>(a, s);
    case 1: return rev_dispatch<Tsit5GroupMethod, VanDerPolGroup, double>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gs
