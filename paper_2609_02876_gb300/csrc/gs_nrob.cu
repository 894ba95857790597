// Rodas5P instantiations for the neural Robertson (FP64): the per-lane form and,
// for small ensembles, the lane-group form.
#include "gs_kernels.cuh"

namespace gs {

// Rodas5P with stored stages for the lane-group form: a step's segment holds,
// besides its stage data, the network's activations at the eight stages, so the
// reverse sweep evaluates no network at all (a unit spent 116000 of its 209000
// cycles on the step's recompute). The lanes of a group write and read their own
// neurons' activations, 128 bytes in a row each time (from any 16-byte boundary);
// the leader writes the rest.
struct NrGroupMethod : Rodas5PMethod {
  using G = NeuralRobertsonGroup;
  static constexpr bool kDirect = true;
  static constexpr int D = 3, ACT = G::ACT;
  using Data = G::Data;
  template <class Pb, class R>
  struct StageData {
    Data d;
    G::Tape tape;
  };
  template <int>
  static constexpr int step_payload() {
    return NRG_STAGE_DOUBLES;
  }
  template <int>
  static constexpr int side_payload() {
    return NRG_STAGE_DOUBLES;
  }
  template <class Pb, class R>
  __device__ __forceinline__ static bool trial_s(const R (&y)[D], const R (&p)[Pb::NP], double h, const Carry<Pb, R>&,
                                                 R (&ynew)[D], R (&e)[D], Carry<Pb, R>&, StageData<Pb, R>& sd) {
    int piv[D];
    const bool ok = rodas_step<Pb>(y, p, h, sd.d.Y, sd.d.U, sd.d.LU, piv, sd.d.rinv, ynew, sd.tape);
#pragma unroll
    for (int c = 0; c < D; ++c) {
      e[c] = sd.d.U[7][c];
      sd.d.ynew[c] = ynew[c];
      sd.d.piv[c] = (double)piv[c];
    }
    return ok;
  }
  template <class SD>
  __device__ __forceinline__ static void store_stages(double* dst, const SD& sd) {
    const int i = G::me();
    Data d = sd.d;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      dst[32 * j + i] = sd.tape.F[j].h1;
      dst[32 * j + 16 + i] = sd.tape.F[j].h2;
      d.z3[j] = sd.tape.F[j].z3;
    }
    if (i == 0) {
      const double2* src = reinterpret_cast<const double2*>(&d);
      double2* o = reinterpret_cast<double2*>(dst + ACT);
#pragma unroll
      for (int w = 0; w < (int)(sizeof(Data) / sizeof(double2)); ++w) o[w] = src[w];
    }
  }
  template <class SD>
  __device__ __forceinline__ static void load_stages(const double* src, SD& sd) {
    const int i = G::me();
    const double2* o = reinterpret_cast<const double2*>(src + ACT);
    double2* d = reinterpret_cast<double2*>(&sd.d);
#pragma unroll
    for (int w = 0; w < (int)(sizeof(Data) / sizeof(double2)); ++w) d[w] = o[w];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      sd.tape.F[j].h1 = src[32 * j + i];
      sd.tape.F[j].h2 = src[32 * j + 16 + i];
      sd.tape.F[j].z3 = sd.d.z3[j];
    }
  }
  template <class Pb, class R, bool USER_COT, bool SOFT, class Acc>
  __device__ __forceinline__ static bool unit_stored(const RevArgs& a, long long k, int mode, bool active, int us,
                                                     const R (&x)[D], double h, const R (&p)[Pb::NP],
                                                     StageData<Pb, R>& sd, R (&lam)[D], Acc& pacc, double& loss) {
    const bool side = (mode == U_SIDE);
    double cv[D], v[D];
    int piv[D];
#pragma unroll
    for (int c = 0; c < D; ++c) piv[c] = (int)sd.d.piv[c];
    unit_cotangent<Pb, R, USER_COT>(a, k, active, side, us, sd.d.ynew, lam, cv, loss);
    rodas_reverse<Pb>(x, p, h, sd.d.Y, sd.d.U, sd.d.LU, piv, sd.d.rinv, cv, v, pacc, sd.tape);
#pragma unroll
    for (int c = 0; c < D; ++c) lam[c] = !active ? lam[c] : (side ? add_(lam[c], v[c]) : v[c]);
    return true;
  }
};

// The lane-group form (16 lanes per trajectory, gs_nrob.cuh) up to NR_GROUP_MAX
// trajectories, or NR_GROUP_STAGES_MAX where the record stores stages. Record +
// reverse, rtol 1e-6: up to 1216 trajectories (one group warp per FP64 unit) 30 ms
// with stored stages and 44 ms without, then 20 and 34 ms per 1000 (146 ms and
// 245 ms at 7168); the per-lane form 262 ms from 1 to 19456 trajectories.
bool group_launch(int64_t n, int stages) { return stages || n <= NR_GROUP_MAX; }

cudaError_t launch_nrob_forward(const FwdArgs& a, cudaStream_t s) {
  if (group_launch(a.n, a.stages)) return fwd_dispatch<NrGroupMethod, NeuralRobertsonGroup, double>(a, s);
  return fwd_dispatch<Rodas5PMethod, NeuralRobertson, double>(a, s);
}

cudaError_t launch_nrob_reverse(const RevArgs& a, cudaStream_t s) {
  if (group_launch(a.n, a.stages)) return rev_dispatch<NrGroupMethod, NeuralRobertsonGroup, double>(a, s);
  return rev_dispatch<Rodas5PMethod, NeuralRobertson, double>(a, s);
}

cudaError_t launch_nrob_refresh(const RevArgs& a, double* arena, double* y_final, const double* y0, cudaStream_t s) {
  return refresh_dispatch<Rodas5PMethod, NeuralRobertson, double>(a, arena, y_final, y0, s);
}

}  // namespace gs
