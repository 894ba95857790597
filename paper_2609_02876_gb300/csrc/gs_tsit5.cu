// Tsit5 (non-stiff) instantiations of the record and reverse-sweep kernels:
// Lorenz, Van der Pol and the linear test problem, FP64 and FP32-mixed.
#include "gs_kernels.cuh"

// The LV UDE reverse sweep's network: 0 (default) the warp-collective form
// (LvUdeWarp, mma.sync), 1 the CTA-collective form with the hidden layer on
// tcgen05 (LvUdeCta). Both give the same gradients to FP32 rounding (the UDE
// parity tests pass with either); measured at 2^18 trajectories the CTA form's
// reverse sweep takes 45.9 ms against 15.7 ms, because its four warps must meet
// at a CTA barrier and a tensor-memory round trip for each of the ~18
// hidden-layer products of a unit.
#ifndef GS_UDE_CTA
#define GS_UDE_CTA 0
#endif

namespace gs {

bool tsit5_supports(int problem, int precision) {
  if (problem == 5) return precision == 1;  // LV UDE: FP32 network and state, FP64 control
  return (problem == 0 || problem == 1 || problem == 4) && (precision == 0 || precision == 1);
}

// Other FP64 launches in soft arithmetic (SoftD, multiplications on the integer
// pipes): every ensemble of the two-dimensional problems, and ensembles of more
// than one warp per FP64 unit (four per SM: 19456 trajectories) of the three-dimensional
// ones. Gradient of n trajectories, record + reverse, hardware against soft:
// Lorenz 10007: 0.99 / 0.99 ms; 26000: 1.56 / 1.33; 60000: 3.07 / 2.37; 2^22:
// 151.7 / 120.4; Van der Pol 700: 2.26 / 2.12 ms; 26000: 3.44 / 2.87; 65521: 6.83
// / 5.01; 2^20: 73.1 / 53.5.
bool soft_launch(int problem, int precision, int64_t n) {
  return precision == 0 && (problem == 1 || problem == 4 || n > 4ll * sm_count() * 32);
}

// FP64 launches with a lane per state component (gs_group.cuh): Lorenz and Van
// der Pol up to 16 trajectories per FP64 unit, 9728 (Lorenz: two group warps per unit;
// Van der Pol: one). Gradient, record + reverse, per-lane against groups: Lorenz 1024:
// 0.96 / 0.64 ms; 9728: 0.99 / 0.85; 10007: 0.99 / 1.15 (some units hold three);
// Van der Pol 700: 2.12 / 1.95; 9728: 2.24 / 2.04; 14000: 2.26 / 2.64.
bool group_launch(int problem, int precision, int64_t n) {
  return precision == 0 && (problem == 0 || problem == 1) && n <= 4ll * sm_count() * 16;
}

cudaError_t launch_tsit5_forward(int problem, int precision, const FwdArgs& a, cudaStream_t s) {
  if (group_launch(problem, precision, a.n)) return launch_tsit5_group_forward(problem, a, s);
  if (soft_launch(problem, precision, a.n)) return launch_tsit5_soft_forward(problem, a, s);
  switch (problem * 2 + precision) {
    case 0: return fwd_dispatch<Tsit5Method, Lorenz, double>(a, s);
    case 1: return fwd_dispatch<Tsit5Method, Lorenz, float>(a, s);
    case 3: return fwd_dispatch<Tsit5Method, VanDerPol, float>(a, s);
    case 9: return fwd_dispatch<Tsit5Method, Linear2, float>(a, s);
    case 11: return fwd_dispatch<Tsit5Method, LvUde, float>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_tsit5_reverse(int problem, int precision, const RevArgs& a, cudaStream_t s) {
  if (a.k == 1 && group_launch(problem, precision, a.n)) return launch_tsit5_group_reverse(problem, a, s);
  if (a.k == 1 && soft_launch(problem, precision, a.n)) return launch_tsit5_soft_reverse(problem, a, s);
  switch (problem * 2 + precision) {
    case 0: return rev_dispatch<Tsit5Method, Lorenz, double>(a, s);
    case 1: return rev_dispatch<Tsit5Method, Lorenz, float>(a, s);
    case 2: return rev_many_dispatch<Tsit5Method, VanDerPol, double>(a, s);  // (k = 1: soft_launch)
    case 3: return rev_dispatch<Tsit5Method, VanDerPol, float>(a, s);
    case 8: return rev_many_dispatch<Tsit5Method, Linear2, double>(a, s);
    case 9: return rev_dispatch<Tsit5Method, Linear2, float>(a, s);
#if GS_UDE_CTA
    case 11: return rev_dispatch<Tsit5Method, LvUdeCta, float>(a, s);  // CTA-collective network (tcgen05)
#else
    case 11: return rev_dispatch<Tsit5Method, LvUdeWarp, float>(a, s);  // warp-collective network (mma.sync)
#endif
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_tsit5_refresh(int problem, int precision, const RevArgs& a, double* arena, double* y_final,
                                 const double* y0, cudaStream_t s) {
  switch (problem * 2 + precision) {
    case 0: return refresh_dispatch<Tsit5Method, Lorenz, double>(a, arena, y_final, y0, s);
    case 1: return refresh_dispatch<Tsit5Method, Lorenz, float>(a, arena, y_final, y0, s);
    case 2: return refresh_dispatch<Tsit5Method, VanDerPol, double>(a, arena, y_final, y0, s);
    case 3: return refresh_dispatch<Tsit5Method, VanDerPol, float>(a, arena, y_final, y0, s);
    case 8: return refresh_dispatch<Tsit5Method, Linear2, double>(a, arena, y_final, y0, s);
    case 9: return refresh_dispatch<Tsit5Method, Linear2, float>(a, arena, y_final, y0, s);
    case 11: return refresh_dispatch<Tsit5Method, LvUde, float>(a, arena, y_final, y0, s);
  }
  return cudaErrorInvalidValue;
}

int ude_max_warps() {
  int dev = 0, sms = 0, threads = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&threads, cudaDevAttrMaxThreadsPerMultiProcessor, dev);
  return (sms > 0 ? sms : 1) * (threads > 0 ? threads : 2048) / 32;
}

}  // namespace gs
