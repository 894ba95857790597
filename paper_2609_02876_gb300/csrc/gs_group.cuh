// Tsit5 with a lane per state component, for small FP64 ensembles of Lorenz and
// Van der Pol.
//
// A warp's FP64 instruction holds its SM quarter's FP64 unit for 64 cycles
// however many lanes are active, so below one warp per unit (19456
// trajectories) a launch's time is the instruction count of one step times the
// longest trajectory. Here a group of lanes (4 for Lorenz, 2 for Van der Pol)
// carries one trajectory: every lane holds the whole state and does the
// bookkeeping, but computes its own component's stage sums, slope, error and
// cotangent recursion, and the group exchanges each stage vector by shuffles. A
// Lorenz trial takes 63 FP64 instructions instead of 148, a reverse unit 70
// instead of 171 (Van der Pol 61 / 94 and 75 / 121). Every component's operations
// and their order are the per-lane form's: the results are the same bits.
// Measured at 1024 Lorenz trajectories: record 0.50 -> 0.32 ms, reverse sweep
// 0.46 -> 0.31 ms; what bounds it then is the warp's instruction chain (about
// 1300 instructions per trial, 8 cycles each with one warp per SM quarter).
#pragma once

#include "gs_kernels.cuh"

namespace gs {

// Lane q of the group's value.
template <int G>
__device__ __forceinline__ double group_get(double v, int q) {
  const unsigned mask = ((1u << G) - 1u) << (threadIdx.x & (32 - G));
  return __shfl_sync(mask, v, q, G);
}
template <int G, int D>
__device__ __forceinline__ void group_gather(double v, double (&o)[D]) {
#pragma unroll
  for (int c = 0; c < D; ++c) o[c] = group_get<G>(v, c);
}

// A group problem gives, for the lane's component c: f_own (its slope) and
// vjp_own (its component of J^T v, accumulating the lane's parameter gradient;
// parameter q belongs to lane owner(q)). The component selects are on integer
// pipes, which idle here.
struct LorenzGroup {
  using Lane = Lorenz;
  static constexpr int D = 3, NP = 3, kGroup = 4;
  // lane 0: the pb of rho, lane 1: of sigma (which needs y - x, as its slope does not), lane 2: of beta
  __device__ __forceinline__ static int owner(int q) { return q == 2 ? 2 : 1 - q; }
  __device__ __forceinline__ static double f_own(int c, const double (&y)[D], const double (&p)[NP]) {
    const double u = sub_(c == 0 ? y[1] : p[1], c == 0 ? y[0] : y[2]);          // y - x | rho - z
    const double m = mul_(c == 0 ? p[0] : p[2], c == 0 ? u : y[2]);             // sigma (y - x) | beta z
    const double r = fma_(y[0], c == 1 ? u : y[1], c == 1 ? -y[1] : -m);
    return c == 0 ? m : r;
  }
  __device__ __forceinline__ static double vjp_own(int c, const double (&y)[D], const double (&p)[NP],
                                                   const double (&v)[D], double& pb) {
    const double m = mul_(c == 0 ? p[0] : p[2], c == 0 ? v[0] : v[2]);          // sigma v0 | beta v2
    const double i = fma_(c == 0 ? y[1] : y[0], c == 2 ? v[1] : v[2], c == 0 ? -m : (c == 1 ? -v[1] : m));
    const double u = sub_(c == 0 ? p[1] : y[1], c == 0 ? y[2] : y[0]);          // rho - z | y - x
    const double r = fma_(c == 0 ? u : p[0], c == 0 ? v[1] : v[0], i);
    pb = fma_(c == 1 ? u : (c == 0 ? y[0] : -y[2]), c == 1 ? v[0] : (c == 0 ? v[1] : v[2]), pb);
    return c == 2 ? -i : r;
  }
};

struct VanDerPolGroup {
  using Lane = VanDerPol;
  static constexpr int D = 2, NP = 1, kGroup = 2;
  __device__ __forceinline__ static int owner(int) { return 1; }
  __device__ __forceinline__ static double f_own(int c, const double (&y)[D], const double (&p)[NP]) {
    const double g = mul_(p[0], fma_(fma_(-y[0], y[0], 1.0), y[1], -y[0]));
    return c == 0 ? y[1] : g;
  }
  __device__ __forceinline__ static double vjp_own(int c, const double (&y)[D], const double (&p)[NP],
                                                   const double (&v)[D], double& pb) {
    const double w = fma_(-y[0], y[0], 1.0);
    const double mv = mul_(p[0], v[1]);
    const double t = fma_(c == 0 ? add_(y[0], y[0]) : w, y[1], c == 0 ? 1.0 : -y[0]);  // 2 x v + 1 | (1 - x^2) v - x
    const double r = fma_(mv, c == 0 ? t : w, c == 0 ? -0.0 : v[0]);  // (a product plus -0 is the product)
    pb = fma_(t, v[1], pb);
    return c == 0 ? -r : r;
  }
};

// Each lane's share of theta_bar: the sum of the parameter it owns.
template <class Pb>
struct GroupAcc {
  double s;
  __device__ void zero() { s = 0.0; }
  __device__ double get(int q) const { return group_get<Pb::kGroup>(s, Pb::owner(q)); }
};
template <>
struct GroupAccOf<LorenzGroup> {
  using type = GroupAcc<LorenzGroup>;
};
template <>
struct GroupAccOf<VanDerPolGroup> {
  using type = GroupAcc<VanDerPolGroup>;
};

struct Tsit5GroupMethod {
  using LaneMethod = Tsit5Method;
  static constexpr int ORDER = Tsit5Method::ORDER, ERR_ORDER = Tsit5Method::ERR_ORDER;
  static constexpr bool kStages = true, kControl64 = true, kSoft = false, kCarryIsF = true;
  static constexpr int REV_MINB_F32 = 0, REV_MINB_STAGES = 0;
  static constexpr double IDLE_H = 0.0;

  template <class Pb, class R>
  struct Carry {
    double k;  // the lane's component of f(y)
  };
  template <class Pb>
  __device__ __forceinline__ static int own() {
    const int c = threadIdx.x & (Pb::kGroup - 1);
    return c < Pb::D ? c : Pb::D - 1;  // a lane without a component repeats the last one
  }
  template <class Pb>
  __device__ __forceinline__ static double own(const double (&x)[Pb::D]) {
    const int c = own<Pb>();
    double v = x[0];
#pragma unroll
    for (int q = 1; q < Pb::D; ++q) v = c == q ? x[q] : v;
    return v;
  }
  template <class Pb, class R, class Get>
  __device__ __forceinline__ static void set_carry_f(Carry<Pb, R>& cy, Get f) {
    cy.k = f(own<Pb>());
  }
  template <class Pb, class R>
  __device__ __forceinline__ static void start(const double (&y)[Pb::D], const double (&p)[Pb::NP], Carry<Pb, R>& cy,
                                               float (&f0)[Pb::D]) {
    double f[Pb::D];
    Pb::Lane::f(y, p, f);
    cy.k = own<Pb>(f);
#pragma unroll
    for (int c = 0; c < Pb::D; ++c) f0[c] = (float)f[c];
  }

  // tsit5_stages for the lane's component: Y[1..6] gathered, K its own slopes.
  template <class Pb, int KN>
  __device__ __forceinline__ static void stages(const double (&y)[Pb::D], const double (&p)[Pb::NP], double h,
                                                double (&Y)[7][Pb::D], double (&K)[7]) {
    constexpr int D = Pb::D;
    const int c = own<Pb>();
    const double yc = own<Pb>(y);
#pragma unroll
    for (int q = 0; q < D; ++q) Y[0][q] = y[q];
#pragma unroll
    for (int i = 1; i < 7; ++i) {
      double s = mul_(tsit5::A(i, 0), K[0]);
#pragma unroll
      for (int j = 1; j < i; ++j) s = fma_(tsit5::A(i, j), K[j], s);
      group_gather<Pb::kGroup, D>(fma_(h, s, yc), Y[i]);
      if (i < 6 || KN == 7) K[i] = Pb::f_own(c, Y[i], p);
    }
  }
  template <class Pb>
  __device__ __forceinline__ static void trial_y(const double (&y)[Pb::D], const double (&p)[Pb::NP], double h,
                                                 double k1, double (&Y)[7][Pb::D], double (&e)[Pb::D], double& k7) {
    double K[7];
    K[0] = k1;
    stages<Pb, 7>(y, p, h, Y, K);
    double s = mul_(tsit5::Btilde(0), K[0]);
#pragma unroll
    for (int j = 1; j < 7; ++j) s = fma_(tsit5::Btilde(j), K[j], s);
    group_gather<Pb::kGroup, Pb::D>(mul_(h, s), e);
    k7 = K[6];
  }
  template <class Pb, class R>
  __device__ __forceinline__ static bool trial(const double (&y)[Pb::D], const double (&p)[Pb::NP], double h,
                                               const Carry<Pb, R>& cy, double (&ynew)[Pb::D], double (&e)[Pb::D],
                                               Carry<Pb, R>& next) {
    double Y[7][Pb::D];
    trial_y<Pb>(y, p, h, cy.k, Y, e, next.k);
#pragma unroll
    for (int c = 0; c < Pb::D; ++c) ynew[c] = Y[6][c];
    return true;
  }

  // Stored stages: Tsit5Method's layout.
  template <class Pb, class R>
  using StageData = Tsit5Method::StageData<Pb, R>;
  template <int D>
  static constexpr int step_payload() {
    return Tsit5Method::step_payload<D>();
  }
  template <int D>
  static constexpr int side_payload() {
    return Tsit5Method::side_payload<D>();
  }
  template <class Pb, class R>
  __device__ __forceinline__ static bool trial_s(const double (&y)[Pb::D], const double (&p)[Pb::NP], double h,
                                                 const Carry<Pb, R>& cy, double (&ynew)[Pb::D], double (&e)[Pb::D],
                                                 Carry<Pb, R>& next, StageData<Pb, R>& sd) {
    trial_y<Pb>(y, p, h, cy.k, sd.Y, e, next.k);
#pragma unroll
    for (int c = 0; c < Pb::D; ++c) ynew[c] = sd.Y[6][c];
    return true;
  }
  template <class Pb, class R, class W>
  __device__ __forceinline__ static void pack(const StageData<Pb, R>& sd, bool side, W&& write) {
    Tsit5Method::pack<Pb, R>(sd, side, write);
  }
  template <class Pb, class R, class Rd>
  __device__ __forceinline__ static void unpack(bool side, const double (&x)[Pb::D], Rd&& read, StageData<Pb, R>& sd) {
    Tsit5Method::unpack<Pb, R>(side, x, read, sd);
  }

  // tsit5_reverse for the lane's component.
  template <class Pb, class Acc>
  __device__ __forceinline__ static void reverse(const double (&Y)[7][Pb::D], const double (&p)[Pb::NP], double h,
                                                 const double (&cv)[Pb::D], double (&v)[Pb::D], Acc& pacc) {
    constexpr int D = Pb::D, G = Pb::kGroup;
    const int c = own<Pb>();
    const double co = own<Pb>(cv);
    double acc[6], vo = co;
#pragma unroll
    for (int j = 5; j >= 0; --j) {
      const double b = (j == 5) ? mul_(tsit5::B(j), co) : fma_(tsit5::B(j), co, acc[j]);
      double kb[D];
      group_gather<G, D>(mul_(h, b), kb);
      const double yb = Pb::vjp_own(c, Y[j], p, kb, pacc.s);
      vo = add_(vo, yb);
#pragma unroll
      for (int l = 0; l < j; ++l)
        acc[l] = (j == 5) ? mul_(tsit5::A(j, l), yb) : fma_(tsit5::A(j, l), yb, acc[l]);
    }
    group_gather<G, D>(vo, v);
  }
  template <class Pb, class R, bool USER_COT, bool SOFT, class Acc>
  __device__ __forceinline__ static bool unit_stored(const RevArgs& a, long long k, int mode, bool active, int us,
                                                     const R (&x)[Pb::D], double h, const R (&p)[Pb::NP],
                                                     const StageData<Pb, R>& sd, R (&lam)[Pb::D], Acc& pacc,
                                                     double& loss) {
    constexpr int D = Pb::D;
    const bool side = (mode == U_SIDE);
    double cv[D], v[D];
    unit_cotangent<Pb, R, USER_COT>(a, k, active, side, us, sd.Y[6], lam, cv, loss);
    reverse<Pb>(sd.Y, p, h, cv, v, pacc);
#pragma unroll
    for (int c = 0; c < D; ++c) lam[c] = !active ? lam[c] : (side ? add_(lam[c], v[c]) : v[c]);
    return true;
  }
  template <class Pb, class R, bool USER_COT, bool SOFT, class Acc>
  __device__ __forceinline__ static bool unit(const RevArgs& a, long long k, int mode, bool active, int us,
                                              const R (&x)[Pb::D], double h, const R (&p)[Pb::NP], R (&lam)[Pb::D],
                                              Acc& pacc, double& loss, R (&ynew)[Pb::D]) {
    StageData<Pb, R> sd;
    double K[7];
    K[0] = Pb::f_own(own<Pb>(), x, p);
    stages<Pb, 6>(x, p, h, sd.Y, K);
#pragma unroll
    for (int c = 0; c < Pb::D; ++c) ynew[c] = sd.Y[6][c];
    return unit_stored<Pb, R, USER_COT, SOFT>(a, k, mode, active, us, x, h, p, sd, lam, pacc, loss);
  }
};

}  // namespace gs
