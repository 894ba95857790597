// FP32-mixed Tsit5 record and reverse sweep over packed segments, for the
// workspaces of gs_solve_grad (whose records no other call reads).
//
// The general kernels keep a state of doubles per accepted step (48 bytes for
// Lorenz), staged through shared memory. The mixed form's state is FP32 and its
// kernels are bound by instruction issue and by the sweep's scattered segment
// reads, so here a segment is one 32-byte DRAM sector, [t (FP64) | h (FP32, as the
// stages use it) | previous segment (32 bits) | y (FP32)], written and read by one
// 256-bit access straight from registers: no conversions, no staging, no 64-bit
// index arithmetic. The arithmetic of steps, control and sweep is the general
// kernels', operation by operation; results are the same bits (a state below the
// FP32 normal range excepted, which the general segment flushes to zero). Lorenz
// 2^24 in chunks of 2^21: record 17.4 -> 9.3 ms, sweep 21.9 -> 15.5 ms; Van der Pol
// 10^6 at rtol 1e-4: 1.02 -> 0.55 and 1.57 -> 1.08 ms.
//
// Per-trajectory work (writing results, taking the next trajectory) is warp code
// that few lanes need at a time, with FP64 conversions that hold the SM quarter's
// FP64 unit for 64 cycles each: a warp does it when BATCH lanes wait for it, or
// when it has nothing else to do.
#pragma once

#include "gs_kernels.cuh"

namespace gs {

constexpr int PACKED_SEGW = PACKED_SEGW_HOST;

struct PackedSeg {
  double t;
  float h;
  int prev;
  float y[3];
};
__device__ __forceinline__ void store_seg(double* arena, unsigned idx, const PackedSeg& s) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(arena + (size_t)idx * PACKED_SEGW),
               "r"(__double2loint(s.t)), "r"(__double2hiint(s.t)), "r"(__float_as_int(s.h)), "r"(s.prev),
               "r"(__float_as_int(s.y[0])), "r"(__float_as_int(s.y[1])), "r"(__float_as_int(s.y[2])), "r"(0)
               : "memory");
}
__device__ __forceinline__ PackedSeg load_seg(const double* arena, unsigned idx) {
  int r[8];
  asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(arena + (size_t)idx * PACKED_SEGW)
               : "memory");
  return {__hiloint2double(r[1], r[0]), __int_as_float(r[2]), r[3],
          {__int_as_float(r[4]), __int_as_float(r[5]), __int_as_float(r[6])}};
}

// to_f of a positive double: one subtraction and one shift inside the float
// normal range, the general form outside it.
__device__ __forceinline__ float to_f_pos(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), e = hi - 0x38000000u;  // exponent rebased by 896
  if (e - 0x00100000u < 0x0fe00000u) return __int_as_float((int)__funnelshift_l((unsigned)__double2loint(x), e, 3));
  return to_f(x);
}
// to_d of a positive normal float.
__device__ __forceinline__ double to_d_pos(float x) {
  const unsigned u = __float_as_uint(x);
  return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}

template <class Pb, bool C64, int BATCH>
__global__ void __launch_bounds__(TPB_FWD) record_packed_kernel(const FwdArgs a) {
  using M = Tsit5Method;
  using R = float;
  constexpr int D = Pb::D, NP = Pb::NP;
  static_assert(D <= 3, "a packed segment holds three states");
  using Carry = typename M::template Carry<Pb, R>;
  const long long n = a.n;
  const double t1 = a.t1;
  const double sliver = 1e-12 * fmax(1.0, fabs(t1));
  const long long key_end = dkey(t1 - sliver);
  const float rtf = (float)a.rtol, atf = (float)a.atol;
  // no step below it passes the step-size floor anywhere in the span
  const float h_floor = 1e-14f * fmaxf(1.0f, fmaxf(fabsf(to_f(a.t0)), fabsf(to_f(t1))));
  const int max_steps = a.max_steps < 0x7fffffff ? (int)a.max_steps : 0x7fffffff;
  long long k = -1;
  bool drained = false;
  double t = 0.0, h = 0.0;
  float hf = 0.0f;
  R y[D], p[NP];
  Carry cy;
  int S = 0, natt = 0, status = TRAJ_OK, prev = -1;
  bool rej = false, ended = false;
  unsigned res_next = 0, res_end = 0;  // this warp's reserved arena slots (warp-uniform)
  const unsigned cap = (unsigned)a.arena_cap;

  for (;;) {
    // ---- finished lanes write their results, free lanes take the next trajectory
    const bool wait = k >= 0 ? ended : !drained;
    const unsigned wm = __ballot_sync(FULL_MASK, wait);
    if (wm) {
      const unsigned busy = __ballot_sync(FULL_MASK, k >= 0 && !ended);
      if (__popc(wm) >= BATCH || busy == 0) {
        if (k >= 0 && ended) {
          a.head[k] = prev;
          a.S[k] = S;
          a.natt[k] = natt;
          a.status[k] = status;
#pragma unroll
          for (int c = 0; c < D; ++c) a.y_final[c * n + k] = (double)y[c];
          if (a.step_counts) {
            a.step_counts[k] = S;
            a.step_counts[n + k] = natt;
          }
          if (status != TRAJ_OK) *a.any_failed = 1;
          k = -1;
        }
        const bool need = k < 0 && !drained;
        const long long got = warp_ticket(a.work, need);
        if (need) {
          if (got < n) {
            k = got;
            bool fin = true;
            float yf[D], pf[NP], ff[D];
            double yd[D], pd[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) {
              pd[q] = a.params[q * n + k];
              p[q] = pf[q] = (R)pd[q];
              fin = fin && finite_d(pd[q]);
            }
#pragma unroll
            for (int c = 0; c < D; ++c) {
              yd[c] = a.y0[c * n + k];
              y[c] = yf[c] = (R)yd[c];
              fin = fin && finite_d(yd[c]);
            }
            t = a.t0;
            S = natt = 0;
            status = TRAJ_OK;
            rej = false;
            prev = -1;
            M::template start<Pb, R>(y, p, cy, ff);
            if (a.h0 > 0.0) {
              h = a.h0;
            } else if (a.h0_pre) {
              h = a.y_final[k];
            } else if constexpr (C64) {
              double fd[D];
              Pb::f(yd, pd, fd);
              h = initial_step_f64<Pb, M::ORDER>(yd, pd, fd, a.t0, t1, a.rtol, a.atol);
            } else {
              h = initial_step_f32<Pb, M::ORDER>(yf, pf, ff, a.t0, t1, a.rtol, a.atol);
            }
            fin = fin && positive(h) && finite_nonneg(h);
            hf = to_f(h);
            ended = !fin;
            if (!fin) status = TRAJ_NONFINITE;
          } else {
            drained = true;
          }
        }
      }
    }
    if (!__any_sync(FULL_MASK, k >= 0)) {
      if (__all_sync(FULL_MASK, drained)) break;
      continue;
    }

    // ---- a trial step for every lane with a trajectory under way
    bool run = k >= 0 && !ended;
    if (run && natt >= max_steps) {
      status = TRAJ_MAXSTEPS;
      ended = true;
      run = false;
    }
    const double tsum = add_(t, h);
    const bool last = run && dkey(tsum) >= key_end;
    if (__any_sync(FULL_MASK, last)) {
      if (last) {
        h = sub_(t1, t);
        hf = to_f(h);
      }
    }
    __syncwarp();
    R yn[D], e[D];
    Carry next;
    bool accept = false;
    double qd = 2.0;
    float q = 2.0f;
    if (run) {
      R Y[7][D], K[7][D];
      typename TapeOf<Pb>::type tape;
#pragma unroll
      for (int c = 0; c < D; ++c) K[0][c] = cy.k1[c];
      tsit5_stages<Pb, R, 7>(y, p, hf, Y, K, tape);
      tsit5_error<Pb, R>(K, hf, e);
#pragma unroll
      for (int c = 0; c < D; ++c) {
        yn[c] = Y[6][c];
        next.k1[c] = K[6][c];
      }
      ++natt;
      if constexpr (C64) {
        qd = err_meansq_f64<D>(e, y, yn, a.rtol, a.atol);
        accept = rms_le_one(qd);
      } else {
        q = err_meansq_f32<D>(e, y, yn, rtf, atf);
        accept = q <= 1.0f;  // (NaN rejects)
      }
    }
    // ---- segment of the accepted step, from the warp's reserved slots
    const unsigned fm = __ballot_sync(FULL_MASK, accept);
    if (fm) {
      const int cnt = __popc(fm), rem = (int)(res_end - res_next);
      unsigned nb = 0;
      if (cnt > rem) {
        unsigned long long base = 0;
        if (lane_id() == 0) base = atomicAdd(a.arena_top, (unsigned long long)a.arena_block);
        base = __shfl_sync(FULL_MASK, base, 0);
        nb = base < 0x7ffff000ull ? (unsigned)base : 0x7ffff000u;  // (past any capacity)
      }
      const int rank = __popc(fm & ((1u << lane_id()) - 1u));
      const unsigned idx = rank < rem ? res_next + rank : nb + (rank - rem);
      if (cnt > rem) {
        res_next = nb + (cnt - rem);
        res_end = nb + (unsigned)a.arena_block;
      } else {
        res_next += cnt;
      }
      if (accept) {
        if (idx < cap)
          store_seg(a.arena, idx, PackedSeg{t, hf, prev, {y[0], y[1], D > 2 ? y[D - 1] : 0.0f}});
        else
          *a.overflow = 1;
        prev = (int)idx;
        t = last ? t1 : tsum;
#pragma unroll
        for (int c = 0; c < D; ++c) y[c] = yn[c];
        cy = next;
        ++S;
        ended = last;
      }
    }
    // ---- step-size control (as in the general record kernel)
    if (run && !ended) {
      bool under, nf;
      if constexpr (C64) {
        nf = !finite_nonneg(qd);
        double fac = nf ? 0.2 : ctrl_factor_ms_f64<M::ERR_ORDER>(qd);
        if (accept && rej) fac = fmin(fac, 1.0);
        h = mul_(h, fac);
        hf = to_f(h);
        under = fabs(h) < mul_(1e-14, fmax(1.0, fabs(t)));
      } else {
        nf = !(q < __int_as_float(0x7f800000));
        float fac = nf ? 0.2f : ctrl_factor_f32<M::ERR_ORDER>(q);
        if (accept && rej) fac = fminf(fac, 1.0f);
        h = mul_(h, to_d_pos(fac));
        hf = to_f_pos(h);
        under = false;
        if (hf < h_floor) under = hf < 1e-14f * fmaxf(1.0f, fabsf(to_f(t)));
      }
      rej = !accept;
      if (under) {
        status = (!accept && nf) ? TRAJ_NONFINITE : TRAJ_DT_UNDERFLOW;
        ended = true;
      }
    }
  }
}

// Reverse sweep over packed segments, built-in loss.
template <class Pb, int BATCH>
__global__ void __launch_bounds__(TPB_REV, 8) reverse_packed_kernel(const RevArgs a) {
  using R = float;
  constexpr int D = Pb::D, NP = Pb::NP;
  extern __shared__ double s_save[];
  const int ns = a.n_save;
  for (int i = threadIdx.x; i < ns; i += blockDim.x) s_save[i] = a.save_t[i];
  __syncthreads();

  const long long n = a.n;
  constexpr long long NO_SAVE = (long long)0x8000000000000000ull;  // below the key of every time
  long long k = -1, key_s = NO_SAVE;                                // key_s: the key of save js
  bool drained = false;
  int end = 0;  // 1: swept, 2: inconsistent record
  R p[NP], lam[D], yx[D];
  CompensatedAcc<NP> pacc;
  double loss = 0.0, tx = 0.0;
  int seg = -1, js = -1, segs_left = 0;
  const unsigned cap = (unsigned)a.arena_cap;

  // saves on the mesh point (tx, yx): their cotangent and loss terms
  auto saves_here = [&]() {
    const long long key_tx = dkey(tx);
    while (key_s == key_tx) {
#pragma unroll
      for (int c = 0; c < D; ++c) {
        lam[c] = add_(lam[c], add_(yx[c], yx[c]));
        loss = acc_loss(loss, mul_(yx[c], yx[c]));
      }
      --js;
      key_s = js >= 0 ? dkey(s_save[js]) : NO_SAVE;
    }
    return key_tx;
  };

  for (;;) {
    // ---- swept lanes write their gradients, free lanes take the next trajectory
    const bool wait = k >= 0 ? end != 0 : !drained;
    const unsigned wm = __ballot_sync(FULL_MASK, wait);
    if (wm) {
      const unsigned busy = __ballot_sync(FULL_MASK, k >= 0 && end == 0);
      if (__popc(wm) >= BATCH || busy == 0) {
        if (k >= 0 && end != 0) {
          if (end == 1)
            write_grad<NP, D, R>(a, k, pacc, lam, loss);
          else
            write_nan<NP, D>(a, k);
          k = -1;
        }
        const bool need = k < 0 && !drained;
        const long long got = warp_ticket(a.work, need);
        if (need) {
          if (got < n) {
            const long long hd = a.head[got];
            if (a.status[got] != TRAJ_OK || hd < 0) {
              write_nan<NP, D>(a, got);  // (takes another ticket next time)
            } else {
              k = got;
              end = 0;
#pragma unroll
              for (int q = 0; q < NP; ++q) p[q] = (R)a.params[q * n + k];
#pragma unroll
              for (int c = 0; c < D; ++c) {
                lam[c] = R(0);
                yx[c] = (R)a.y_final[c * n + k];
              }
              pacc.zero();
              loss = 0.0;
              tx = a.t1;
              seg = (int)hd;
              segs_left = a.S[k];
              js = ns - 1;
              key_s = js >= 0 ? dkey(s_save[js]) : NO_SAVE;
              saves_here();
            }
          } else {
            drained = true;
          }
        }
      }
    }
    if (!__any_sync(FULL_MASK, k >= 0)) {
      if (__all_sync(FULL_MASK, drained)) break;
      continue;
    }

    // ---- this lane's unit: a side step to a save after (tx, yx), else the next segment's step
    bool unit = false, side = false;
    float hf = 0.0f;
    if (k >= 0 && end == 0) {
      const long long key_tx = saves_here();
      if (key_s > key_tx) {
        side = unit = true;
      } else if (seg < 0) {
        end = segs_left == 0 ? 1 : 2;
      } else if ((unsigned)seg >= cap || segs_left <= 0) {
        end = 2;
      } else {
        const PackedSeg s = load_seg(a.arena, (unsigned)seg);
        seg = s.prev;
        tx = s.t;
        hf = s.h;
#pragma unroll
        for (int c = 0; c < D; ++c) yx[c] = s.y[c];
        --segs_left;
        unit = true;
      }
    }
    __syncwarp();
    if (__any_sync(FULL_MASK, side)) {
      if (side) {
        hf = to_f(sub_(s_save[js], tx));
        --js;
        key_s = js >= 0 ? dkey(s_save[js]) : NO_SAVE;
      }
    }
    if (unit) {
      R Y[7][D], K[7][D], cv[D], v[D];
      typename TapeOf<Pb>::type tape;
      Pb::f(yx, p, K[0]);
      tsit5_stages<Pb, R, 6>(yx, p, hf, Y, K, tape);
      unit_cotangent<Pb, R, false>(a, k, true, side, 0, Y[6], lam, cv, loss);
      tsit5_reverse<Pb, R>(Y, p, hf, cv, v, pacc, tape);
#pragma unroll
      for (int c = 0; c < D; ++c) lam[c] = side ? add_(lam[c], v[c]) : v[c];
    }
  }
}

}  // namespace gs
