// rrg_lane.cuh -- device code shared by the single-problem kernels
// (rrg_kernels.cu) and the batched kernels (rrg_batch.cu): the trajectory
// loop with its constraint check, the binary64 re-run from Philox counters,
// the equilibrium solve of the steady-state check, per-scenario model
// constants and the k-section grids.
#pragma once

#include <cfloat>
#include <cmath>

#include "rrg_device.cuh"
#include "rrg_internal.h"

namespace rrg {

template <typename T> __device__ __forceinline__ T max_finite();
template <> __device__ __forceinline__ float max_finite<float>() { return FLT_MAX; }
template <> __device__ __forceinline__ double max_finite<double>() { return DBL_MAX; }
template <typename T> __device__ __forceinline__ T inf_v();
template <> __device__ __forceinline__ float inf_v<float>() { return __int_as_float(0x7f800000); }
template <> __device__ __forceinline__ double inf_v<double>() { return __longlong_as_double(0x7ff0000000000000ll); }

// ---------------------------------------------------------------------------
// Equilibrium manifold (Sec. II-A).  At rest the cathode balance fixes the
// cathode gauge pressure from the air flow W, the orifice fixes the supply
// manifold pressure and the compressor map the speed, leaving the shaft
// torque balance g(W) = 0, with g decreasing in W and g(W_o2) > 0.  The root
// lies close to the controller's target flow W_ref = lam_ref W_o2 / x_O2, so
// a secant iteration started there converges in a handful of binary64
// evaluations; every iterate is kept inside a sign-change bracket and a
// step that leaves it is replaced by bisection.
template <typename T>
__device__ __forceinline__ T eq_torque(const Fc3K<T>& K, const CandK<T>& C, T inv_k_ca, T inv_k_sm, T a_p,
                       T inv_a_w, T W, T q[3]) {
  q[0] = (W - C.W_o2) * inv_k_ca;
  q[2] = q[0] + W * inv_k_sm;
  q[1] = (W + a_p * q[2]) * inv_a_w;
  T a, b, c;
  fc3_rhs<T>(K, C, q[0], q[1], q[2], a, b, c);
  return b;
}

template <typename T> __device__ __forceinline__ T eq_tol();
template <> __device__ __forceinline__ double eq_tol<double>() { return 1e-15; }
// binary32: the screen only needs y_ss to about 1e-5 (it defers to binary64
// within 1e-4 of the threshold); a tighter stop can stall on rounding noise
// and run every iteration.
template <> __device__ __forceinline__ float eq_tol<float>() { return 1e-6f; }

// Returns 0 and the gauge state q at the equilibrium (C: W_o2 and V0; xs: the
// first guess), or < 0.  One evaluation site: the stages of the iteration (the
// sign at W_o2, two points around the target flow, the bracket's upper end,
// secants) only choose the next flow.
template <typename T>
__device__ __forceinline__ int equilibrium_solve(const Fc3K<T>& K, const CandK<T>& C, T guess, T q[3]) {
  // reciprocals in the solve's own precision (binary32 divisions in the
  // binary32 screen, none of GB300's slow binary64 ones)
  const T ikca = T(1) / K.k_ca, iksm = T(1) / K.k_sm;
  const T a_p = K.a_p, iaw = T(1) / K.a_w;
  const T big = static_cast<T>(1e30);
  T lo = C.W_o2, hi = big, x = lo;
  T x0 = guess, g0 = T(0), x1 = T(0), g1 = T(0);
  int stage = 0, n = 0;
#pragma unroll 1
  for (;;) {
    const T g = eq_torque<T>(K, C, ikca, iksm, a_p, iaw, x, q);
    if (stage == 0) {
      if (!(g > T(0))) return -2;
      x = x0;
      stage = 1;
      continue;
    }
    if (stage == 1) {
      g0 = g;
      if (g > T(0)) lo = x; else hi = x;
      x = x0 * (g > T(0) ? T(1.001) : T(0.999));
      stage = 2;
      continue;
    }
    if (stage == 2) {
      x1 = x;
      g1 = g;
      if (g > T(0)) { if (x > lo) lo = x; } else if (x < hi) hi = x;
      stage = 3;
    } else if (stage == 3) {  // closing the bracket before bisection can be needed
      if (g > T(0)) lo = x; else hi = x;
      if (++n >= 60 && hi == big) return -2;
    } else {
      if (g == T(0)) return 0;
      if (g > T(0)) lo = x; else hi = x;
      if (fabs(x - x1) <= eq_tol<T>() * x || hi - lo <= T(0.4) * eq_tol<T>() * hi) return 0;
      x0 = x1; g0 = g1;
      x1 = x; g1 = g;
      if (++n >= 100) return 0;
    }
    if (hi == big) {
      x = T(2) * lo;
      continue;
    }
    if (stage == 3) {
      stage = 4;
      n = 0;
    }
    x = x1 - g1 * (x1 - x0) / (g1 - g0);
    if (!(x > lo && x < hi)) x = T(0.5) * (lo + hi);
  }
}

// Returns 0 and the gauge state q, output *y_ss at the equilibrium, or < 0.
template <typename T>
__device__ __forceinline__ int equilibrium_from(const Fc3K<T>& K, const double* __restrict__ P,
                                                const CandK<double>& Cd, T q[3], T* y_ss) {
  CandK<T> C;
  C.W_o2 = static_cast<T>(Cd.W_o2);
  C.V0 = static_cast<T>(Cd.V0);
  C.y_scale = static_cast<T>(Cd.y_scale);
  const int rc = equilibrium_solve<T>(K, C, static_cast<T>(P[P_LAM_REF] * Cd.W_o2 / P[P_X_O2]), q);
  if (rc == 0) *y_ss = fc3_output<T>(C, q[0], q[2]);
  return rc;
}

// The same from the setpoint I alone.
template <typename T>
__device__ __forceinline__ int equilibrium_dev(const Fc3K<T>& K, const double* __restrict__ P,
                                               double I, T q[3], T* y_ss) {
  if (!(I > 0.0) || !(I <= DBL_MAX)) return -1;
  return equilibrium_from<T>(K, P, cand_consts(P, I), q, y_ss);
}

__device__ __forceinline__ bool pos_finite(double v) {  // off the binary64 pipe
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  return b - 1ull < 0x7fefffffffffffffull;
}

// Candidate set-up shared by the single-problem and batched searches: the
// binary32 equilibrium of setpoint v (Sec. II-A) is the reference point of
// the rollouts' deviation coordinates (0 when it cannot be found), the
// candidate's rollout constants are folded about it, and, when ss_check is
// set, the steady-state check of Eq. 3 (y_ss(v) >= thr_ss) is decided by it
// unless y_ss lands within 1e-4 of the threshold (its error is ~1e-6), in
// which case a binary64 solve decides.  Returns the check's outcome (1 when
// off).
//
// One thread's serial chain between two rollouts, so what counts is the number
// of binary64 instructions (64 cycles each) and of instruction lines fetched
// once: 29 of them (constants from EqModel, no division; conversions of the
// reference by bits) and one site of the equilibrium's right-hand side, where
// every constant was formed from the parameters with three divisions and the
// right-hand side stood six times in the code.  One candidate's kernel 8.9 -> 5.5
// us (about 2 of them the launch's).
__device__ __forceinline__ int candidate_setup(const Fc3K<double>& k64, const Fc3K<float>& k32, const EqModel& eq,
                                               const ModelC& mc, const double* __restrict__ P, double v,
                                               int ss_check, double y_min, RhsC<double>* c64, RhsC<float>* c32) {
  float q32[3] = {0.0f, 0.0f, 0.0f};
  CandK<float> C;
  C.W_o2 = static_cast<float>(__dmul_rn(eq.w1, v));
  C.V0 = static_cast<float>(fma_rn(fma_rn(eq.v2, v, eq.v1), v, eq.v0));
  C.y_scale = 0.0f;
  const bool v_ok = pos_finite(v);
  const int rc32 = v_ok ? equilibrium_solve<float>(k32, C, eq.guess * C.W_o2, q32) : -1;
  const bool found = rc32 == 0 && fabsf(q32[0]) <= FLT_MAX && fabsf(q32[1]) <= FLT_MAX && fabsf(q32[2]) <= FLT_MAX;
  double q_r[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float q = found && fabsf(q32[i]) >= FLT_MIN ? q32[i] : 0.0f;
    q_r[i] = q == 0.0f ? 0.0 : widen_bits(q);
  }
  const RhsC<double> R = fold_cand(mc, v, q_r, y_min);
  *c64 = R;
  const RhsC<float> F = round_cand(R);
  *c32 = F;
  if (!ss_check) return 1;
  const float y32 = F.y_scale * (q32[2] - q32[0]);
  if (rc32 == 0 && y32 > eq.y_pass) return 1;
  if (rc32 == 0 && y32 < eq.y_fail) return 0;
  double q[3], y_ss = 0.0;
  return v_ok && equilibrium_from<double>(k64, P, cand_consts(P, v), q, &y_ss) == 0 && y_ss >= eq.thr_ss;
}

// Start of a trajectory: the deviation z = q - q_r of the absolute state x
// (pressures measured from p_atm), formed in binary64 and rounded once, and
// the absolute speed w_r + z_w that rk4_step_fast carries next to it.
template <typename T>
__device__ __forceinline__ void start_state(const RhsC<T>& C, const double* x, double p_atm, T& z_ca,
                                            T& z_w, T& z_sm, T& w_abs) {
  z_ca = static_cast<T>((x[0] - p_atm) - static_cast<double>(C.r_ca));
  z_w = static_cast<T>(x[1] - static_cast<double>(C.r_w));
  z_sm = static_cast<T>((x[2] - p_atm) - static_cast<double>(C.r_sm));
  w_abs = C.r_w + z_w;
}

// ---------------------------------------------------------------------------
// One trajectory: x_0 = x_t, x_{j+1} = RK4(x_j, v) + d_j, slack s_j =
// h(x_j, v) - y_min at j = 0..H; a non-finite state or output counts as
// s = -inf.  Stops when s < thr (thr = -inf: never) and, checked once per
// block of PF steps, when *dead is set.  Returns min_j s_j; *steps
// receives the RK4 steps done.
//
// The disturbances of step j are loaded PF steps ahead into a small
// register ring, so the L2 latency of the three loads (larger than one RK4
// step on a two-die GB300) overlaps the arithmetic of the steps in between.
// The candidate's dead flag is read at the start of a block and used at its
// end, for the same reason.
// Depth 8 in binary32 (16,384 x 16 x 1,000 steps: 920 us, 943 at 16, which
// holds 136 registers, 1,028 at 12), 8 in binary64.
#ifndef RRG_PREFETCH
#define RRG_PREFETCH 8
#endif
#ifndef RRG_PREFETCH64
#define RRG_PREFETCH64 8
#endif
template <typename T> struct PrefetchDepth { static constexpr int value = RRG_PREFETCH; };
template <> struct PrefetchDepth<double> { static constexpr int value = RRG_PREFETCH64; };

// A finite value (the binary64 test by the exponent bits, off the slow
// binary64 pipe).
__device__ __forceinline__ bool finite_v(float x) { return fabsf(x) <= FLT_MAX; }
__device__ __forceinline__ bool finite_v(double x) { return (__double2hiint(x) & 0x7fffffff) < 0x7ff00000; }

// The slack y_j - y_min of the deviation state (y_min is folded into s_off).
template <typename T>
__device__ __forceinline__ T slack_of(const StepC<T>& C, T q_ca, T q_sm) {
  return fma_rn(C.y_scale, q_sm - q_ca, C.s_off);
}
template <typename T>
__device__ __forceinline__ T checked_slack(const StepC<T>& C, T q_ca, T w, T q_sm) {
  const T s = slack_of<T>(C, q_ca, q_sm);
  return finite_v(q_ca) && finite_v(w) && finite_v(q_sm) && finite_v(s) ? s : -inf_v<T>();
}

// The minimum of a block's slacks and whether all of them, and the state at
// its end, are finite (a block: an even number of steps; step u of it calls
// add(s, u)).  A non-finite state contaminates every component through the
// next step and NaN and inf never return to a finite value through +, -, x
// and / by a finite or NaN operand, so testing each slack and the block's last
// state finds it; the block's minimum is then -inf, as a per-step test would
// give.
//   binary32: the three-operand minimum and maximum take two steps at a time
// (one instruction a step where a minimum and a finiteness sum took two).
//   binary64: on the integer pipe (a binary64 compare costs a scheduler 64
// cycles): the minimum of the order-preserving keys, the maximum of the high
// words without their signs.
template <typename T> struct BlockMin;
template <>
struct BlockMin<float> {
  float mn, mx, prev;
  __device__ __forceinline__ BlockMin() : mn(inf_v<float>()), mx(0.0f), prev(0.0f) {}
  __device__ __forceinline__ void add(float s, int u) {
    if (u & 1) {
      asm("min.f32 %0, %1, %2, %3;" : "=f"(mn) : "f"(mn), "f"(prev), "f"(s));
      abs3(prev, s);
    } else {
      prev = s;
    }
  }
  __device__ __forceinline__ float result(float q_ca, float w, float q_sm) {
    abs3(q_ca, w);
    abs3(q_sm, q_sm);
    return mx <= FLT_MAX ? mn : -inf_v<float>();
  }
  __device__ __forceinline__ void abs3(float a, float b) {
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(mx) : "f"(mx), "f"(a), "f"(b));
  }
};
template <>
struct BlockMin<double> {
  long long mn;
  int mx;
  static __device__ __forceinline__ long long key(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffll); }
  __device__ __forceinline__ BlockMin() : mn(0x7ff0000000000000ll), mx(0) {}
  __device__ __forceinline__ void add(double s, int) {
    const long long k = key(__double_as_longlong(s));
    mn = k < mn ? k : mn;
    mx = max(mx, __double2hiint(s) & 0x7fffffff);
  }
  __device__ __forceinline__ double result(double q_ca, double w, double q_sm) {
    mx = max(max(mx, __double2hiint(q_ca) & 0x7fffffff),
             max(__double2hiint(w) & 0x7fffffff, __double2hiint(q_sm) & 0x7fffffff));
    return mx < 0x7ff00000 ? __longlong_as_double(key(mn)) : -inf_v<double>();
  }
};

// Lane outcome of run_lane.
enum LaneEnd : int { LANE_REACHED_END = 0, LANE_VIOLATED = 1, LANE_STOPPED = 2 };

// Steps j0+1..j_end of one trajectory, from the state (q_ca, w, q_sm) at
// step j0 (updated in place); with j0 = 0 the output at step 0 is checked
// first (for j0 > 0 it was checked by the run that stopped there).  smin_in
// is the min slack so far.
//
// *jlast (in/out) bounds the last step whose slack was below `band`: it is
// raised to the end of each block of steps that had one (so it may overshoot
// the step by less than PF).  The binary64 recheck of a binary32 lane needs
// only steps 0..*jlast: every later step had a binary32 slack of at least the
// band, which the band's error bound makes non-negative in binary64.
// band = -inf tracks nothing.
template <typename T, int PF = PrefetchDepth<T>::value>
__device__ __forceinline__ T run_lane(const StepU<T>& K, const PowTable* pw, const StepC<T>& C,
                                      const T* __restrict__ d, int k, int N, int H, int j0,
                                      int j_end, T& q_ca, T& w, T& q_sm, T& w_abs, T smin_in,
                                      T thr, const volatile int32_t* dead, unsigned* steps,
                                      int* end, T band, int* jlast) {
  T smin = smin_in;
  int j = j0;
  int jl = *jlast;
  int how = LANE_REACHED_END;
  bool go = j < j_end;
  if (j0 == 0) {
    const T s0 = checked_slack<T>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      go = false;
    }
  }
  if (go) {
    const size_t HN = static_cast<size_t>(H) * N;
    T r0[PF], r1[PF], r2[PF];
    const T* pf = d + static_cast<size_t>(j0) * N + k;  // next step to prefetch
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      if (j0 + u < j_end) {
        r0[u] = __ldg(pf);
        r1[u] = __ldg(pf + HN);
        r2[u] = __ldg(pf + 2 * HN);
      } else {
        r0[u] = r1[u] = r2[u] = T(0);
      }
      pf += N;
    }
    bool stop = false;
    // Whole blocks of PF steps (PF = prefetch depth) run without a per-step exit branch: the
    // running min is tested once per block.  A lane that violates inside a
    // block runs to the block's end; that only lowers its min slack, so no
    // decision changes.  The last, partial block steps one at a time.
    //
    // Finiteness is also settled once per block (BlockMin).
    while (!stop && j + PF <= j_end) {
      const int dead_now = dead != nullptr ? *dead : 0;
      BlockMin<T> bm;
#pragma unroll
      for (int u = 0; u < PF; ++u) {
        const T e0 = r0[u], e1 = r1[u], e2 = r2[u];
        if (j + PF < j_end) {
          r0[u] = __ldg(pf);
          r1[u] = __ldg(pf + HN);
          r2[u] = __ldg(pf + 2 * HN);
        }
        pf += N;
        rk4_step_fast<T>(K, pw, C, q_ca, w, q_sm, w_abs, e0, e1, e2);
        ++j;
        bm.add(slack_of<T>(C, q_ca, q_sm), u);
      }
      const T bmin = bm.result(q_ca, w, q_sm);
      smin = fmin(smin, bmin);
      if (bmin < band) jl = j;
      if (smin < thr) {
        how = LANE_VIOLATED;
        stop = true;
      } else if (dead_now != 0 && j < j_end) {
        how = LANE_STOPPED;
        stop = true;
      }
    }
    const T* dp = d + static_cast<size_t>(j) * N + k;
    while (!stop && j < j_end) {
      const T e0 = __ldg(dp), e1 = __ldg(dp + HN), e2 = __ldg(dp + 2 * HN);
      dp += N;
      rk4_step_fast<T>(K, pw, C, q_ca, w, q_sm, w_abs, e0, e1, e2);
      ++j;
      const T s = checked_slack<T>(C, q_ca, w, q_sm);
      smin = fmin(smin, s);
      if (s < band) jl = j;
      if (s < thr) {
        how = LANE_VIOLATED;
        stop = true;
      }
    }
  }
  *steps = static_cast<unsigned>(j - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// ---------------------------------------------------------------------------
// run_lane on the handles' quad layout: the disturbances of four steps come
// with one 16-byte load per component, Q quads ahead in registers.  Same
// contract, arithmetic and results as run_lane<float>; the exit and finiteness
// tests come every 4 Q steps.  A segment that starts inside a quad
// (SEG_CONTINUE after an odd probe length) steps to its end one step at a time.
// The form without shared memory: single problems stage their quads
// (run_lane_qring), whose deeper look-ahead a lone warp needs (177 against 203
// cycles a step).
// The binary32 step, packed or not (the same bits).
template <bool PACK>
__device__ __forceinline__ void lane_step(const StepU<float>& K, const StepC<float>& C, float& q_ca, float& w,
                                          float& q_sm, float& w_abs, float e0, float e1, float e2) {
  if constexpr (PACK) rk4_step_packed(K, C, q_ca, w, q_sm, w_abs, e0, e1, e2);
  else rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0, e1, e2);
}

// One step with run_lane's per-step tests; false once the lane has violated.
__device__ __forceinline__ bool lane_step_checked(const StepU<float>& K, const StepC<float>& C, float e0, float e1,
                                                  float e2, float& q_ca, float& w, float& q_sm, float& w_abs,
                                                  int& j, float& smin, float thr, float band, int& jl) {
  rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0, e1, e2);
  ++j;
  const float s = checked_slack<float>(C, q_ca, w, q_sm);
  smin = fmin(smin, s);
  if (s < band) jl = j;
  return !(s < thr);
}

template <int Q = 2>
__device__ __forceinline__ float run_lane_q(const StepU<float>& K, const StepC<float>& C,
                                            const float* __restrict__ d, int k, int N, int H, int j0, int j_end,
                                            float& q_ca, float& w, float& q_sm, float& w_abs, float smin_in,
                                            float thr, const volatile int32_t* dead, unsigned* steps, int* end,
                                            float band, int* jlast) {
  constexpr int B = 4 * Q;
  float smin = smin_in;
  int j = j0;
  int jl = *jlast;
  int how = LANE_REACHED_END;
  bool go = j < j_end;
  if (j0 == 0) {
    const float s0 = checked_slack<float>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      go = false;
    }
  }
  const size_t row = 4 * static_cast<size_t>(N), comp = quad_rows(H) * row;
  auto one = [&]() {
    const float* p = d + static_cast<size_t>(j >> 2) * row + 4 * static_cast<size_t>(k) + (j & 3);
    if (!lane_step_checked(K, C, __ldg(p), __ldg(p + comp), __ldg(p + 2 * comp), q_ca, w, q_sm, w_abs, j, smin, thr,
                           band, jl)) {
      how = LANE_VIOLATED;
      go = false;
    }
  };
  while (go && j < j_end && (j & 3) != 0) one();
  if (go && j + B <= j_end) {
    const float4* p0 = reinterpret_cast<const float4*>(d + static_cast<size_t>(j >> 2) * row) + k;
    const float4* p1 = reinterpret_cast<const float4*>(d + comp + static_cast<size_t>(j >> 2) * row) + k;
    const float4* p2 = reinterpret_cast<const float4*>(d + 2 * comp + static_cast<size_t>(j >> 2) * row) + k;
    float4 r0[Q], r1[Q], r2[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      r0[q] = __ldg(p0); r1[q] = __ldg(p1); r2[q] = __ldg(p2);
      p0 += N; p1 += N; p2 += N;
    }
    do {
      const int dead_now = dead != nullptr ? *dead : 0;
      const bool more = j + 2 * B <= j_end;  // the next block is whole too
      BlockMin<float> bm;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float4 e0 = r0[q], e1 = r1[q], e2 = r2[q];
        if (more) {
          r0[q] = __ldg(p0); r1[q] = __ldg(p1); r2[q] = __ldg(p2);
        }
        p0 += N; p1 += N; p2 += N;
        rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0.x, e1.x, e2.x);
        bm.add(slack_of<float>(C, q_ca, q_sm), 0);
        rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0.y, e1.y, e2.y);
        bm.add(slack_of<float>(C, q_ca, q_sm), 1);
        rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0.z, e1.z, e2.z);
        bm.add(slack_of<float>(C, q_ca, q_sm), 0);
        rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0.w, e1.w, e2.w);
        bm.add(slack_of<float>(C, q_ca, q_sm), 1);
      }
      j += B;
      const float bmin = bm.result(q_ca, w, q_sm);
      smin = fmin(smin, bmin);
      if (bmin < band) jl = j;
      if (smin < thr) {
        how = LANE_VIOLATED;
        go = false;
      } else if (dead_now != 0 && j < j_end) {
        how = LANE_STOPPED;
        go = false;
      }
    } while (go && j + B <= j_end);
  }
  while (go && j < j_end) one();
  *steps = static_cast<unsigned>(j - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// ---------------------------------------------------------------------------
// Two trajectories of one scenario k -- candidates A and B, the same
// disturbances -- in one thread: each quad's three loads, their addressing and
// the loop's bookkeeping serve both, and the two step chains are independent
// work for the scheduler.  Same arithmetic as run_lane_q for each trajectory:
// the decisions, and the min slack of a trajectory that does not violate,
// equal its bit for bit (a violating one may be integrated a little longer, so
// its min slack, an upper bound either way, can come out lower).
//
// From step 0 (its slack checked first: a violation there runs nothing in
// pair) over whole blocks of two quads while
// neither candidate has been stopped: a trajectory that violates keeps being
// integrated with its partner (its min slack only falls, so no decision
// changes) and, when dead_X is given, marks its candidate dead at once, so
// the stop reaches every lane together at a block end (read at the block's
// start, as in run_lane) instead of splitting the warp.  Without dead flags
// (no candidate-level exit) a lane leaves the pair when either trajectory
// has violated.  The survivor then finishes alone in run_lane_q from the
// step reached; the last, partial block too.  z_X[4] = (q_ca, w, q_sm,
// w_abs) in and out; smin, steps, end, jlast per trajectory as run_lane's.
// Returns the steps both trajectories ran together.
__device__ __forceinline__ int run_lane_pair(const StepU<float>& K, const StepC<float>& CA, const StepC<float>& CB,
                                              const float* __restrict__ d, int k, int N, int H, int j_end,
                                              float* za, float* zb, float thr, float band,
                                              volatile int32_t* deadA, volatile int32_t* deadB,
                                              float* smin, unsigned* steps, int* end, int* jlast) {
  constexpr int Q = 2, B = 4 * Q;
  smin[0] = checked_slack<float>(CA, za[0], za[1], za[2]);
  smin[1] = checked_slack<float>(CB, zb[0], zb[1], zb[2]);
  jlast[0] = smin[0] < band ? 0 : -1;
  jlast[1] = smin[1] < band ? 0 : -1;
  int how[2] = {smin[0] < thr ? LANE_VIOLATED : LANE_REACHED_END,
                smin[1] < thr ? LANE_VIOLATED : LANE_REACHED_END};
  if (how[0] == LANE_VIOLATED && deadA != nullptr) *deadA = 1;
  if (how[1] == LANE_VIOLATED && deadB != nullptr) *deadB = 1;
  const bool cand_stop = deadA != nullptr;
  int j = 0;
  bool pair = how[0] == LANE_REACHED_END && how[1] == LANE_REACHED_END;
  bool stopA = false, stopB = false;  // candidate stopped (dead flag) while not violated
  if (pair && B <= j_end) {
    const size_t row = 4 * static_cast<size_t>(N), comp = quad_rows(H) * row;
    const float4* p0 = reinterpret_cast<const float4*>(d) + k;
    const float4* p1 = reinterpret_cast<const float4*>(d + comp) + k;
    const float4* p2 = reinterpret_cast<const float4*>(d + 2 * comp) + k;
    float4 r0[Q], r1[Q], r2[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      r0[q] = __ldg(p0); r1[q] = __ldg(p1); r2[q] = __ldg(p2);
      p0 += N; p1 += N; p2 += N;
    }
    while (pair && j + B <= j_end) {
      const int dA = cand_stop ? *deadA : 0, dB = cand_stop ? *deadB : 0;
      const bool more = j + 2 * B <= j_end;
      BlockMin<float> bma, bmb;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float e0[4] = {r0[q].x, r0[q].y, r0[q].z, r0[q].w}, e1[4] = {r1[q].x, r1[q].y, r1[q].z, r1[q].w},
                    e2[4] = {r2[q].x, r2[q].y, r2[q].z, r2[q].w};
        if (more) {
          r0[q] = __ldg(p0); r1[q] = __ldg(p1); r2[q] = __ldg(p2);
        }
        p0 += N; p1 += N; p2 += N;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          rk4_step_fast<float>(K, nullptr, CA, za[0], za[1], za[2], za[3], e0[u], e1[u], e2[u]);
          rk4_step_fast<float>(K, nullptr, CB, zb[0], zb[1], zb[2], zb[3], e0[u], e1[u], e2[u]);
          bma.add(slack_of<float>(CA, za[0], za[2]), u);
          bmb.add(slack_of<float>(CB, zb[0], zb[2]), u);
        }
      }
      j += B;
      const float ba = bma.result(za[0], za[1], za[2]), bb = bmb.result(zb[0], zb[1], zb[2]);
      smin[0] = fmin(smin[0], ba);
      smin[1] = fmin(smin[1], bb);
      if (ba < band) jlast[0] = j;
      if (bb < band) jlast[1] = j;
      if (how[0] == LANE_REACHED_END && smin[0] < thr) {
        how[0] = LANE_VIOLATED;
        if (cand_stop) *deadA = 1;
      }
      if (how[1] == LANE_REACHED_END && smin[1] < thr) {
        how[1] = LANE_VIOLATED;
        if (cand_stop) *deadB = 1;
      }
      if (cand_stop) {
        // a candidate's stop comes to every lane at once: from the flag
        stopA = dA != 0 && j < j_end;
        stopB = dB != 0 && j < j_end;
        pair = !stopA && !stopB;
        if (how[0] == LANE_VIOLATED && how[1] == LANE_VIOLATED) pair = false;
      } else {
        pair = how[0] == LANE_REACHED_END && how[1] == LANE_REACHED_END;
      }
    }
  }
  unsigned extra[2] = {0u, 0u};
  // each trajectory still running finishes alone
  if (how[0] == LANE_REACHED_END && stopA) how[0] = LANE_STOPPED;
  if (how[1] == LANE_REACHED_END && stopB) how[1] = LANE_STOPPED;
  if (how[0] == LANE_REACHED_END && j < j_end) {
    int e = LANE_REACHED_END;
    smin[0] = run_lane_q(K, CA, d, k, N, H, j, j_end, za[0], za[1], za[2], za[3], smin[0], thr,
                              deadA, &extra[0], &e, band, &jlast[0]);
    how[0] = e;
  }
  if (how[1] == LANE_REACHED_END && j < j_end) {
    int e = LANE_REACHED_END;
    smin[1] = run_lane_q(K, CB, d, k, N, H, j, j_end, zb[0], zb[1], zb[2], zb[3], smin[1], thr,
                              deadB, &extra[1], &e, band, &jlast[1]);
    how[1] = e;
  }
  steps[0] = static_cast<unsigned>(j) + extra[0];
  steps[1] = static_cast<unsigned>(j) + extra[1];
  end[0] = how[0];
  end[1] = how[1];
  return j;
}

// ---------------------------------------------------------------------------
// The same trajectory loop with the disturbances staged through a ring of D
// steps in shared memory, filled by cp.async (LDGSTS) D steps ahead.  The
// exit and finiteness tests come every B steps as in run_lane (the candidate's
// dead flag is read at the start of a block and used at the end of the next
// one, since the read queues behind the ring's fills), and the block's body
// is unrolled U steps at a time.  A warp that runs one trajectory alone on
// its scheduler issues its steps in order: the register ring's 16-step
// unrolled body then costs more than the ring's extra instructions, and
// shallower register rings expose the load latency.  Measured on GB300 with
// a single warp and the scenario array in DRAM: 332 cycles per step for the
// register ring at depth 16, 262 for this ring; in the 1,024-scenario closed
// loop the average rollout launch took 70.5 us with D = 32, B = 16, U = 8
// against 78.4 us with the register ring; on another box 69.1 us with
// B = 32 against 70.2 us with B = 16 (U = 16 with B = 16: 78.3, a body too
// large for the instruction cache).  Results equal run_lane's bit for
// bit (same arithmetic in the same order); a lane may run one block longer
// after its candidate died, which changes no decision.
//
// ring: this block's ring, ring[(3 s + c) blockDim.x + threadIdx.x] holds
// component c of the step in slot s; each thread uses only its own column.
#ifndef RRG_RING_DEPTH
#define RRG_RING_DEPTH 32
#endif
#ifndef RRG_RING_UNROLL
#define RRG_RING_UNROLL 8
#endif
#ifndef RRG_RING_BLOCK
#define RRG_RING_BLOCK 32
#endif
static_assert((RRG_RING_DEPTH & (RRG_RING_DEPTH - 1)) == 0, "ring depth: a power of two");
static_assert(RRG_RING_BLOCK % RRG_RING_UNROLL == 0, "block: a multiple of the unroll");

__device__ __forceinline__ void cp_async4(float* smem_dst, const float* gmem_src) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int D = RRG_RING_DEPTH, int B = RRG_RING_BLOCK, int U = RRG_RING_UNROLL>
__device__ __forceinline__ float run_lane_ring(const StepU<float>& K, const StepC<float>& C,
                                               const float* __restrict__ d, int k, int N, int H,
                                               int j0, int j_end, float& q_ca, float& w,
                                               float& q_sm, float& w_abs, float smin_in,
                                               float thr, const volatile int32_t* dead,
                                               unsigned* steps, int* end, float band, int* jlast,
                                               float* ring) {
  float smin = smin_in;
  int j = j0;
  int jl = *jlast;
  int how = LANE_REACHED_END;
  bool go = j < j_end;
  if (j0 == 0) {
    const float s0 = checked_slack<float>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      go = false;
    }
  }
  if (go) {
    const size_t HN = static_cast<size_t>(H) * N;
    const int bd = blockDim.x;
    float* my = ring + threadIdx.x;
    const float* pf = d + static_cast<size_t>(j0) * N + k;  // next step to fetch
    // one commit group per step (empty past j_end), so that waiting until at
    // most D - 1 groups are pending means the oldest step has landed
#pragma unroll 1
    for (int u = 0; u < D; ++u) {
      if (j0 + u < j_end) {
        cp_async4(my + (3 * u) * bd, pf);
        cp_async4(my + (3 * u + 1) * bd, pf + HN);
        cp_async4(my + (3 * u + 2) * bd, pf + 2 * HN);
      }
      cp_async_commit();
      pf += N;
    }
    int slot = 0;  // slot of step j
    bool stop = false;
    // the dead flag read at the start of a block is used at the end of the
    // next one: the read queues behind the block's ring fills
    int dead_prev = 0;
    while (!stop && j + B <= j_end) {
      const int dead_now = dead != nullptr ? *dead : 0;
      BlockMin<float> bm;
#pragma unroll U
      for (int u = 0; u < B; ++u) {
        cp_async_wait<D - 1>();
        float* e = my + (3 * slot) * bd;
        const float e0 = e[0], e1 = e[bd], e2 = e[2 * bd];
        rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0, e1, e2);
        // the slot is free once its values are in registers: step j + D
        if (j + D < j_end) {
          cp_async4(e, pf);
          cp_async4(e + bd, pf + HN);
          cp_async4(e + 2 * bd, pf + 2 * HN);
        }
        cp_async_commit();
        pf += N;
        slot = (slot + 1) & (D - 1);
        ++j;
        bm.add(slack_of<float>(C, q_ca, q_sm), u);
      }
      const float bmin = bm.result(q_ca, w, q_sm);
      smin = fmin(smin, bmin);
      if (bmin < band) jl = j;
      if (smin < thr) {
        how = LANE_VIOLATED;
        stop = true;
      } else if (dead_prev != 0 && j < j_end) {
        how = LANE_STOPPED;
        stop = true;
      }
      dead_prev = dead_now;
    }
    while (!stop && j < j_end) {
      cp_async_wait<D - 1>();
      float* e = my + (3 * slot) * bd;
      const float e0 = e[0], e1 = e[bd], e2 = e[2 * bd];
      rk4_step_fast<float>(K, nullptr, C, q_ca, w, q_sm, w_abs, e0, e1, e2);
      if (j + D < j_end) {
        cp_async4(e, pf);
        cp_async4(e + bd, pf + HN);
        cp_async4(e + 2 * bd, pf + 2 * HN);
      }
      cp_async_commit();
      pf += N;
      slot = (slot + 1) & (D - 1);
      ++j;
      const float s = checked_slack<float>(C, q_ca, w, q_sm);
      smin = fmin(smin, s);
      if (s < band) jl = j;
      if (s < thr) {
        how = LANE_VIOLATED;
        stop = true;
      }
    }
    cp_async_wait<0>();  // nothing in flight into the ring when the lane ends
  }
  *steps = static_cast<unsigned>(j - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// ---------------------------------------------------------------------------
// run_lane_q with the quads staged through a ring of D in shared memory, filled
// by 16-byte asynchronous copies D quads ahead (each thread copies and reads
// its own column, so no thread waits for another).  A lone warp's step takes 177
// cycles, 211 when every value was copied by itself; launches that fill the SMs
// 117 a step and scheduler.
__device__ __forceinline__ void cp_async16(uint32_t smem_dst, const float4* gmem_src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ float4 ld_shared16(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}

constexpr int kQringDepth = 8;   // quads fetched ahead
constexpr int kQringBlock = 4;   // quads between exit tests
// Dynamic or static shared memory of a block of THREADS lanes.
constexpr size_t qring_bytes(int threads) { return static_cast<size_t>(3 * 16) * kQringDepth * threads; }

// A lane's ring: its column in the block's ring of THREADS columns, and the
// quads it still has to fetch.
template <int THREADS>
struct Qring {
  static constexpr uint32_t kComp = THREADS * 16, kSlot = 3 * kComp;
  uint32_t my, slot;   // the lane's column; byte offset of the next quad to read
  int left;            // whole quads not fetched yet
  size_t N, comp;      // in 16-byte elements
  const float4* pf;    // next quad to fetch

  // From quad j / 4 (j a multiple of 4) of scenario k, whole quads before j_end.
  __device__ __forceinline__ Qring(void* ring, const float* d, int k, int N_, int H, int j, int j_end)
      : my(static_cast<uint32_t>(__cvta_generic_to_shared(ring)) + threadIdx.x * 16), slot(0u),
        left((j_end - j) / 4), N(static_cast<size_t>(N_)), comp(quad_rows(H) * static_cast<size_t>(N_)),
        pf(reinterpret_cast<const float4*>(d) + static_cast<size_t>(j >> 2) * static_cast<size_t>(N_) + k) {
#pragma unroll 1
    for (int q = 0; q < kQringDepth; ++q) fetch(my + static_cast<uint32_t>(q) * kSlot);
  }
  // One commit group per quad (empty past the last), so that waiting until at
  // most kQringDepth - 1 groups are pending means the oldest quad has landed.
  __device__ __forceinline__ void fetch(uint32_t o) {
    if (left > 0) {
      cp_async16(o, pf);
      cp_async16(o + kComp, pf + comp);
      cp_async16(o + 2 * kComp, pf + 2 * comp);
    }
    cp_async_commit();
    pf += N;
    --left;
  }
  // The next quad's values; first(its first step's) runs between the reads and
  // the refill of their slot.
  template <typename First>
  __device__ __forceinline__ void next(float4& e0, float4& e1, float4& e2, const First& first) {
    cp_async_wait<kQringDepth - 1>();
    const uint32_t o = my + slot;
    e0 = ld_shared16(o);
    e1 = ld_shared16(o + kComp);
    e2 = ld_shared16(o + 2 * kComp);
    first(e0.x, e1.x, e2.x);
    fetch(o);  // the slot is free once its values are in registers
    slot = slot + kSlot == kQringDepth * kSlot ? 0u : slot + kSlot;
  }
  // Nothing in flight into the ring when the lane ends.
  __device__ __forceinline__ void drain() { cp_async_wait<0>(); }
};

// THREADS: threads of the block (at most); ring_mem: its qring_bytes(THREADS).
template <int THREADS, bool PACK = false>
__device__ __forceinline__ float run_lane_qring(const StepU<float>& K, const StepC<float>& C,
                                                const float* __restrict__ d, int k, int N, int H, int j0, int j_end,
                                                float& q_ca, float& w, float& q_sm, float& w_abs, float smin_in,
                                                float thr, const volatile int32_t* dead, unsigned* steps, int* end,
                                                float band, int* jlast, void* ring_mem) {
  constexpr int B = 4 * kQringBlock;
  float smin = smin_in;
  int j = j0;
  int jl = *jlast;
  int how = LANE_REACHED_END;
  bool go = j < j_end;
  if (j0 == 0) {
    const float s0 = checked_slack<float>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      go = false;
    }
  }
  const size_t row = 4 * static_cast<size_t>(N), comp = quad_rows(H) * row;
  auto one = [&]() {
    const float* p = d + static_cast<size_t>(j >> 2) * row + 4 * static_cast<size_t>(k) + (j & 3);
    if (!lane_step_checked(K, C, __ldg(p), __ldg(p + comp), __ldg(p + 2 * comp), q_ca, w, q_sm, w_abs, j, smin, thr,
                           band, jl)) {
      how = LANE_VIOLATED;
      go = false;
    }
  };
  while (go && j < j_end && (j & 3) != 0) one();
  if (go && j + B <= j_end) {
    Qring<THREADS> ring(ring_mem, d, k, N, H, j, j_end);
    int dead_prev = 0;  // read at the start of a block, used at the end of the next one
    do {
      const int dead_now = dead != nullptr ? *dead : 0;
      BlockMin<float> bm;
#pragma unroll
      for (int q = 0; q < kQringBlock; ++q) {
        float4 e0, e1, e2;
        ring.next(e0, e1, e2, [&](float f0, float f1, float f2) {
          lane_step<PACK>(K, C, q_ca, w, q_sm, w_abs, f0, f1, f2);
          bm.add(slack_of<float>(C, q_ca, q_sm), 0);
        });
        lane_step<PACK>(K, C, q_ca, w, q_sm, w_abs, e0.y, e1.y, e2.y);
        bm.add(slack_of<float>(C, q_ca, q_sm), 1);
        lane_step<PACK>(K, C, q_ca, w, q_sm, w_abs, e0.z, e1.z, e2.z);
        bm.add(slack_of<float>(C, q_ca, q_sm), 0);
        lane_step<PACK>(K, C, q_ca, w, q_sm, w_abs, e0.w, e1.w, e2.w);
        bm.add(slack_of<float>(C, q_ca, q_sm), 1);
      }
      j += B;
      const float bmin = bm.result(q_ca, w, q_sm);
      smin = fmin(smin, bmin);
      if (bmin < band) jl = j;
      if (smin < thr) {
        how = LANE_VIOLATED;
        go = false;
      } else if (dead_prev != 0 && j < j_end) {
        how = LANE_STOPPED;
        go = false;
      }
      dead_prev = dead_now;
    } while (go && j + B <= j_end);
    ring.drain();
  }
  while (go && j < j_end) one();
  *steps = static_cast<unsigned>(j - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// ---------------------------------------------------------------------------
// The trajectory loop fed by the Tensor Memory Accelerator.  Each warp owns a
// two-stage ring of T-step chunks in shared memory; a chunk is one
// cp.async.bulk.tensor copy of the box (32 scenarios from the warp's first,
// T / 4 quads of steps, 3 components) of the handle's quad layout, issued by
// lane 0 and counted on the stage's mbarrier, so four steps read their values
// with three 16-byte shared loads at fixed offsets.
// Scenarios and steps of a box beyond the array are filled with zeros by the
// copy (the ragged last warp, the last chunk).
//
// The warp walks the chunks together: the copies serve every lane, so a lane
// that has stopped keeps its place, does no arithmetic, and the chunk loop
// ends once no lane runs.  Per trajectory the arithmetic is run_lane's in the
// same order, so the min slack and the decisions equal it bit for bit; the
// exit and finiteness tests come at each whole chunk's end (the last, partial
// chunk steps one at a time with run_lane's per-step test); the candidate's
// dead flag is read at a chunk's start and used at its end, and a lane that
// violates marks `mark` at once.  on = false: the lane only keeps the warp
// company (inactive scenario, or finished in an earlier segment).
//
// Waits are bounded.  A stage whose copy has not landed after kTmaWaitLimit
// polls or kTmaWaitNs of the global timer ends the loop for the whole warp: the call counts one timeout in
// *timeouts and every lane still running reports a violation (min slack
// -inf, so no candidate is accepted on data that did not arrive).  Before
// returning, the warp waits (bounded again) for every copy it issued, so
// nothing lands in shared memory after the block has left.
//
// stages: the warp's 2 * 3 * T * 32 floats (128-byte aligned); bars: its two
// mbarriers.  Called by all 32 lanes of the warp.
#ifndef RRG_TMA_CHUNK
#define RRG_TMA_CHUNK 16
#endif
constexpr int kTmaChunk = RRG_TMA_CHUNK;
static_assert(RRG_TMA_CHUNK % 4 == 0, "whole quads of steps");
constexpr int kTmaStageFloats = 3 * kTmaChunk * 32;
constexpr int kTmaComp = kTmaChunk * 32;  // floats of a component in a stage: [quad][32 scenarios][4 steps]
constexpr unsigned kTmaStageBytes = kTmaStageFloats * 4u;
constexpr int kTmaWaitLimit = 1 << 22;          // polls
constexpr unsigned long long kTmaWaitNs = 100000000ull;  // and at most 0.1 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
// Makes the initialised barriers visible to the asynchronous proxy.
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Orders this thread's (and, after a warp barrier, the warp's) generic-proxy
// shared-memory accesses before the asynchronous proxy's next writes.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Makes a tensor map in global memory, written before the launch, visible to
// this thread's tensor copies.
__device__ __forceinline__ void fence_tensormap(const void* tmap) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Polls until the phase of the given parity has completed, at most
// kTmaWaitLimit times and kTmaWaitNs of the global timer; false if it has
// not.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (int it = 1; it < kTmaWaitLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255) == 0 && global_ns() - t0 > kTmaWaitNs) return false;
  }
  return false;
}
// Chunk copy: box (x = 4 k0, y = j / 4, z = 0) of the tensor map into `dst`,
// completion counted on `bar` (lane 0 only).  tmap == nullptr (the test
// switch RRG_INJECT_TMA_NO_COPY): nothing is issued, so the stage's wait runs
// out.
__device__ __forceinline__ void tma_chunk(const void* tmap, uint32_t dst, uint32_t bar, int k0, int j) {
  if (tmap == nullptr) return;
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kTmaStageBytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(4 * k0), "r"(j >> 2), "r"(0), "r"(bar)
      : "memory");
}

// PACK: rk4_step_packed (the same bits).  Returns *lost = true (if given) when a
// copy may still be in flight into the warp's stages although the bounded waits
// ran out: the warp must not use its stages and barriers again.
template <bool PACK>
__device__ __forceinline__ float run_lane_tma(const StepU<float>& K, const StepC<float>& C, const void* tmap,
                                              const float* __restrict__ d, int k, int N, int H,
                                              bool on, int j0, int j_end, float& q_ca, float& w,
                                              float& q_sm, float& w_abs, float smin_in, float thr,
                                              const volatile int32_t* dead, volatile int32_t* mark,
                                              unsigned* steps, int* end, float band, int* jlast,
                                              float* stages, uint64_t* bars,
                                              unsigned long long* timeouts, bool* lost = nullptr) {
  constexpr int T = kTmaChunk;
  const int lane = threadIdx.x & 31;
  float smin = smin_in;
  int j = j0;
  int jl = *jlast;
  int how = LANE_REACHED_END;
  bool run = on && j0 < j_end;
  if (on && j0 == 0) {
    const float s0 = checked_slack<float>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      run = false;
      if (mark != nullptr) *mark = 1;
    }
  }
  // a segment that starts inside a quad steps to its end one step at a time
  const int k0 = k & ~31;
  int jb = j0;  // the first chunk's step
  for (; (jb & 3) != 0 && jb < j_end; ++jb) {
    if (!run) continue;
    const float* p = d + quad_index(0, jb, k, H, N);
    const size_t comp = quad_rows(H) * 4 * static_cast<size_t>(N);
    if (!lane_step_checked(K, C, __ldg(p), __ldg(p + comp), __ldg(p + 2 * comp), q_ca, w, q_sm, w_abs, j, smin, thr,
                           band, jl)) {
      how = LANE_VIOLATED;
      run = false;
      if (mark != nullptr) *mark = 1;
    }
  }
  if (jb >= j_end) run = false;
  const int nchunks = j_end > jb ? (j_end - jb + T - 1) / T : 0;
  if (nchunks > 0 && __any_sync(0xffffffffu, run)) {
    const uint32_t st0 = smem_u32(stages), bar0 = smem_u32(bars);
    if (lane == 0) {
      mbar_init(bar0, 1u);
      mbar_init(bar0 + 8u, 1u);
      fence_mbar_init();
    }
    __syncwarp();
    if (lane == 0) {
      fence_proxy_async_smem();  // the warp may have read these stages for a tile before
      tma_chunk(tmap, st0, bar0, k0, jb);
      if (nchunks > 1) tma_chunk(tmap, st0 + kTmaStageBytes, bar0 + 8u, k0, jb + T);
    }
    int issued = nchunks > 1 ? 2 : 1;  // chunks whose copy was issued
    int waited = 0;                     // chunks whose copy has landed
    bool timed_out = false;
    for (int c = 0; c < nchunks; ++c) {
      const int sg = c & 1;
      const uint32_t bar = bar0 + 8u * static_cast<uint32_t>(sg);
      const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar, static_cast<uint32_t>((c >> 1) & 1)));
      if (!ok) {
        timed_out = true;
        break;
      }
      waited = c + 1;
      const float* e = stages + sg * kTmaStageFloats + 4 * lane;
      const int nst = j_end - (jb + c * T) < T ? j_end - (jb + c * T) : T;
      const int dead_now = (run && dead != nullptr) ? *dead : 0;
      if (run) {
        if (nst == T) {
          BlockMin<float> bm;
#pragma unroll
          for (int q = 0; q < T / 4; ++q) {
            float e0[4], e1[4], e2[4];
            const float4 f0 = *reinterpret_cast<const float4*>(e + 128 * q),
                         f1 = *reinterpret_cast<const float4*>(e + kTmaComp + 128 * q),
                         f2 = *reinterpret_cast<const float4*>(e + 2 * kTmaComp + 128 * q);
            e0[0] = f0.x; e0[1] = f0.y; e0[2] = f0.z; e0[3] = f0.w;
            e1[0] = f1.x; e1[1] = f1.y; e1[2] = f1.z; e1[3] = f1.w;
            e2[0] = f2.x; e2[1] = f2.y; e2[2] = f2.z; e2[3] = f2.w;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              lane_step<PACK>(K, C, q_ca, w, q_sm, w_abs, e0[u], e1[u], e2[u]);
              bm.add(slack_of<float>(C, q_ca, q_sm), u);
            }
          }
          j += T;
          const float bmin = bm.result(q_ca, w, q_sm);
          smin = fmin(smin, bmin);
          if (bmin < band) jl = j;
          if (smin < thr) {
            how = LANE_VIOLATED;
            run = false;
            if (mark != nullptr) *mark = 1;
          } else if (dead_now != 0 && j < j_end) {
            how = LANE_STOPPED;
            run = false;
          }
        } else {
          for (int u = 0; u < nst && run; ++u) {
            const int o = 128 * (u >> 2) + (u & 3);
            if (!lane_step_checked(K, C, e[o], e[kTmaComp + o], e[2 * kTmaComp + o], q_ca, w, q_sm, w_abs, j, smin,
                                   thr, band, jl)) {
              how = LANE_VIOLATED;
              run = false;
              if (mark != nullptr) *mark = 1;
            }
          }
        }
      }
      if (!__any_sync(0xffffffffu, run)) break;
      // every lane is done reading this stage: refill it with chunk c + 2
      __syncwarp();
      if (c + 2 < nchunks) {
        if (lane == 0) {
          fence_proxy_async_smem();
          tma_chunk(tmap, st0 + static_cast<uint32_t>(sg) * kTmaStageBytes, bar, k0, jb + (c + 2) * T);
        }
        issued = c + 3;
      }
    }
    // nothing may land after the warp leaves: wait for the copies issued and
    // not yet waited for
    bool drained = true;
    for (int c = waited; c < issued; ++c)
      drained = mbar_wait_bounded(bar0 + 8u * static_cast<uint32_t>(c & 1),
                                  static_cast<uint32_t>((c >> 1) & 1)) && drained;
    drained = __all_sync(0xffffffffu, drained);
    if (lost != nullptr) *lost = !drained;
    if (timed_out || !drained) {
      if (lane == 0) atomicAdd(timeouts, 1ull);
      if (run) {
        smin = -inf_v<float>();
        how = LANE_VIOLATED;
        run = false;
      }
    }
    __syncwarp();
    if (lane == 0 && drained) {
      mbar_inval(bar0);
      mbar_inval(bar0 + 8u);
    }
  }
  *steps = static_cast<unsigned>(j - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// ---------------------------------------------------------------------------
// Two candidates of one scenario per thread on the TMA ring: the warp's chunk
// copies, waits and shared loads serve both trajectories, whose step chains
// are independent work for the scheduler (run_lane_pair's idea on
// run_lane_tma's ring).  Per trajectory the arithmetic, the chunk-end tests
// and the dead-flag handling are run_lane_tma's, so the decisions and the min
// slack of a trajectory that does not violate equal it bit for bit.  A chunk
// in which both trajectories of a lane run takes one body for both; one that
// has stopped leaves the other to a single-trajectory body.
struct TmaTraj {
  float q_ca, w, q_sm, w_abs;  // deviation state and absolute speed
  float smin;
  int jl, how, j;
  bool run;
};

__device__ __forceinline__ void tma_traj_start(TmaTraj& t, const StepC<float>& C, bool on, int j0, int j_end,
                                               float thr, float band, volatile int32_t* mark) {
  t.j = j0;
  t.how = LANE_REACHED_END;
  t.run = on && j0 < j_end;
  if (on && j0 == 0) {
    const float s0 = checked_slack<float>(C, t.q_ca, t.w, t.q_sm);
    t.smin = fmin(t.smin, s0);
    if (s0 < band) t.jl = 0;
    if (s0 < thr) {
      t.how = LANE_VIOLATED;
      t.run = false;
      if (mark != nullptr) *mark = 1;
    }
  }
}

// The tests at the end of a whole chunk of T steps (run_lane_tma's).
__device__ __forceinline__ void tma_traj_chunk_end(TmaTraj& t, BlockMin<float>& bm, int T, int j_end, float thr,
                                                   float band, int dead_now, volatile int32_t* mark) {
  t.j += T;
  const float bmin = bm.result(t.q_ca, t.w, t.q_sm);
  t.smin = fmin(t.smin, bmin);
  if (bmin < band) t.jl = t.j;
  if (t.smin < thr) {
    t.how = LANE_VIOLATED;
    t.run = false;
    if (mark != nullptr) *mark = 1;
  } else if (dead_now != 0 && t.j < j_end) {
    t.how = LANE_STOPPED;
    t.run = false;
  }
}

// A whole chunk for one trajectory (e: the lane's column of the stage).
template <int T>
__device__ __forceinline__ void tma_traj_chunk(TmaTraj& t, const StepU<float>& K, const StepC<float>& C,
                                               const float* e, BlockMin<float>& bm) {
#pragma unroll 8
  for (int u = 0; u < T; ++u) {
    const int o = 128 * (u >> 2) + (u & 3);
    rk4_step_fast<float>(K, nullptr, C, t.q_ca, t.w, t.q_sm, t.w_abs, e[o], e[kTmaComp + o], e[2 * kTmaComp + o]);
    bm.add(slack_of<float>(C, t.q_ca, t.q_sm), u);
  }
}

// A whole chunk for both trajectories, one load of each value for the two.
template <int T>
__device__ __forceinline__ void tma_pair_chunk(TmaTraj& a, TmaTraj& b, const StepU<float>& K,
                                               const StepC<float>& CA, const StepC<float>& CB,
                                               const float* e, BlockMin<float>& bma,
                                               BlockMin<float>& bmb) {
#pragma unroll 8
  for (int u = 0; u < T; ++u) {
    const int o = 128 * (u >> 2) + (u & 3);
    const float e0 = e[o], e1 = e[kTmaComp + o], e2 = e[2 * kTmaComp + o];
    rk4_step_fast<float>(K, nullptr, CA, a.q_ca, a.w, a.q_sm, a.w_abs, e0, e1, e2);
    rk4_step_fast<float>(K, nullptr, CB, b.q_ca, b.w, b.q_sm, b.w_abs, e0, e1, e2);
    bma.add(slack_of<float>(CA, a.q_ca, a.q_sm), u);
    bmb.add(slack_of<float>(CB, b.q_ca, b.q_sm), u);
  }
}

// The last, partial chunk: step by step with the per-step test (run_lane's).
__device__ __forceinline__ void tma_traj_tail(TmaTraj& t, const StepU<float>& K, const StepC<float>& C,
                                              const float* e, int nst, float thr, float band,
                                              volatile int32_t* mark) {
  for (int u = 0; u < nst && t.run; ++u) {
    const int o = 128 * (u >> 2) + (u & 3);
    if (!lane_step_checked(K, C, e[o], e[kTmaComp + o], e[2 * kTmaComp + o], t.q_ca, t.w, t.q_sm, t.w_abs, t.j,
                           t.smin, thr, band, t.jl)) {
      t.how = LANE_VIOLATED;
      t.run = false;
      if (mark != nullptr) *mark = 1;
    }
  }
}

// The chunk loop of run_lane_tma for two trajectories per lane (a: candidate
// A, b: candidate B; state, smin and jl in, everything out; steps = j - j0).
// dead_X / mark_X: the candidates' flags (nullptr without a candidate-level
// exit).  *paired: steps this lane ran for both trajectories at once.  Called
// by all 32 lanes of the warp.
__device__ __forceinline__ void run_lane_tma_pair(const StepU<float>& K, const StepC<float>& CA,
                                                  const StepC<float>& CB, const void* tmap, int k0, bool onA,
                                                  bool onB, int j0, int j_end, TmaTraj& a, TmaTraj& b,
                                                  float thr, float band, const volatile int32_t* deadA,
                                                  const volatile int32_t* deadB, volatile int32_t* markA,
                                                  volatile int32_t* markB, float* stages, uint64_t* bars,
                                                  unsigned long long* timeouts, unsigned* paired) {
  constexpr int T = kTmaChunk;
  const int lane = threadIdx.x & 31;
  tma_traj_start(a, CA, onA, j0, j_end, thr, band, markA);
  tma_traj_start(b, CB, onB, j0, j_end, thr, band, markB);
  *paired = 0u;
  const int nchunks = j_end > j0 ? (j_end - j0 + T - 1) / T : 0;
  if (nchunks > 0 && __any_sync(0xffffffffu, a.run || b.run)) {
    const uint32_t st0 = smem_u32(stages), bar0 = smem_u32(bars);
    if (lane == 0) {
      mbar_init(bar0, 1u);
      mbar_init(bar0 + 8u, 1u);
      fence_mbar_init();
    }
    __syncwarp();
    if (lane == 0) {
      tma_chunk(tmap, st0, bar0, k0, j0);
      if (nchunks > 1) tma_chunk(tmap, st0 + kTmaStageBytes, bar0 + 8u, k0, j0 + T);
    }
    int issued = nchunks > 1 ? 2 : 1;
    int waited = 0;
    bool timed_out = false;
    for (int c = 0; c < nchunks; ++c) {
      const int sg = c & 1;
      const uint32_t bar = bar0 + 8u * static_cast<uint32_t>(sg);
      const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar, static_cast<uint32_t>((c >> 1) & 1)));
      if (!ok) {
        timed_out = true;
        break;
      }
      waited = c + 1;
      const float* e = stages + sg * kTmaStageFloats + 4 * lane;
      const int nst = j_end - (j0 + c * T) < T ? j_end - (j0 + c * T) : T;
      const int da = (a.run && deadA != nullptr) ? *deadA : 0;
      const int db = (b.run && deadB != nullptr) ? *deadB : 0;
      if (nst == T) {
        BlockMin<float> bma, bmb;
        if (a.run && b.run) {
          tma_pair_chunk<T>(a, b, K, CA, CB, e, bma, bmb);
          *paired += 2u * T;
          tma_traj_chunk_end(a, bma, T, j_end, thr, band, da, markA);
          tma_traj_chunk_end(b, bmb, T, j_end, thr, band, db, markB);
        } else if (a.run) {
          tma_traj_chunk<T>(a, K, CA, e, bma);
          tma_traj_chunk_end(a, bma, T, j_end, thr, band, da, markA);
        } else if (b.run) {
          tma_traj_chunk<T>(b, K, CB, e, bmb);
          tma_traj_chunk_end(b, bmb, T, j_end, thr, band, db, markB);
        }
      } else {
        tma_traj_tail(a, K, CA, e, nst, thr, band, markA);
        tma_traj_tail(b, K, CB, e, nst, thr, band, markB);
      }
      if (!__any_sync(0xffffffffu, a.run || b.run)) break;
      // every lane is done reading this stage: refill it with chunk c + 2
      __syncwarp();
      if (c + 2 < nchunks) {
        if (lane == 0) {
          fence_proxy_async_smem();
          tma_chunk(tmap, st0 + static_cast<uint32_t>(sg) * kTmaStageBytes, bar, k0, j0 + (c + 2) * T);
        }
        issued = c + 3;
      }
    }
    bool drained = true;
    for (int c = waited; c < issued; ++c)
      drained = mbar_wait_bounded(bar0 + 8u * static_cast<uint32_t>(c & 1),
                                  static_cast<uint32_t>((c >> 1) & 1)) && drained;
    drained = __all_sync(0xffffffffu, drained);
    if (timed_out || !drained) {
      if (lane == 0) atomicAdd(timeouts, 1ull);
      if (a.run) {
        a.smin = -inf_v<float>();
        a.how = LANE_VIOLATED;
        a.run = false;
      }
      if (b.run) {
        b.smin = -inf_v<float>();
        b.how = LANE_VIOLATED;
        b.run = false;
      }
    }
    __syncwarp();
    if (lane == 0 && drained) {
      mbar_inval(bar0);
      mbar_inval(bar0 + 8u);
    }
  }
}

// Disturbance component of Philox word w with half-range a: the binary32
// copy (top 24 bits, a 2^-23 folded in) or the binary64 value, exactly as the
// sampler stores them.
template <typename T> __device__ __forceinline__ T draw(uint64_t w, double a);
template <> __device__ __forceinline__ float draw<float>(uint64_t w, double a) {
  return uniform_sym32(w, static_cast<float>(a * 0x1.0p-23));
}
template <> __device__ __forceinline__ double draw<double>(uint64_t w, double a) {
  return uniform_sym(w, a);
}

// The binary32 copy of scenario k's quads q0 .. q1 - 1 (of a block's threads:
// the same quads).  Steps past the horizon in its last quad are drawn too; no
// trajectory reads them.
__device__ __forceinline__ void sample_quads(float* __restrict__ d, int N, int H, int k, int q0, int q1,
                                             uint64_t kbase, uint64_t upd, uint64_t seed, float s0, float s1,
                                             float s2) {
  const PhiloxCols<1> P(kbase + static_cast<uint64_t>(k), 0, upd, seed);
  const size_t rows = quad_rows(H);
  for (int q = q0; q < q1; ++q) {
    float a[4], b[4], c[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      P.step(4 * q + u, [&](int, uint64_t w0, uint64_t w1, uint64_t w2) {
        a[u] = uniform_sym32(w0, s0);
        b[u] = uniform_sym32(w1, s1);
        c[u] = uniform_sym32(w2, s2);
      });
    if (k < N) {
      float4* o = reinterpret_cast<float4*>(d) + static_cast<size_t>(q) * N + k;
      o[0] = make_float4(a[0], a[1], a[2], a[3]);
      o[rows * N] = make_float4(b[0], b[1], b[2], b[3]);
      o[2 * rows * N] = make_float4(c[0], c[1], c[2], c[3]);
    }
  }
}

// run_lane with the disturbances drawn from their Philox counters (j, k,
// update, 0) inside the loop instead of read from the stored array: the
// same values, so the same trajectory and decisions.  Same contract as
// run_lane.
template <typename T, int PF = PrefetchDepth<T>::value>
__device__ __forceinline__ T run_lane_gen(const StepU<T>& K, const PowTable* pw, const StepC<T>& C,
                                          const ScenSrc& src,
                                          int k, int j0, int j_end, T& q_ca, T& w, T& q_sm,
                                          T& w_abs, T smin_in, T thr,
                                          const volatile int32_t* dead, unsigned* steps, int* end,
                                          T band, int* jlast) {
  T smin = smin_in;
  int j = j0;
  int jl = *jlast;
  int how = LANE_REACHED_END;
  bool go = j < j_end;
  if (j0 == 0) {
    const T s0 = checked_slack<T>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      go = false;
    }
  }
  bool stop = !go;
  while (!stop && j + PF <= j_end) {
    const int dead_now = dead != nullptr ? *dead : 0;
    BlockMin<T> bm;
#pragma unroll 4
    for (int u = 0; u < PF; ++u) {
      const U64x4 r = philox4x64_10(static_cast<uint64_t>(j), src.base + static_cast<uint64_t>(k), src.update,
                                    0ull, src.seed, 0ull);
      rk4_step_fast<T>(K, pw, C, q_ca, w, q_sm, w_abs, draw<T>(r.w[0], src.amp[0]),
                       draw<T>(r.w[1], src.amp[1]), draw<T>(r.w[2], src.amp[2]));
      ++j;
      bm.add(slack_of<T>(C, q_ca, q_sm), u);
    }
    const T bmin = bm.result(q_ca, w, q_sm);
    smin = fmin(smin, bmin);
    if (bmin < band) jl = j;
    if (smin < thr) {
      how = LANE_VIOLATED;
      stop = true;
    } else if (dead_now != 0 && j < j_end) {
      how = LANE_STOPPED;
      stop = true;
    }
  }
  while (!stop && j < j_end) {
    const U64x4 r = philox4x64_10(static_cast<uint64_t>(j), src.base + static_cast<uint64_t>(k), src.update, 0ull,
                                  src.seed, 0ull);
    rk4_step_fast<T>(K, pw, C, q_ca, w, q_sm, w_abs, draw<T>(r.w[0], src.amp[0]),
                     draw<T>(r.w[1], src.amp[1]), draw<T>(r.w[2], src.amp[2]));
    ++j;
    const T s = checked_slack<T>(C, q_ca, w, q_sm);
    smin = fmin(smin, s);
    if (s < band) jl = j;
    if (s < thr) {
      how = LANE_VIOLATED;
      stop = true;
    }
  }
  *steps = static_cast<unsigned>(j - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// Binary32 lanes whose disturbances are drawn, not stored.  A draw costs three
// times a step's instructions (15 64-bit products), and every candidate of a
// scenario takes the same one: ROWS warps of a block run different candidates
// of the same 32 scenarios and share it.  A chunk is 4 ROWS steps in one of two
// shared buffers; a quad of the next chunk is drawn by each of the ROWS warps
// themselves, or (SPLIT) by each of ROWS further warps, which fills the gaps of
// a step's dependent chain while there are few warps on an SM.  One barrier a
// chunk.  Measured on GB300, 1,000 steps of 1,000 scenarios and 1 / 16 / 64
// candidates, every lane drawing for itself: 319 / 322 / 921 us; here 119 /
// 122 / 313 us.
// Same contract, values and decisions as run_lane_gen; exits are taken at the
// end of each 16 steps, and a lane that violates marks `dead` at once.  Called
// by every thread of the block; on = false: the lane only draws.
template <int ROWS, bool SPLIT>
struct GenShape {
  static constexpr int kRows = ROWS, kThreads = 32 * ROWS * (SPLIT ? 2 : 1);
  static constexpr int kSteps = 4 * ROWS, kComp = 32 * kSteps;  // steps of a chunk, floats of a component
};
template <int ROWS, bool SPLIT, bool PACK>
__device__ __forceinline__ float run_lane_gen_shared(const StepU<float>& K, const StepC<float>& C, const ScenSrc& src,
                                                     int k, bool on, int j0, int j_end, float& q_ca, float& w,
                                                     float& q_sm, float& w_abs, float smin_in, float thr,
                                                     volatile int32_t* dead, unsigned* steps, int* end, float band,
                                                     int* jlast, float* buf) {
  constexpr int kSteps = GenShape<ROWS, SPLIT>::kSteps, kComp = GenShape<ROWS, SPLIT>::kComp;
  const int lane = threadIdx.x & 31, quad = static_cast<int>(threadIdx.x >> 5) - (SPLIT ? ROWS : 0);
  float smin = smin_in;
  int j = j0, jl = *jlast, how = LANE_REACHED_END;
  bool run = on && j0 < j_end;
  if (on && j0 == 0) {
    const float s0 = checked_slack<float>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      run = false;
      if (dead != nullptr) *dead = 1;
    }
  }
  const PhiloxCols<1> P(src.base + static_cast<uint64_t>(k), 0, src.update, src.seed);
  const float a0 = static_cast<float>(src.amp[0] * 0x1.0p-23), a1 = static_cast<float>(src.amp[1] * 0x1.0p-23),
              a2 = static_cast<float>(src.amp[2] * 0x1.0p-23);
  auto fill = [&](int jc, float* b) {  // this warp's quad of the chunk that starts at jc
    const int jq = jc + 4 * quad;
    if (quad < 0 || jq >= j_end) return;
    float e0[4], e1[4], e2[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      P.step(jq + u, [&](int, uint64_t w0, uint64_t w1, uint64_t w2) {
        e0[u] = uniform_sym32(w0, a0);
        e1[u] = uniform_sym32(w1, a1);
        e2[u] = uniform_sym32(w2, a2);
      });
    float4* o = reinterpret_cast<float4*>(b + 128 * quad + 4 * lane);
    o[0] = make_float4(e0[0], e0[1], e0[2], e0[3]);
    o[kComp / 4] = make_float4(e1[0], e1[1], e1[2], e1[3]);
    o[kComp / 2] = make_float4(e2[0], e2[1], e2[2], e2[3]);
  };
  if (__syncthreads_or(run)) {
    fill(j0, buf);
    __syncthreads();
    for (int jc = j0, sg = 0; jc < j_end; jc += kSteps, sg ^= 1) {
      if (jc + kSteps < j_end) fill(jc + kSteps, buf + (sg ^ 1) * 3 * kComp);
#pragma unroll 1
      for (int h = 0; h < kSteps / 16; ++h) {
        const float* e = buf + sg * 3 * kComp + h * 512 + 4 * lane;
        const int left = j_end - (jc + 16 * h);
        const int dead_now = (run && dead != nullptr) ? *dead : 0;
        if (run && left >= 16) {
          BlockMin<float> bm;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float e0[4], e1[4], e2[4];
            const float4 f0 = *reinterpret_cast<const float4*>(e + 128 * q),
                         f1 = *reinterpret_cast<const float4*>(e + kComp + 128 * q),
                         f2 = *reinterpret_cast<const float4*>(e + 2 * kComp + 128 * q);
            e0[0] = f0.x; e0[1] = f0.y; e0[2] = f0.z; e0[3] = f0.w;
            e1[0] = f1.x; e1[1] = f1.y; e1[2] = f1.z; e1[3] = f1.w;
            e2[0] = f2.x; e2[1] = f2.y; e2[2] = f2.z; e2[3] = f2.w;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              lane_step<PACK>(K, C, q_ca, w, q_sm, w_abs, e0[u], e1[u], e2[u]);
              bm.add(slack_of<float>(C, q_ca, q_sm), u);
            }
          }
          j += 16;
          const float bmin = bm.result(q_ca, w, q_sm);
          smin = fmin(smin, bmin);
          if (bmin < band) jl = j;
          if (smin < thr) {
            how = LANE_VIOLATED;
            run = false;
            if (dead != nullptr) *dead = 1;
          } else if (dead_now != 0 && j < j_end) {
            how = LANE_STOPPED;
            run = false;
          }
        } else if (run) {
          for (int u = 0; u < left && run; ++u) {
            const int o = 128 * (u >> 2) + (u & 3);
            if (!lane_step_checked(K, C, e[o], e[kComp + o], e[2 * kComp + o], q_ca, w, q_sm, w_abs, j, smin,
                                   thr, band, jl)) {
              how = LANE_VIOLATED;
              run = false;
              if (dead != nullptr) *dead = 1;
            }
          }
        }
      }
      if (!__syncthreads_or(run)) break;
    }
  }
  *steps = static_cast<unsigned>(j - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// Scenario k's model under parametric uncertainty: the parameters theta_p
// m_p^k folded like the nominal ones (the step of size dt included).
__device__ __forceinline__ void scenario_fold(const double* __restrict__ P, const double* __restrict__ m_k,
                                              double dt, const PowTable* pws, StepModel<double>* out) {
  double Pk[RRG_NPARAM];
#pragma unroll
  for (int p = 0; p < RRG_NPARAM; ++p) Pk[p] = __dmul_rn(P[p], m_k[p]);
  Fc3K<double> k64;
  Fc3K<float> k32;
  fold_constants(Pk, &k64, &k32);
  // the table only if the scenario's exponent is the table's
  k64.pws = (pws != nullptr && pws->e == k64.e) ? pws : nullptr;
  fold_model(k64, Pk, dt, out);
}

// The model a lane integrates: the launch's own, or scenario k's under
// parametric uncertainty (PU), with the candidate constants at setpoint v
// about the reference point of the nominal ones that R comes in with
// (replaced on return).  Returns the origin of the lane's gauge coordinates.
//   binary32: scenario k's model is read from the arrays that
// scenario_fold_kernel wrote with the draw; only the candidate constants are
// formed here (about 20 binary64 instructions; folding the model in every lane
// took about 600, 1.6 ms of the 65,536-scenario sweep).
//   binary64 (recheck, binary64 handles): the lane folds it.
template <typename T>
struct LaneModel {
  StepU<T> U;
  StepC<T> C;
  const PowTable* pw;
};
__device__ __forceinline__ double lane_model_pu(const Launch& L, const ScenFold& sf, const double*, int k,
                                                double v, RhsC<float>& R, LaneModel<float>& M) {
  const size_t N = static_cast<size_t>(L.N);
  ModelC mc;
  double* d = &mc.l_ca;
#pragma unroll
  for (int j = 0; j < kFoldDoubles; ++j) d[j] = __ldg(sf.d + j * N + k);
  StepPhi<float> F;
  float* u = &M.U.ip;
  constexpr int nu = sizeof(StepU<float>) / sizeof(float);
#pragma unroll
  for (int j = 0; j < nu; ++j) u[j] = __ldg(sf.f + j * N + k);
  float* p = &F.h;
#pragma unroll
  for (int j = 0; j < kFoldFloats - nu; ++j) p[j] = __ldg(sf.f + (nu + j) * N + k);
  // products of the step size alone: the launch's, constant-bank operands
  // instead of registers (16,384 x 16 x 1,000 steps: 851 -> 823 us)
  M.U.w2n1 = L.m32.U.w2n1;
  M.U.w3n2 = L.m32.U.w3n2;
  M.U.w4n3 = L.m32.U.w4n3;
  M.U.fwn4 = L.m32.U.fwn4;
  const double q_r[3] = {static_cast<double>(R.r_ca), static_cast<double>(R.r_w), static_cast<double>(R.r_sm)};
  R = round_cand(fold_cand(mc, v, q_r, L.y_min));
  M.C = step_consts<float>(M.U, F, R);
  M.pw = nullptr;
  return mc.p_atm;
}
__device__ __forceinline__ double lane_model_pu(const Launch& L, const ScenFold&, const double* pm, int k,
                                                double v, RhsC<double>& R, LaneModel<double>& M) {
  StepModel<double> sm;
  scenario_fold(L.params, pm + static_cast<size_t>(k) * RRG_NPARAM, L.dt, L.m64.pw, &sm);
  const double q_r[3] = {R.r_ca, R.r_w, R.r_sm};
  R = fold_cand(sm.c, v, q_r, L.y_min);
  M.U = sm.U;
  M.C = step_consts<double>(sm.U, sm.F, R);
  M.pw = sm.pw;
  return sm.c.p_atm;
}
template <typename T> __device__ __forceinline__ const StepModel<T>& launch_model(const Launch& L);
template <> __device__ __forceinline__ const StepModel<float>& launch_model<float>(const Launch& L) { return L.m32; }
template <> __device__ __forceinline__ const StepModel<double>& launch_model<double>(const Launch& L) { return L.m64; }
// pair: the scenario pair the lane reads (0 or 1); pm: its multipliers.
template <typename T, bool PU>
__device__ __forceinline__ double lane_model(const Launch& L, int pair, int k, double v, RhsC<T>& R,
                                             LaneModel<T>& M) {
  if constexpr (PU) {
    return lane_model_pu(L, pair ? L.foldb : L.fold, pair ? L.pmulb : L.pmul, k, v, R, M);
  } else {
    const StepModel<T>& m = launch_model<T>(L);
    M.U = m.U;
    M.C = step_consts<T>(m.U, m.F, R);
    M.pw = m.pw;
    return m.c.p_atm;
  }
}

// ---------------------------------------------------------------------------
// Four lanes per binary64 trajectory.  A binary64 instruction holds a warp
// scheduler for 64 cycles however many lanes it serves, so while there are
// fewer warps than schedulers a trajectory's time is its instruction count.
// The lanes 4 g .. 4 g + 3 of a warp share trajectory g: one instruction forms
// one multiply-add of up to four rows of rk4_step_fast's combinations (R0: x
// and w of stage 2, x of stage 1; R1: x and w of stage 3, the cathode
// pressure; R2: x and w of stage 4, the manifold pressure, the speed), and in
// a torque lane 0 evaluates the power, lane 1 the reciprocal and lane 2 the
// factor it multiplies side by side: 42 instead of 110 binary64 instructions a
// step.  Every row's operations and their order are rk4_step_fast's (a row
// without a term adds a product with 0), so the trajectory equals the one-lane
// form's.  The rest of a step is selects and shuffles of operands (446
// instructions in all); a branch around the power's cell or the reciprocal
// cost more than all lanes doing both.  Measured on GB300, a step of a lone
// warp: 7,000 cycles one lane per trajectory, 3,850 here (42 x 64 held by the
// pipe, the rest shuffle and select latency); 257 x 8 trajectories of 500
// steps 1.90 -> 1.05 ms a call.
struct Coop64 {
  int role, lane0;  // lane in its group, the group's first lane
  int src1, src2, srcp;  // lane each operand comes from: its own or another's of the group
  uint32_t neg1, neg2;   // sign flips of lane 1's and lane 2's products
  bool live = true;      // false: the group's values are not read (no power off the table for them)
  double r_w, e, A, B, cv;           // r_w: lane 2's, 0 elsewhere
  double k0[3], k1[3], k2[3];        // rows of (a, s, w)
  double c0, c1, c2;                 // their constants
  double n10, n11, n12, n21, n22, n32, n42;
  double y_scale, s_off;
  const PowCell* cells;
  bool table;

  // cells: a table; pw: the trajectory's (nullptr: its exponent has none).
  __device__ __forceinline__ Coop64(const StepU<double>& U, const PowTable* pw, const PowTable* any,
                                    const StepC<double>& C)
      : role(static_cast<int>(threadIdx.x & 3)), lane0(static_cast<int>(threadIdx.x & 28)), e(U.e), A(U.A),
        B(U.B), y_scale(C.y_scale), s_off(C.s_off), cells(any->cell), table(pw != nullptr) {
    auto pick = [&](double v0, double v1, double v2, double v3) {
      return role == 0 ? v0 : role == 1 ? v1 : role == 2 ? v2 : v3;
    };
    src1 = role == 1 ? lane0 + 1 : lane0;
    src2 = role == 2 ? lane0 + 1 : lane0 + role;
    srcp = role == 2 ? lane0 + 3 : lane0 + role;
    neg1 = role == 1 ? 0x80000000u : 0u;
    neg2 = role == 2 ? 0x80000000u : 0u;
    r_w = pick(0.0, 0.0, C.r_w, 0.0);
    cv = pick(-1.0, 1.0, -U.B, 0.0);
    k0[0] = pick(U.x2a, 0.0, 0.0, 0.0);
    k0[1] = pick(U.x2s, U.w2s, U.ip, 0.0);
    k0[2] = pick(U.x2w, U.w2w, 0.0, 0.0);
    c0 = pick(C.x2, C.w2, C.x1, 0.0);
    k1[0] = pick(U.x3a, U.w3a, U.faa, 0.0);
    k1[1] = pick(U.x3s, U.w3s, U.fas, 0.0);
    k1[2] = pick(U.x3w, U.w3w, U.faw, 0.0);
    c1 = pick(C.x3, C.w3, C.fa, 0.0);
    k2[0] = pick(U.x4a, U.w4a, U.fsa, U.fwa);
    k2[1] = pick(U.x4s, U.w4s, U.fss, U.fws);
    k2[2] = pick(U.x4w, U.w4w, U.fsw, U.fww);
    c2 = pick(C.x4, C.w4, C.fs, C.fw);
    n10 = pick(0.0, U.w2n1, 0.0, 0.0);
    n11 = pick(U.x3n1, U.w3n1, U.fan1, 0.0);
    n12 = pick(U.x4n1, U.w4n1, U.fsn1, U.fwn1);
    n21 = pick(0.0, U.w3n2, U.fan2, 0.0);
    n22 = pick(U.x4n2, U.w4n2, U.fsn2, U.fwn2);
    n32 = pick(0.0, U.w4n3, U.fsn3, U.fwn3);
    n42 = U.fwn4;
  }
  __device__ __forceinline__ static double get(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
  __device__ __forceinline__ static double flip(double v, uint32_t sign) {
    return __hiloint2double(__double2hiint(v) ^ static_cast<int>(sign), __double2loint(v));
  }
  // N(x, w) in every lane; X: w in lane 1, x in the others.
  __device__ __forceinline__ double torque4(double X) const {
    const int hi = __double2hiint(X);
    const bool in = table && (hi >> 20) == 0x3ff;
    // pow_m1_table's cell (some cell when x is off the table)
    const PowCell* __restrict__ c = cells + ((hi >> 11) & (kPowCells - 1));
    const double2 ia = __ldg(reinterpret_cast<const double2*>(c));
    const double2 a12 = __ldg(reinterpret_cast<const double2*>(c) + 1);
    const float4 f = __ldg(reinterpret_cast<const float4*>(c) + 2);
    double r0;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(X));
    const uint32_t b = (static_cast<uint32_t>(hi) & 0xfffffu) << 3 |
                       static_cast<uint32_t>(__double2loint(X)) >> 29;
    const float tf = fma_rn(__uint_as_float(0x3f800000u | b), f.w, -1.0f);
    const double p3 = widen_bits(fma_rn(fma_rn(f.z, tf, f.y), tf, f.x));
    const bool l1 = role == 1, l2 = role == 2;
    const double v1 = fma_rn(flip(X, neg1), l1 ? r0 : l2 ? B : ia.x, cv);
    const double v2 = fma_rn(v1, l1 ? r0 : p3, l1 ? r0 : a12.y);
    const double v3 = fma_rn(v1, v2, l1 ? r0 : a12.x);
    double v4 = fma_rn(flip(v1, neg2), get(v3, src2), l2 ? A : ia.y);
    if (__any_sync(0xffffffffu, !in && live && role == 0)) {
      if (!in && role == 0) v4 = pow(X, e) - 1.0;
      __syncwarp();
    }
    return get(v4, lane0) * get(v4, lane0 + 2);
  }
  // One step; every lane of the group holds the state.  e1, e2: lane 2's are
  // the cathode and manifold pressure's disturbance, lane 3's e2 the speed's,
  // the others 0.
  __device__ __forceinline__ void step(double& a, double& w, double& s, double& w_abs, double e1, double e2) const {
    double R0 = fma_rn(k0[2], w, fma_rn(k0[1], s, fma_rn(k0[0], a, c0)));  // lane 2: x of stage 1
    const double x = get(R0, lane0 + 2);
    const double n1 = torque4(role == 1 ? w_abs : x);
    double R1 = fma_rn(k1[2], w, fma_rn(k1[1], s, fma_rn(k1[0], a, e1 + c1)));
    double R2 = fma_rn(k2[2], w, fma_rn(k2[1], s, fma_rn(k2[0], a, e2 + c2)));
    R0 = fma_rn(n10, n1, R0);
    const double n2 = torque4(get(R0, src1));
    R1 = fma_rn(n11, n1, R1);
    R2 = fma_rn(n12, n1, R2);
    R1 = fma_rn(n21, n2, R1);
    const double n3 = torque4(get(R1, src1));
    R2 = fma_rn(n22, n2, R2);
    R2 = fma_rn(n32, n3, R2);
    const double n4 = torque4(get(R2, src1));
    const double V = fma_rn(n42, n4, get(R2, srcp) + r_w);
    a = get(R1, lane0 + 2);
    s = get(R2, lane0 + 2);
    w = get(V, lane0 + 3);
    w_abs = get(V, lane0 + 2);
  }
  __device__ __forceinline__ double slack(double a, double s) const { return fma_rn(y_scale, s - a, s_off); }
};

// run_lane<double> for a group of four lanes (called by every lane of the warp;
// on = false: the group only keeps the warp company).  The warp steps together
// while any of its groups runs; one that has stopped keeps stepping without
// recording.  Same contract and results as run_lane, in blocks of four steps.
__device__ __forceinline__ double run_lane_coop64(const StepU<double>& U, const PowTable* pw, const PowTable* any,
                                                  const StepC<double>& C,
                                                  const double* __restrict__ d, int k, bool on, int N, int H,
                                                  int j0, int j_end, double& q_ca, double& w, double& q_sm,
                                                  double& w_abs, double smin_in, double thr,
                                                  volatile int32_t* dead, unsigned* steps, int* end,
                                                  double band, int* jlast) {
  constexpr int B = 4;
  Coop64 G(U, pw, any, C);
  double smin = smin_in;
  int j = j0, j_stop = j0, jl = *jlast, how = LANE_REACHED_END;
  bool run = on && j0 < j_end;
  if (on && j0 == 0) {
    const double s0 = checked_slack<double>(C, q_ca, w, q_sm);
    smin = fmin(smin, s0);
    if (s0 < band) jl = 0;
    if (s0 < thr) {
      how = LANE_VIOLATED;
      run = false;
    }
  }
  const size_t HN = static_cast<size_t>(H) * N;
  const bool ld1 = on && G.role == 2, ld2 = on && G.role >= 2;
  const double* p1 = d + static_cast<size_t>(j0) * N + k;
  const double* p2 = p1 + (G.role == 2 ? 2 * HN : HN);
  double a = q_ca, v = w, s = q_sm, va = w_abs;
  double e1 = ld1 && j0 < j_end ? __ldg(p1) : 0.0, e2 = ld2 && j0 < j_end ? __ldg(p2) : 0.0;
  auto one = [&]() {  // a step, the next one's disturbances on their way
    const double f1 = e1, f2 = e2;
    p1 += N;
    p2 += N;
    if (j + 1 < j_end) {
      if (ld1) e1 = __ldg(p1);
      if (ld2) e2 = __ldg(p2);
    }
    G.step(a, v, s, va, f1, f2);
    ++j;
  };
  while (j + B <= j_end && __any_sync(0xffffffffu, run)) {
    const int dead_now = (run && dead != nullptr) ? *dead : 0;
    G.live = run;
    BlockMin<double> bm;
#pragma unroll 2
    for (int u = 0; u < B; ++u) {
      one();
      bm.add(G.slack(a, s), u);
    }
    if (run) {
      const double bmin = bm.result(a, v, s);
      smin = fmin(smin, bmin);
      if (bmin < band) jl = j;
      j_stop = j;
      q_ca = a; w = v; q_sm = s; w_abs = va;
      if (smin < thr) {
        how = LANE_VIOLATED;
        run = false;
        if (dead != nullptr && G.role == 0) *dead = 1;  // the warp's other groups leave at their next look
      } else if (dead_now != 0 && j < j_end) {
        how = LANE_STOPPED;
        run = false;
      }
    }
  }
  while (j < j_end && __any_sync(0xffffffffu, run)) {
    G.live = run;
    one();
    if (run) {
      const double sl = checked_slack<double>(C, a, v, s);
      smin = fmin(smin, sl);
      if (sl < band) jl = j;
      j_stop = j;
      q_ca = a; w = v; q_sm = s; w_abs = va;
      if (sl < thr) {
        how = LANE_VIOLATED;
        run = false;
      }
    }
  }
  *steps = static_cast<unsigned>(j_stop - j0);
  *end = how;
  *jlast = jl;
  return smin;
}

// Warp minimum in the lane's own precision (a binary32 lane's value needs no
// binary64 shuffles or compares on GB300's narrow binary64 pipe).
template <typename T>
__device__ __forceinline__ T warp_min(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// One binary64 trajectory whose disturbances are regenerated from their
// Philox counters step by step (the pair was sampled in a binary32 mode, so
// its binary64 array was never written).  Same contract as run_lane over
// steps 1..H with early exit at s < thr.
__device__ __forceinline__ double run_lane_philox(const StepU<double>& K, const PowTable* pw,
                                  const StepC<double>& C, const ScenSrc& src, int k, int H, double q_ca, double w,
                                  double q_sm, double w_abs, double thr,
                                  unsigned* steps) {
  double smin = checked_slack<double>(C, q_ca, w, q_sm);
  int j = 0;
  if (!(smin < thr)) {
    while (j < H) {
      const U64x4 r = philox4x64_10(static_cast<uint64_t>(j), src.base + static_cast<uint64_t>(k), src.update,
                                    0ull, src.seed, 0ull);
      rk4_step_fast<double>(K, pw, C, q_ca, w, q_sm, w_abs, uniform_sym(r.w[0], src.amp[0]),
                            uniform_sym(r.w[1], src.amp[1]), uniform_sym(r.w[2], src.amp[2]));
      ++j;
      const double s = checked_slack<double>(C, q_ca, w, q_sm);
      smin = fmin(smin, s);
      if (s < thr) break;
    }
  }
  *steps = static_cast<unsigned>(j);
  return smin;
}

// k-section grids (Alg. 3 / Eq. 5 for round 1; M points strictly inside the
// bracket for the later rounds).
__device__ __forceinline__ int grid_points(double* cand_kappa, int M) {
  for (int i = 0; i < M; ++i)
    cand_kappa[i] = __ddiv_rn(static_cast<double>(i), static_cast<double>(M - 1));
  return M;
}

__device__ __forceinline__ int interior_points(double* cand_kappa, int M, double lo, double hi) {
  const double w = __dsub_rn(hi, lo);
  for (int i = 0; i < M; ++i)
    cand_kappa[i] = __dadd_rn(lo, __ddiv_rn(__dmul_rn(w, static_cast<double>(i + 1)),
                                            static_cast<double>(M + 1)));
  return M;
}

// ---------------------------------------------------------------------------
// One step of the simulated plant at setpoint v (Fig. 1): x_{t+1} =
// RK4(x_t, v) + (e_ca, e_w, e_sm), the plant's own draw added after the step
// as in Eq. 4.  Binary64, the rollouts' step in gauge coordinates: the plant
// sits on the closed loop's critical path.
__device__ __forceinline__ void plant_step_fast(const StepModel<double>& M, double v, const double x[3],
                                                double e_ca, double e_w, double e_sm, double x_next[3]) {
  const double q0[3] = {0.0, 0.0, 0.0};
  const StepC<double> C = step_consts<double>(M.U, M.F, fold_cand(M.c, v, q0, 0.0));
  const double p_atm = M.c.p_atm;
  double q_ca = x[0] - p_atm, w = x[1], q_sm = x[2] - p_atm, w_abs = x[1];
  rk4_step_fast<double>(M.U, M.pw, C, q_ca, w, q_sm, w_abs, e_ca, e_w, e_sm);
  x_next[0] = q_ca + p_atm;
  x_next[1] = w;
  x_next[2] = q_sm + p_atm;
}

}  // namespace rrg
