// rrg_adjoint.cu -- discrete adjoint of the robust RG objective.
//
// g(kappa) = min over scenarios k and steps j = 0..H of the slack
// s_j^k = h(x_j^k, v) - y_min, v = v_prev + kappa (r - v_prev) (Eq. 2), with
// x_{j+1} = RK4(x_j, v) + d_j^k (Eq. 4): the admissibility test of Alg. 3
// is g >= 0 (without the steady-state part).  Its derivative at the argmin
// (k*, j*) (a subgradient where the argmin is not unique) is obtained by the
// reverse (adjoint) sweep of the RK4 recursion of trajectory k* from j* back
// to 0:
//   forward  adjoint_forward_kernel: one thread per (kappa, scenario), full
//            horizon, with the rollouts' binary32/binary64 step, the state
//            saved every `checkpoint` steps, per-lane min and argmin;
//   argmin   adjoint_argmin_kernel: per kappa, the first (k, then j)
//            attaining the min;
//   reverse  adjoint_reverse_kernel: the checkpoint segments before j* are
//            recomputed in parallel, storing every step's state; from j* down,
//            32 steps at a time, every stage's Jacobian in parallel, the
//            adjoint recursion over them (three multiply-adds a stage, the
//            only serial part) and every stage's share of the constants'
//            adjoints in parallel; these are mapped to the 27 model
//            parameters, to x_t and (through the setpoint) to kappa.
#include <cfloat>
#include <cmath>

#include "rrg_device.cuh"
#include "rrg_internal.h"
#include "rrg_lane.cuh"

namespace rrg {

namespace {

// Adjoints of the constants the right-hand side and output read.
template <typename T>
struct ConstAdj {
  T a_w, a_p, k_sm, k_ca, e, C_cp, C_m, k_v, K_p, RT_Vca, RT_Vsm, inv_J, inv_p_atm;
  T W_o2, V0, y_scale;
};

// The elementary functions of the reverse sweep.  binary32: MUFU forms
// (__powf, __logf, approximate reciprocal), relative errors of a few 1e-7,
// far inside what a binary32 gradient carries anyway; binary64: x^e through
// the handle's table (pow_m1_table falls back to pow outside [1, 2) or for
// another exponent), log and IEEE division.
template <typename T> struct VjpMath;
template <>
struct VjpMath<float> {
  static __device__ __forceinline__ float pw(float x, float e, const PowTable*) { return __powf(x, e); }
  static __device__ __forceinline__ float ln(float x) { return __logf(x); }
  static __device__ __forceinline__ float inv(float x) { return __fdividef(1.0f, x); }
};
template <>
struct VjpMath<double> {
  static __device__ __forceinline__ double pw(double x, double e, const PowTable* S) {
    return pow_m1_table(S, x, e) + 1.0;
  }
  static __device__ __forceinline__ double ln(double x) { return log(x); }
  static __device__ __forceinline__ double inv(double x) { return 1.0 / x; }
};

// Vector-Jacobian product of fc3_rhs at q with output adjoint (b_ca, b_w,
// b_sm): adds J^T b to (qb_ca, qb_w, qb_sm) and the constants' adjoints to g.
template <typename T>
__device__ void fc3_rhs_vjp(const Fc3K<T>& K, const CandK<T>& C, T q_ca, T w, T q_sm, T b_ca,
                            T b_w, T b_sm, T& qb_ca, T& qb_w, T& qb_sm, ConstAdj<T>& g) {
  // forward intermediates (as in fc3_rhs)
  const T W_cp = K.a_w * w - K.a_p * q_sm;
  const T W_sm = K.k_sm * (q_sm - q_ca);
  const T W_ca = K.k_ca * q_ca;
  const T Pi = T(1) + q_sm * K.inv_p_atm;
  const T Pe = VjpMath<T>::pw(Pi, K.e, K.pws);
  const T pr = Pe - T(1);
  const T inv_w = VjpMath<T>::inv(w);
  const T tau_cp = K.C_cp * pr * W_cp * inv_w;
  const T v_cm = C.V0 - K.K_p * W_cp;
  const T tau_cm = K.C_m * (v_cm - K.k_v * w);
  // d_ca = RT_Vca (W_sm - W_ca - W_o2)
  g.RT_Vca += b_ca * (W_sm - W_ca - C.W_o2);
  T Wsm_b = K.RT_Vca * b_ca;
  const T Wca_b = -K.RT_Vca * b_ca;
  g.W_o2 += -K.RT_Vca * b_ca;
  // d_w = (tau_cm - tau_cp) inv_J
  g.inv_J += b_w * (tau_cm - tau_cp);
  const T tcm_b = K.inv_J * b_w, tcp_b = -K.inv_J * b_w;
  // d_sm = RT_Vsm (W_cp - W_sm)
  g.RT_Vsm += b_sm * (W_cp - W_sm);
  T Wcp_b = K.RT_Vsm * b_sm;
  Wsm_b += -K.RT_Vsm * b_sm;
  // tau_cm = C_m (v_cm - k_v w)
  g.C_m += tcm_b * (v_cm - K.k_v * w);
  const T vcm_b = K.C_m * tcm_b;
  T w_b = -K.C_m * K.k_v * tcm_b;
  g.k_v += -K.C_m * w * tcm_b;
  // v_cm = V0 - K_p W_cp
  g.V0 += vcm_b;
  g.K_p += -W_cp * vcm_b;
  Wcp_b += -K.K_p * vcm_b;
  // tau_cp = C_cp pr W_cp / w
  g.C_cp += tcp_b * pr * W_cp * inv_w;
  const T pr_b = tcp_b * K.C_cp * W_cp * inv_w;
  Wcp_b += tcp_b * K.C_cp * pr * inv_w;
  w_b += -tcp_b * tau_cp * inv_w;
  // pr = Pi^e - 1
  g.e += pr_b * Pe * VjpMath<T>::ln(Pi);
  const T Pi_b = pr_b * K.e * Pe * VjpMath<T>::inv(Pi);
  // Pi = 1 + q_sm inv_p_atm
  T qsm_b = Pi_b * K.inv_p_atm;
  g.inv_p_atm += Pi_b * q_sm;
  // W_ca = k_ca q_ca
  g.k_ca += Wca_b * q_ca;
  T qca_b = K.k_ca * Wca_b;
  // W_sm = k_sm (q_sm - q_ca)
  g.k_sm += Wsm_b * (q_sm - q_ca);
  qsm_b += K.k_sm * Wsm_b;
  qca_b += -K.k_sm * Wsm_b;
  // W_cp = a_w w - a_p q_sm
  g.a_w += Wcp_b * w;
  g.a_p += -Wcp_b * q_sm;
  w_b += K.a_w * Wcp_b;
  qsm_b += -K.a_p * Wcp_b;
  qb_ca += qca_b;
  qb_w += w_b;
  qb_sm += qsm_b;
}

// Stage point `stage` (0: the state itself) of the RK4 step from y, in place.
template <typename T>
__device__ __forceinline__ void rk4_stage_point(const Fc3K<T>& K, const CandK<T>& C, T dt, int stage, T y[3]) {
  const T x[3] = {y[0], y[1], y[2]};
#pragma unroll 1
  for (int u = 0; u < stage; ++u) {
    const T h = u < 2 ? T(0.5) * dt : dt;
    T a, b, c;
    fc3_rhs<T>(K, C, y[0], y[1], y[2], a, b, c);
    y[0] = x[0] + h * a;
    y[1] = x[1] + h * b;
    y[2] = x[2] + h * c;
  }
}

// Register slots of the forward pass's disturbance prefetch ring.

constexpr int kFwdRing = 8;

// The candidate constants in precision T.
template <typename T> __device__ __forceinline__ RhsC<T> launch_c(const Launch& L, int i);
template <> __device__ __forceinline__ RhsC<float> launch_c<float>(const Launch& L, int i) { return L.cand_c32[i]; }
template <> __device__ __forceinline__ RhsC<double> launch_c<double>(const Launch& L, int i) { return L.cand_c64[i]; }

// The binary32 forward pass on the stored binary32 array saves states between
// blocks of kAdjBlock steps only: the caller's spacing rounded up.
constexpr int kAdjBlock = 16;
constexpr int adj_spacing(int checkpoint) { return (checkpoint + kAdjBlock - 1) / kAdjBlock * kAdjBlock; }

// Forward: one thread per (candidate slot i = blockIdx.y, scenario k), full
// horizon, with the rollouts' arithmetic (deviation coordinates about the
// candidate's reference point, the multiplied-out right-hand side, the
// slot's constants from the candidate set-up; under parametric uncertainty
// the scenario's own model): the state x_j is saved in gauge coordinates at
// j = 0, C, 2C, ... (j < H) into ckpt[((i N + k) nseg + c) 3 + .], and the
// lane's min slack and the first step attaining it go to lane_min / lane_arg
// [i N + k].  DT: the disturbance array's type (the stored binary32 copy for
// binary32 gradients when the handle draws one, else the binary64 values
// rounded to T).  The disturbances pass through a ring of kFwdRing register
// slots: step j takes slot j % kFwdRing and refills it with step j +
// kFwdRing's values (steps past the horizon re-read the last one), so each
// load has kFwdRing steps to arrive.
template <typename T, typename DT>
__global__ void __launch_bounds__(128)
adjoint_forward_kernel(const Launch L, const DT* __restrict__ d, int checkpoint,
                       double* __restrict__ ckpt, double* __restrict__ lane_min,
                       int* __restrict__ lane_arg) {
  const int i = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int N = L.N, H = L.H;
  if (k >= N) return;
  RhsC<T> R = launch_c<T>(L, i);
  LaneModel<T> M;
  double p_atm;
  if (L.pmul != nullptr)
    p_atm = lane_model<T, true>(L, 0, k, L.cand_v[i], R, M);
  else
    p_atm = lane_model<T, false>(L, 0, k, 0.0, R, M);
  const StepU<T>& K = M.U;
  const StepC<T>& C = M.C;
  T z_ca, z_w, z_sm, w_abs;
  start_state<T>(R, L.st->x, p_atm, z_ca, z_w, z_sm, w_abs);
  const double r_ca = static_cast<double>(R.r_ca), r_w = static_cast<double>(R.r_w),
               r_sm = static_cast<double>(R.r_sm);
  const int nseg = H / checkpoint + 1;
  const size_t HN = static_cast<size_t>(H) * N;
  double* ck = ckpt + (static_cast<size_t>(i) * N + k) * nseg * 3;
  T smin = slack_of<T>(C, z_ca, z_sm);
  int arg = 0;
  int next_ck = 0;  // the next step whose state is saved
  if constexpr (sizeof(T) == 4 && sizeof(DT) == 4) {
    // binary32 from the stored binary32 array: the rollouts' ring of quads in
    // shared memory, in blocks without a branch (a warp runs its chain alone on
    // its scheduler; the state is saved between blocks, whose length the
    // spacing is a multiple of), then the last steps past a whole block
    __shared__ __align__(16) unsigned char qring[qring_bytes(128)];
    constexpr int B = kAdjBlock;
    static_assert(B == 4 * kQringBlock, "saved states lie between blocks");
    int j = 0;
    auto save = [&]() {
      if (j != next_ck) return;
      double* c = ck + (j / checkpoint) * 3;
      c[0] = static_cast<double>(z_ca) + r_ca;
      c[1] = static_cast<double>(z_w) + r_w;
      c[2] = static_cast<double>(z_sm) + r_sm;
      next_ck += checkpoint;
    };
    if (B <= H) {
      Qring<128> ring(qring, d, k, N, H, 0, H);
      do {
        save();
        int at = 0;  // step of the block that lowered the minimum last
        auto step = [&](int u, float e0, float e1, float e2) {
          rk4_step_fast<T>(K, M.pw, C, z_ca, z_w, z_sm, w_abs, e0, e1, e2);
          const T s = slack_of<T>(C, z_ca, z_sm);
          at = s < smin ? u : at;
          smin = s < smin ? s : smin;
        };
#pragma unroll
        for (int q = 0; q < kQringBlock; ++q) {
          float4 a, b, c;
          ring.next(a, b, c, [&](float e0, float e1, float e2) { step(4 * q + 1, e0, e1, e2); });
          step(4 * q + 2, a.y, b.y, c.y);
          step(4 * q + 3, a.z, b.z, c.z);
          step(4 * q + 4, a.w, b.w, c.w);
        }
        if (at) arg = j + at;
        j += B;
      } while (j + B <= H);
      ring.drain();
    }
    if (j < H) save();
    const size_t comp = quad_rows(H) * 4 * static_cast<size_t>(N);
    while (j < H) {
      const size_t o = quad_index(0, j, k, H, N);
      rk4_step_fast<T>(K, M.pw, C, z_ca, z_w, z_sm, w_abs, __ldg(d + o), __ldg(d + comp + o), __ldg(d + 2 * comp + o));
      ++j;
      const T s = slack_of<T>(C, z_ca, z_sm);
      if (s < smin) { smin = s; arg = j; }
    }
    lane_min[static_cast<size_t>(i) * N + k] = static_cast<double>(smin);
    lane_arg[static_cast<size_t>(i) * N + k] = arg;
    return;
  }
  auto at = [&](int j) { return static_cast<size_t>(j < H ? j : H - 1) * N + k; };
  T ring[kFwdRing][3];
#pragma unroll
  for (int u = 0; u < kFwdRing; ++u) {
    const size_t o = at(u);
    ring[u][0] = static_cast<T>(d[o]);
    ring[u][1] = static_cast<T>(d[HN + o]);
    ring[u][2] = static_cast<T>(d[2 * HN + o]);
  }
  for (int j0 = 0; j0 < H; j0 += kFwdRing) {
#pragma unroll
    for (int u = 0; u < kFwdRing; ++u) {
      const int j = j0 + u;
      if (j >= H) break;
      const T e0 = ring[u][0], e1 = ring[u][1], e2 = ring[u][2];
      const size_t o = at(j + kFwdRing);
      ring[u][0] = static_cast<T>(d[o]);
      ring[u][1] = static_cast<T>(d[HN + o]);
      ring[u][2] = static_cast<T>(d[2 * HN + o]);
      if (j == next_ck) {
        double* c = ck + (j / checkpoint) * 3;
        c[0] = static_cast<double>(z_ca) + r_ca;
        c[1] = static_cast<double>(z_w) + r_w;
        c[2] = static_cast<double>(z_sm) + r_sm;
        next_ck += checkpoint;
      }
      rk4_step_fast<T>(K, M.pw, C, z_ca, z_w, z_sm, w_abs, e0, e1, e2);
      const T s = slack_of<T>(C, z_ca, z_sm);
      if (s < smin) { smin = s; arg = j + 1; }
    }
  }
  lane_min[static_cast<size_t>(i) * N + k] = static_cast<double>(smin);
  lane_arg[static_cast<size_t>(i) * N + k] = arg;
}

// The binary64 forward pass with four lanes per trajectory (Coop64): the same
// states, minima and steps as adjoint_forward_kernel<double, double>.
__global__ void __launch_bounds__(128)
adjoint_forward_coop_kernel(const Launch L, const double* __restrict__ d, int checkpoint,
                            double* __restrict__ ckpt, double* __restrict__ lane_min,
                            int* __restrict__ lane_arg) {
  const int i = blockIdx.y;
  const int N = L.N, H = L.H;
  const int kt = (blockIdx.x * blockDim.x + threadIdx.x) / 4;
  const bool on = kt < N;
  const int k = on ? kt : N - 1;  // a group past the scenarios keeps its warp company
  RhsC<double> R = L.cand_c64[i];
  LaneModel<double> M;
  double p_atm;
  if (L.pmul != nullptr)
    p_atm = lane_model<double, true>(L, 0, k, L.cand_v[i], R, M);
  else
    p_atm = lane_model<double, false>(L, 0, k, 0.0, R, M);
  double a, w, s, w_abs;
  start_state<double>(R, L.st->x, p_atm, a, w, s, w_abs);
  const Coop64 G(M.U, M.pw, L.m64.pw, M.C);
  const int nseg = H / checkpoint + 1;
  const size_t HN = static_cast<size_t>(H) * N;
  double* ck = ckpt + (static_cast<size_t>(i) * N + k) * nseg * 3;
  const bool lead = on && G.role == 0;
  double smin = slack_of<double>(M.C, a, s);
  int arg = 0, next_ck = 0;
  const bool ld1 = G.role == 2, ld2 = G.role >= 2;
  const double* p1 = d + k;
  const double* p2 = p1 + (G.role == 2 ? 2 * HN : HN);
  double e1 = ld1 ? __ldg(p1) : 0.0, e2 = ld2 ? __ldg(p2) : 0.0;
  for (int j = 0; j < H; ++j) {
    const double f1 = e1, f2 = e2;
    p1 += N;
    p2 += N;
    if (j + 1 < H) {
      if (ld1) e1 = __ldg(p1);
      if (ld2) e2 = __ldg(p2);
    }
    if (j == next_ck) {
      if (lead) {
        double* c = ck + (j / checkpoint) * 3;
        c[0] = a + R.r_ca;
        c[1] = w + R.r_w;
        c[2] = s + R.r_sm;
      }
      next_ck += checkpoint;
    }
    G.step(a, w, s, w_abs, f1, f2);
    const double sl = G.slack(a, s);
    if (sl < smin) { smin = sl; arg = j + 1; }
  }
  if (lead) {
    lane_min[static_cast<size_t>(i) * N + k] = smin;
    lane_arg[static_cast<size_t>(i) * N + k] = arg;
  }
}

// Slot i = blockIdx.x: the first (k, then j) attaining the min of the
// slot's lanes; out[i * kOutStride + 0] = g, [1], [2] = k*, j* (as long long).
constexpr int kOutStride = kAdjOutStride;

// The argmin of slot i by the whole block (blockDim a power of two, at most
// the shared arrays' size): the smallest lane minimum, and among equal ones
// the smallest k, which the reduction order cannot change; written to
// o[0..2] by thread 0, visible to the block after its closing barrier.
// Compared as integers (a binary64 comparison holds the scheduler 64 cycles);
// -0 equals 0 and a NaN is never the least.
constexpr int kArgminWarps = 8;  // of a block, at most
__device__ void block_argmin(const double* __restrict__ lm, const int* __restrict__ la, int N, double* o) {
  __shared__ unsigned long long sv[kArgminWarps];
  __shared__ int sk[kArgminWarps];
  unsigned long long best = dkey(INFINITY);
  int bk = 0x7fffffff;
#pragma unroll 8
  for (int k = threadIdx.x; k < N; k += blockDim.x) {  // ascending k: the first of equal values stays
    const long long u = __double_as_longlong(__ldg(lm + k));
    const unsigned long long mag = static_cast<unsigned long long>(u) & 0x7fffffffffffffffull;
    const unsigned long long key = mag == 0ull ? dkey(0.0) : dkey(__longlong_as_double(u));
    if (mag <= 0x7ff0000000000000ull && (key < best || (key == best && k < bk))) { best = key; bk = k; }
  }
  auto fold = [&](unsigned long long key, int kk) {
    if (key < best || (key == best && kk < bk)) { best = key; bk = kk; }
  };
#pragma unroll
  for (int w = 16; w > 0; w >>= 1)
    fold(__shfl_xor_sync(0xffffffffu, best, w), __shfl_xor_sync(0xffffffffu, bk, w));
  if ((threadIdx.x & 31) == 0) {
    sv[threadIdx.x >> 5] = best;
    sk[threadIdx.x >> 5] = bk;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) fold(sv[w], sk[w]);
    const bool found = bk >= 0 && bk < N;
    long long kj[2] = {bk, found ? la[bk] : 0};
    o[0] = found ? lm[bk] : INFINITY;
    memcpy(o + 1, kj, sizeof kj);
  }
  __syncthreads();
}

__global__ void adjoint_argmin_kernel(const double* __restrict__ lane_min,
                                      const int* __restrict__ lane_arg, int N, double* out) {
  const int i = blockIdx.x;
  block_argmin(lane_min + static_cast<size_t>(i) * N, lane_arg + static_cast<size_t>(i) * N, N,
               out + static_cast<size_t>(i) * kOutStride);
}

// Values stored per step of the recomputed trajectory: x_j.
constexpr int kSegVals = 3;
constexpr int kRevThreads = 128;
constexpr int kRevSteps = kRevThreads / 4;  // steps of a sweep's chunk: one thread per stage

// States of segment c of the trajectory (steps j0 .. j1 - 1, and j1 if it is
// j*) from its checkpoint, by the rollouts' step in deviation coordinates;
// the disturbances of four steps are fetched while the four before them run.
template <typename T, typename DT>
__device__ __forceinline__ void segment_states(const LaneModel<T>& M, const RhsC<T>& R, const DT* __restrict__ d, int k,
                                               int N, int H, const double* __restrict__ ck, int j0, int j1, bool last,
                                               T* __restrict__ seg) {
  T z_ca = static_cast<T>(ck[0] - static_cast<double>(R.r_ca)), z_w = static_cast<T>(ck[1] - static_cast<double>(R.r_w)),
    z_sm = static_cast<T>(ck[2] - static_cast<double>(R.r_sm));
  T w_abs = z_w + R.r_w;
  T e[3][4], f[3][4];
  auto load = [&](int j) {  // steps j .. j + 3 (those before j1)
    if constexpr (sizeof(DT) == 4) {  // the handle's binary32 quads; j is a multiple of 4
      const size_t comp = 4 * quad_rows(H) * static_cast<size_t>(N);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float4 v = j < j1 ? __ldg(reinterpret_cast<const float4*>(d + quad_index(0, j, k, H, N) + c * comp))
                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        f[c][0] = v.x; f[c][1] = v.y; f[c][2] = v.z; f[c][3] = v.w;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          f[c][u] = j + u < j1 ? static_cast<T>(__ldg(d + (static_cast<size_t>(c) * H + j + u) * N + k)) : T(0);
    }
  };
  auto store = [&](int j) {
    T* sj = seg + static_cast<size_t>(j) * kSegVals;
    sj[0] = z_ca + R.r_ca;
    sj[1] = w_abs;
    sj[2] = z_sm + R.r_sm;
  };
  load(j0);
#pragma unroll 1
  for (int j = j0; j < j1; j += 4) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int u = 0; u < 4; ++u) e[c][u] = f[c][u];
    load(j + 4);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j + u < j1) {
        store(j + u);
        rk4_step_fast<T>(M.U, M.pw, M.C, z_ca, z_w, z_sm, w_abs, e[0][u], e[1][u], e[2][u]);
      }
  }
  if (last) store(j1);
}

// The same with four lanes per binary64 trajectory (Coop64), by every lane of
// the warp; `n`: steps the warp runs (its longest segment's).
__device__ __forceinline__ void segment_states_coop(const LaneModel<double>& M, const PowTable* any,
                                                    const RhsC<double>& R, const double* __restrict__ d, int k, int N,
                                                    int H, const double* __restrict__ ck, int j0, int j1, int n, bool on,
                                                    bool last, double* __restrict__ seg) {
  Coop64 G(M.U, M.pw, any, M.C);
  double a = ck[0] - R.r_ca, w = ck[1] - R.r_w, s = ck[2] - R.r_sm;
  double w_abs = w + R.r_w;
  const size_t HN = static_cast<size_t>(H) * N;
  const bool ld1 = G.role == 2, ld2 = G.role >= 2;
  const double* p1 = d + static_cast<size_t>(j0) * N + k;
  const double* p2 = p1 + (G.role == 2 ? 2 * HN : HN);
  double e1 = ld1 && j0 < j1 ? __ldg(p1) : 0.0, e2 = ld2 && j0 < j1 ? __ldg(p2) : 0.0;
  auto store = [&](int j) {
    double* sj = seg + static_cast<size_t>(j) * kSegVals;
    sj[0] = a + R.r_ca;
    sj[1] = w_abs;
    sj[2] = s + R.r_sm;
  };
#pragma unroll 1
  for (int j = j0; j < j0 + n; ++j) {
    const bool mine = on && j < j1;
    if (mine && G.role == 0) store(j);
    const double f1 = e1, f2 = e2;
    p1 += N;
    p2 += N;
    if (j + 1 < j1) {
      if (ld1) e1 = __ldg(p1);
      if (ld2) e2 = __ldg(p2);
    }
    G.live = mine;
    G.step(a, w, s, w_abs, f1, f2);
    if (mine && last && j + 1 == j1 && G.role == 0) store(j1);
  }
}

// Reverse sweep of trajectory k* from j* to 0, then the chain rule from the
// folded constants to the model parameters and kappa.  One block:
//   phase 1: the checkpoint segments before j* are recomputed in parallel,
//     one thread (binary64: four lanes) a segment: x_j into seg[3 j ..];
//   phase 2: 32 steps at a time from j* down, one thread per (step, stage):
//     the stage point and the two state-dependent entries of its Jacobian
//     (the others are products of constants); three lanes then run the
//     adjoint recursion, lane r its component r, leaving every stage's adjoint
//     in shared memory, from which each thread adds its stage's share of the
//     constants' adjoints (fc3_rhs_vjp);
//   phase 3: their sum over the block, and the chain rule with every quotient
//     on a lane of its own.
// The recursion is the only serial part: 5 instructions a stage where one
// thread evaluated power, logarithm and quotients of every stage in turn.
// Measured on GB300 (a call, two kappas, 512 scenarios of 1,000 steps): j* = 530
// binary64 10.3 -> 2.66 ms, binary32 587 -> 209 us; j* = 0 binary32 156 -> 146.
// seg: scratch of (j* + 1) * kSegVals values (at most (H + 1) * kSegVals).
// out[0] = dg/dkappa, out[1..3] = dg/dx_t, out[4..4+NPARAM) = dg/dtheta.
template <typename T, typename DT>
__global__ void __launch_bounds__(kRevThreads)
adjoint_reverse_kernel(const Launch L, const DT* __restrict__ d,
                       int checkpoint, const double* __restrict__ ckpt, T* __restrict__ seg_all,
                       double* __restrict__ out_all, int slot0, const double* __restrict__ lane_min,
                       const int* __restrict__ lane_arg, double* out_h, int32_t* ss_h) {
  const int i = slot0 + static_cast<int>(blockIdx.x);  // candidate slot
  const int N = L.N, H = L.H;
  // the inputs of the candidate set-up the forward pass ran on
  const double v_prev = L.st->v_prev, r = L.st->r;
  double* o = out_all + static_cast<size_t>(i) * kOutStride;
  // the argmin first, by this block (one launch fewer than a separate pass)
  if (lane_min != nullptr)
    block_argmin(lane_min + static_cast<size_t>(i) * N, lane_arg + static_cast<size_t>(i) * N, N, o);
  long long kj[2];
  memcpy(kj, o + 1, sizeof kj);
  double* out = o + 3;
  // the slot's outputs in pinned host memory as well (out_h may be null)
  auto to_host = [&]() {
    if (out_h == nullptr) return;
    for (int u = threadIdx.x; u < kOutStride; u += kRevThreads) out_h[static_cast<size_t>(i) * kOutStride + u] = o[u];
    if (threadIdx.x == 0) ss_h[i] = L.cand_ss[i];
  };
  T* seg = seg_all + static_cast<size_t>(i) * (H + 1) * kSegVals;
  const double v = L.cand_v[i];
  if (kj[0] < 0 || kj[0] >= N || kj[1] < 0 || kj[1] > H) {  // no argmin: same for every thread
    if (threadIdx.x < 4 + RRG_NPARAM) out[threadIdx.x] = NAN;
    __syncthreads();
    to_host();
    return;
  }
  const int k = static_cast<int>(kj[0]), jstar = static_cast<int>(kj[1]);
  // the scenario's constants: the launch's, folded again under parametric uncertainty
  __shared__ double P[RRG_NPARAM];
  if (threadIdx.x < RRG_NPARAM)
    P[threadIdx.x] = L.pmul ? __dmul_rn(L.params[threadIdx.x], L.pmul[static_cast<size_t>(k) * RRG_NPARAM + threadIdx.x])
                            : L.params[threadIdx.x];
  __syncthreads();
  Fc3K<double> K64 = L.k64;
  Fc3K<float> K32 = L.k32;
  CandK<double> C64;
  RhsC<T> R = launch_c<T>(L, i);
  LaneModel<T> M;
  if (L.pmul != nullptr) {
    fold_constants(P, &K64, &K32);
    K64.pws = (L.k64.pws != nullptr && L.k64.pws->e == K64.e) ? L.k64.pws : nullptr;
    C64 = cand_consts(P, v);
    lane_model<T, true>(L, 0, k, v, R, M);
  } else {
    C64.W_o2 = __dmul_rn(L.eq.w1, v);
    C64.V0 = fma_rn(fma_rn(L.eq.v2, v, L.eq.v1), v, L.eq.v0);
    C64.y_scale = L.cand_c64[i].y_scale;
    lane_model<T, false>(L, 0, k, v, R, M);
  }
  Fc3K<T> K;
  CandK<T> C;
  if constexpr (sizeof(T) == 8) {
    K = K64;
    C = C64;
  } else {
    K = K32;
    C = cand_round(C64);
  }
  const T dt = static_cast<T>(L.dt);
  const int nseg = H / checkpoint + 1;
  const double* ck = ckpt + (static_cast<size_t>(i) * N + k) * nseg * 3;
  // phase 1: segment c covers steps c * checkpoint .. min((c + 1) * checkpoint, j*) - 1
  const int nc = jstar > 0 ? (jstar - 1) / checkpoint + 1 : 0;
  bool coop = false;
  if constexpr (sizeof(T) == 8) {
    coop = L.m64.pw != nullptr;
    if (coop) {
      for (int c0 = static_cast<int>(threadIdx.x >> 5) * 8; c0 < nc; c0 += kRevThreads / 4) {  // the warp's first segment
        const int c = c0 + static_cast<int>((threadIdx.x & 31) >> 2);
        const bool on = c < nc;
        const int j0 = (on ? c : nc - 1) * checkpoint;
        const int j1 = (j0 + checkpoint < jstar) ? j0 + checkpoint : jstar;
        const int n = jstar - c0 * checkpoint < checkpoint ? jstar - c0 * checkpoint : checkpoint;
        segment_states_coop(M, L.m64.pw, R, d, k, N, H, ck + static_cast<size_t>(on ? c : nc - 1) * 3, j0, j1, n, on,
                            j1 == jstar, seg);
      }
    }
  }
  if (!coop)
    for (int c = threadIdx.x; c < nc; c += kRevThreads) {
      const int j0 = c * checkpoint;
      const int j1 = (j0 + checkpoint < jstar) ? j0 + checkpoint : jstar;
      segment_states<T, DT>(M, R, d, k, N, H, ck + static_cast<size_t>(c) * 3, j0, j1, j1 == jstar, seg);
    }
  __syncthreads();
  // output at j*: s = y_scale (q_sm - q_ca) - y_min (x_0 is checkpoint 0)
  T q_ca, q_sm;
  if (jstar == 0) {
    q_ca = static_cast<T>(ck[0]);
    q_sm = static_cast<T>(ck[2]);
  } else {
    q_ca = seg[static_cast<size_t>(jstar) * kSegVals];
    q_sm = seg[static_cast<size_t>(jstar) * kSegVals + 2];
  }
  // phase 2
  __shared__ T jac[kRevThreads][2];  // d(dw)/dw, d(dw)/d(p_sm) of (step, stage) 4 u + stage
  __shared__ T adj[kRevThreads][3];  // its adjoint
  const int stage = threadIdx.x & 3, step = threadIdx.x >> 2, comp = threadIdx.x < 3 ? static_cast<int>(threadIdx.x) : 2;
  const T h2 = T(0.5) * dt, h6 = dt / T(6);
  const T cA = comp == 0 ? -(K.k_ca + K.k_sm) * K.RT_Vca : comp == 1 ? T(0) : K.k_sm * K.RT_Vca;
  const T cS = comp == 0 ? K.k_sm * K.RT_Vsm : comp == 1 ? K.a_w * K.RT_Vsm : -(K.k_sm + K.a_p) * K.RT_Vsm;
  T l = comp == 0 ? -C.y_scale : comp == 1 ? T(0) : C.y_scale;  // warp 0, lane r: the adjoint's component r
  ConstAdj<T> g{};
  for (int jt = jstar - 1; jt >= 0; jt -= kRevSteps) {  // chunk of steps jt, jt - 1, ...
    const int j = jt - step, n = jt + 1 < kRevSteps ? jt + 1 : kRevSteps;
    T y[3];
    if (step < n) {
#pragma unroll
      for (int u = 0; u < 3; ++u) y[u] = seg[static_cast<size_t>(j) * kSegVals + u];
      rk4_stage_point<T>(K, C, dt, stage, y);
      ConstAdj<T> unused{};
      T ja = T(0), jw = T(0), js = T(0);
      fc3_rhs_vjp<T>(K, C, y[0], y[1], y[2], T(0), T(1), T(0), ja, jw, js, unused);
      jac[threadIdx.x][0] = jw;
      jac[threadIdx.x][1] = js;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      auto from = [&](T x, int lane) { return __shfl_sync(0xffffffffu, x, lane); };
#pragma unroll 1
      for (int u = 0; u < n; ++u) {
        T cw[4];
#pragma unroll
        for (int st = 0; st < 4; ++st) cw[st] = comp == 0 ? T(0) : jac[4 * u + st][comp - 1 > 0];
        const T hl = h6 * l;
        T b = hl, q = l;
#pragma unroll
        for (int st = 3; st >= 0; --st) {
          if (threadIdx.x < 3) adj[4 * u + st][threadIdx.x] = b;
          const T yb = cA * from(b, 0) + (cw[st] * from(b, 1) + cS * from(b, 2));
          q += yb;
          if (st == 3) b = T(2) * hl + dt * yb;
          else if (st == 2) b = T(2) * hl + h2 * yb;
          else if (st == 1) b = hl + h2 * yb;
        }
        l = q;
      }
    }
    __syncthreads();
    if (step < n) {
      T ja = T(0), jw = T(0), js = T(0);
      fc3_rhs_vjp<T>(K, C, y[0], y[1], y[2], adj[threadIdx.x][0], adj[threadIdx.x][1], adj[threadIdx.x][2], ja, jw, js,
                     g);
    }
  }
  // phase 3: sums over the block, thread (v, s) = (t / 8, t % 8) a part of sum v
  constexpr int kAdj = 15;  // ConstAdj without y_scale
  __shared__ T part[kAdj][kRevThreads];
  __shared__ double tot[16], num[32], den[32], th[RRG_NPARAM], quo[32], lam_x[3];
  const T gv[kAdj] = {g.a_w, g.a_p, g.k_sm, g.k_ca, g.e, g.C_cp, g.C_m, g.k_v, g.K_p, g.RT_Vca, g.RT_Vsm, g.inv_J,
                      g.inv_p_atm, g.W_o2, g.V0};
#pragma unroll
  for (int u = 0; u < kAdj; ++u) part[u][threadIdx.x] = gv[u];
  if (threadIdx.x < 3) lam_x[threadIdx.x] = static_cast<double>(l);
  __syncthreads();
  {
    const int u = threadIdx.x >> 3;
    T s = T(0);
    if (u < kAdj)
      for (int t = threadIdx.x & 7; t < kRevThreads; t += 8) s += part[u][t];
#pragma unroll
    for (int w = 4; w > 0; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
    if ((threadIdx.x & 7) == 0) tot[u] = static_cast<double>(s);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    // chain rule to the parameter vector (binary64): numerators and
    // denominators by lane 0, the quotients by the lanes
    const double g_a_w = tot[0], g_a_p = tot[1], g_k_sm = tot[2], g_k_ca = tot[3], g_e = tot[4], gc = tot[5], gm = tot[6],
                 g_k_v = tot[7], g_K_p = tot[8], ga = tot[9], gs = tot[10], gJ = tot[11], gp = tot[12], gW_o2 = tot[13],
                 gV0 = tot[14], gy = static_cast<double>(q_sm - q_ca);
    const double I = v, W_o2 = C64.W_o2, y_scale = C64.y_scale;
    const double lam = P[P_LAM_REF], xo2 = P[P_X_O2], Kp = P[P_K_P], gamma = P[P_GAMMA];
    if (threadIdx.x == 0) {
      auto set = [&](int q, double a, double b) {
        num[q] = a;
        den[q] = b;
      };
      set(0, gy * y_scale, P[P_K_SM]);
      set(1, g_e, gamma * gamma);
      set(2, gc * P[P_T_ATM], P[P_ETA_CP]);
      set(3, gc * P[P_C_P], P[P_ETA_CP]);
      set(4, -gc * K64.C_cp, P[P_ETA_CP]);
      set(5, gm * P[P_K_T], P[P_R_CM]);
      set(6, gm * P[P_ETA_CM], P[P_R_CM]);
      set(7, -gm * K64.C_m, P[P_R_CM]);
      set(8, ga * P[P_T_ST], P[P_V_CA]);
      set(9, gs * P[P_T_ST], P[P_V_SM]);
      set(10, ga * P[P_R_A], P[P_V_CA]);
      set(11, gs * P[P_R_A], P[P_V_SM]);
      set(12, -ga * K64.RT_Vca, P[P_V_CA]);
      set(13, -gs * K64.RT_Vsm, P[P_V_SM]);
      set(14, -gJ, P[P_J_CP] * P[P_J_CP]);
      set(15, -gp, P[P_P_ATM] * P[P_P_ATM]);
      const double vk = gV0 * Kp, vl = gV0 * lam * W_o2, yg = gy * y_scale;
      set(16, vk * lam, xo2);
      set(17, yg, W_o2);
      set(18, vl, xo2);
      set(19, vk * W_o2, xo2);
      set(20, -vk * lam * W_o2, xo2 * xo2);
      set(21, yg, xo2);
    }
    __syncwarp();
    if (threadIdx.x < 22) quo[threadIdx.x] = num[threadIdx.x] / den[threadIdx.x];
    __syncwarp();
    const double gW = gW_o2 + quo[16] - quo[17];
    if (threadIdx.x < 4) {
      const double a = threadIdx.x == 2 ? -(gW * W_o2) : gW * W_o2;
      const double b = threadIdx.x == 0 ? P[P_M_O2] : threadIdx.x == 1 ? P[P_N_CELL] : threadIdx.x == 2 ? P[P_FARADAY] : I;
      quo[22 + threadIdx.x] = a / b;
    }
    if (threadIdx.x < RRG_NPARAM) th[threadIdx.x] = 0.0;
    __syncwarp();
    if (threadIdx.x == 0) {
      th[P_A_W] = g_a_w;
      th[P_A_P] = g_a_p;
      th[P_K_SM] = g_k_sm + quo[0];
      th[P_K_CA] = g_k_ca;
      th[P_GAMMA] = quo[1];
      th[P_C_P] = quo[2];
      th[P_T_ATM] = quo[3];
      th[P_ETA_CP] = quo[4];
      th[P_ETA_CM] = quo[5];
      th[P_K_T] = quo[6];
      th[P_R_CM] = quo[7];
      th[P_K_V] = g_k_v;
      th[P_K_P] = g_K_p + quo[18];
      th[P_R_A] = quo[8] + quo[9];
      th[P_T_ST] = quo[10] + quo[11];
      th[P_V_CA] = quo[12];
      th[P_V_SM] = quo[13];
      th[P_J_CP] = quo[14];
      // p_atm: through 1/p_atm and through q_0 = x_t - p_atm (pressures)
      th[P_P_ATM] = quo[15] - lam_x[0] - lam_x[2];
      th[P_M_O2] = quo[22];
      th[P_N_CELL] = quo[23];
      th[P_FARADAY] = quo[24];
      th[P_C0] = gV0;
      th[P_C1] = gV0 * I;
      th[P_C2] = gV0 * I * I;
      th[P_LAM_REF] = quo[19];
      th[P_X_O2] = quo[20] + quo[21];
      const double dI = quo[25] + gV0 * (P[P_C1] + 2.0 * P[P_C2] * I);
      out[0] = dI * (r - v_prev);
    }
    if (threadIdx.x < 3) out[1 + threadIdx.x] = lam_x[threadIdx.x];
    __syncwarp();
    // theta'_p = theta_p m_p^{k*}: back to the nominal parameters
    if (threadIdx.x < RRG_NPARAM)
      out[4 + threadIdx.x] =
          L.pmul ? th[threadIdx.x] * L.pmul[static_cast<size_t>(k) * RRG_NPARAM + threadIdx.x] : th[threadIdx.x];
  }
  __syncthreads();
  to_host();
}

}  // namespace

// Host side.  launch_adjoint_forward enqueues the forward pass and the
// argmin for the m candidate slots the last candidate set-up prepared
// (kappas in cand_kappa); launch_adjoint_reverse the reverse sweeps of slots
// slot0 .. slot0 + count - 1 on the states the forward pass saved.
// ckpt: m N (H / checkpoint + 1) 3 doubles; lane_min / lane_arg: m N each;
// seg: m (H + 1) 3 values of T; d_out: m kOutStride doubles (per slot: g,
// k*, j*, then dg/dkappa, dg/dx_t, dg/dtheta).  fwd_begin / fwd_end (either
// may be null): events around the forward kernel.  The binary32 gradient
// reads the stored binary32 disturbances when the handle draws them (the
// values its binary32 rollouts use), otherwise the binary64 array (filled by
// the caller) rounded to binary32.
namespace {
bool reads32(const Launch& L, bool fp64) { return !fp64 && L.precision != RRG_FP64 && !L.scen_gen; }
}  // namespace

cudaError_t launch_adjoint_forward(const Launch& L, bool fp64, int m, int checkpoint, double* ckpt,
                                   double* lane_min, int* lane_arg, double* d_out,
                                   cudaEvent_t fwd_begin, cudaEvent_t fwd_end, bool argmin) {
  // one warp per block until blocks of 128 threads would fill every SM:
  // each scenario is one dependent chain, so spreading them over SMs costs
  // nothing
  if (L.sms <= 0 || m < 1) return cudaErrorInvalidConfiguration;
  const long long lanes = static_cast<long long>(L.N) * m;
  const int threads = (lanes >= 128LL * L.sms) ? 128 : 32;
  const dim3 grid((L.N + threads - 1) / threads, m);
  if (fwd_begin) {
    const cudaError_t er = cudaEventRecord(fwd_begin, L.stream);
    if (er != cudaSuccess) return er;
  }
  // four lanes per binary64 trajectory by the rollouts' rule
  const bool coop = fp64 && coop64_fits(L, m);
  if (coop)
    adjoint_forward_coop_kernel<<<dim3((L.N + 7) / 8, m), 32, 0, L.stream>>>(L, L.d64, checkpoint, ckpt, lane_min,
                                                                             lane_arg);
  else if (fp64)
    adjoint_forward_kernel<double, double><<<grid, threads, 0, L.stream>>>(L, L.d64, checkpoint, ckpt,
                                                                           lane_min, lane_arg);
  else if (reads32(L, fp64))
    adjoint_forward_kernel<float, float><<<grid, threads, 0, L.stream>>>(L, L.d32, adj_spacing(checkpoint), ckpt,
                                                                         lane_min, lane_arg);
  else
    adjoint_forward_kernel<float, double><<<grid, threads, 0, L.stream>>>(L, L.d64, checkpoint, ckpt,
                                                                          lane_min, lane_arg);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (fwd_end) {
    e = cudaEventRecord(fwd_end, L.stream);
    if (e != cudaSuccess) return e;
  }
  if (argmin) adjoint_argmin_kernel<<<m, 256, 0, L.stream>>>(lane_min, lane_arg, L.N, d_out);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_reverse(const Launch& L, bool fp64, int slot0, int count, int checkpoint,
                                   const double* ckpt, void* seg, double* d_out, const double* lane_min,
                                   const int* lane_arg, double* out_h, int32_t* ss_h) {
  if (count < 1 || slot0 < 0) return cudaErrorInvalidConfiguration;
  if (fp64)
    adjoint_reverse_kernel<double, double><<<count, kRevThreads, 0, L.stream>>>(
        L, L.d64, checkpoint, ckpt, static_cast<double*>(seg), d_out, slot0, lane_min, lane_arg, out_h,
        ss_h);
  else if (reads32(L, fp64))
    adjoint_reverse_kernel<float, float><<<count, kRevThreads, 0, L.stream>>>(
        L, L.d32, adj_spacing(checkpoint), ckpt, static_cast<float*>(seg), d_out, slot0, lane_min, lane_arg, out_h,
        ss_h);
  else
    adjoint_reverse_kernel<float, double><<<count, kRevThreads, 0, L.stream>>>(
        L, L.d64, checkpoint, ckpt, static_cast<float*>(seg), d_out, slot0, lane_min, lane_arg, out_h,
        ss_h);
  return cudaGetLastError();
}

}  // namespace rrg
