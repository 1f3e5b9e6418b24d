// rrg_internal.h -- types shared by the kernels (rrg_kernels.cu) and the
// host side of the C ABI (rrg_capi.cu).  Not part of the public interface.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/rrg.h"

#include "rrg_device.cuh"

namespace rrg {

// FC3 parameter indices (the layout documented in rrg.h).
enum ParamIdx {
  P_P_ATM = 0, P_T_ATM, P_T_ST, P_R_A, P_V_SM, P_V_CA, P_K_SM, P_K_CA,
  P_N_CELL, P_FARADAY, P_M_O2, P_X_O2, P_GAMMA, P_C_P, P_ETA_CP, P_J_CP,
  P_ETA_CM, P_K_T, P_K_V, P_R_CM, P_A_W, P_A_P, P_LAM_REF, P_K_P,
  P_C0, P_C1, P_C2, P_COUNT
};
static_assert(P_COUNT == RRG_NPARAM, "parameter layout");

constexpr int kMaxTreeNodes = 2 * RRG_MAX_CANDIDATES;

// What the blocks of one rollout launch do with their candidate slot.
enum SegMode : int32_t {
  SEG_FULL = 0,      // steps 0..H
  SEG_PROBE = 1,     // steps 0..probe_steps; survivors save their state
  SEG_CONTINUE = 2,  // resume a probed trajectory at probe_steps, run to H;
                     // row y continues slot cont_slot[y]
};

// A launch covers up to two slot ranges: blockIdx.y < seg[0].count maps to
// slot seg[0].base + y, the next seg[1].count rows to seg[1].base + ...
struct Seg {
  int32_t mode, count, base;
};

// Saved state of a probed trajectory (status 0: still running, continue it;
// 1: finished in the probe and already reduced).
template <typename T>
struct LaneState {
  T q[3];         // deviation from the candidate's reference point
  T w_abs;        // the absolute speed carried with it
  T smin;
  int32_t status;
  int32_t jlast;  // last step with slack below the recheck band so far (-1: none)
};

// Origin of a scenario pair.  In the binary32 modes the sampler writes only
// the binary32 copy; the binary64 values (needed by the few rechecked
// trajectories) are regenerated from the same Philox counters on demand.
struct ScenSrc {
  int32_t d64_valid;     // 1: the binary64 array holds the values
  int32_t pad;
  unsigned long long seed, update;
  unsigned long long base;  // global index of scenario 0 (the Philox counter's k)
  double amp[3];
};

// Device-resident state of one RG update's search (one per handle).
struct SearchState {
  double x[3];        // x_t (absolute coordinates)
  double v_prev, r;   // v_{t-1}, r_t
  double lo, hi;      // bisection bracket / k-section bracket
  double kappa;       // next kappa Alg. 1 would test
  double kappa_opt;   // best admissible kappa so far
  int32_t iter;       // Alg. 1 iterations consumed
  int32_t any;        // some evaluated candidate was admissible
  int32_t done;       // search finished; outputs written
  int32_t flags;      // RRG flags of the result
  int32_t m;          // candidates of the current round
  int32_t depth;      // tree levels of the current round (bisection)
  int32_t round;      // rounds finished
  int32_t invalid;    // inputs rejected on the device
  double v_t_out;     // governed reference of the finished search
  int32_t buf;        // scenario pair of the current update (0: d64/d32, 1: d64b/d32b)
  ScenSrc src[2];     // where each pair's binary64 values are
  Seg seg[2];         // what the next rollout launch runs
  int32_t prep_base;  // slots the next prepare launch fills: prep_base ..
  int32_t prep_m;     //   prep_base + prep_m - 1
  // pipelined first round of the speculative bisection: the round is probed,
  // the next tree is built from the provisional outcomes, and both run
  // together; the real outcomes are compared with the provisional ones
  int32_t probe;      // 1 while a probed round awaits validation
  int32_t depth1;     // levels of the tree built from provisional outcomes
  int32_t prov_len, prov_done;
  uint32_t prov_bits;
  int32_t cont_slot[16];  // the probed round's slots on the provisional path
  double w_lo, w_hi, w_kappa, w_kopt;  // search state before the probed round
  int32_t w_iter, w_any;
  int32_t slot_of_node[kMaxTreeNodes];   // bisection tree: heap node -> slot
  int32_t slot_of_node1[kMaxTreeNodes];  // tree of the pipelined second round
  int32_t passed[RRG_MAX_CANDIDATES];  // trajectories that passed, per slot (Launch::top_down)
  // A round whose launch is held to one candidate's warps (Launch::held): which
  // launch runs slot i (1, 2; 0: not settled yet), and whether a candidate ran long
  // before it violated.
  int32_t row_launch[RRG_MAX_CANDIDATES];
  int32_t late;
};

// Device counters of a handle.
struct DevStats {
  unsigned long long lane_steps;
  unsigned long long lane_steps_fp64;
  unsigned long long rechecked;
  unsigned long long repairs;   // probed rounds whose provisional outcome was wrong
  // kernels, rollout launches and search rounds run by the conditional body
  // of a captured closed-loop update (counted by the kernel that opens it)
  unsigned long long cond_launches, cond_rollouts, cond_rounds;
  unsigned long long lane_steps_paired;  // of lane_steps, run two trajectories per thread
  unsigned long long wait_timeouts;      // bounded waits that gave up (TMA ring copies)
  unsigned long long lane_steps_tma;     // of lane_steps, fed by the TMA ring
};

// Closed-loop device state.
struct LoopState {
  double x[3];
  double v_prev;
  unsigned long long t;   // updates done since the loop started
};

// Search configuration passed by value to the search kernels.
struct SearchCfg {
  int search;        // RRG_SEARCH_*
  int m_cap;         // candidates per round
  int n_bisect;      // N_kappa
  int n_rounds;      // k-section rounds
  int ss_check;
  int probe_steps;   // > 0: pipeline the first two bisection rounds
  double y_min;
};

// One model's constants in the form the rollouts use: what the candidate
// constants need (binary64), the step's coefficients and what carries the
// candidate constants through the stages (StepU, StepPhi).
struct ModelC {
  double l_ca, l_cs;        // d_ca = -l_ca ca + l_cs sm - b_ca v
  double l_ww, l_ws;        // d_w  = -l_ww w + l_ws sm + d0 + v (d1 + d2 v) - N
  double l_sa, l_sw, l_ss;  // d_sm = l_sa ca + l_sw w - l_ss sm
  double b_ca, d0, d1, d2;
  double ky;                // OER per pascal: ky / v
  double p_atm, inv_p_atm;
};
// A setpoint's constants of the equilibrium solve, folded from the parameters
// (binary64: W_o2 = w1 v, V0 = v0 + v (v1 + v2 v), no division left per
// candidate), the solve's first guess over W_o2, and the threshold of the
// steady-state check with the binary32 values outside which a binary32
// solution decides it.
struct EqModel {
  double w1, v0, v1, v2;
  double thr_ss;
  float guess, y_fail, y_pass;  // y32 < y_fail: fails, y32 > y_pass: passes
};
template <typename T>
struct StepModel {
  ModelC c;
  StepU<T> U;
  StepPhi<T> F;
  const PowTable* pw;       // binary64 x^e - 1 (device memory; nullptr: pow)
};

// The model of every scenario of a pair under parametric uncertainty, folded
// once per draw for the binary32 rollouts; arrays over the scenarios, so a
// warp's reads are coalesced: value j of scenario k at [j * N + k].
constexpr int kFoldDoubles = sizeof(ModelC) / sizeof(double);
constexpr int kFoldFloats = (sizeof(StepU<float>) + sizeof(StepPhi<float>)) / sizeof(float);
struct ScenFold {
  double* d;   // [kFoldDoubles][N]: ModelC
  float* f;    // [kFoldFloats][N]: StepU<float>, StepPhi<float>
};

// Everything a launch needs; filled by the host side from the handle.
struct Launch {
  cudaStream_t stream;
  int N, H, precision, early_exit, m_cap;
  int scen_gen;                 // disturbances drawn inside the trajectory loop
  unsigned long long kbase;     // global index of the handle's scenario 0 (scenario sharding)
  int pair;                     // RRG_PAIR_*: two candidates per thread in binary32 rollouts
                                //   of full-horizon rows (never, launches that fill the SMs, always)
  // conditional-node handle of a captured closed-loop update (0: none); the
  // search kernel that validates the pipelined rounds sets it to "the search
  // is not finished", which runs the remaining rounds
  unsigned long long cond;
  uint32_t cond_launches, cond_rollouts, cond_rounds;  // what one run of that body launches
  double dt, y_min, eps_abs;
  SearchCfg scfg;
  const double* params;         // [RRG_NPARAM] (device)
  Fc3K<double> k64;             // folded model constants, passed by value
  Fc3K<float> k32;
  StepModel<double> m64;        // the rollout step's coefficients
  alignas(16) double m32_line;  // m32, and its U, 8 bytes past a 16-byte line (launch_rollout)
  StepModel<float> m32;
  double* d64;                  // scenarios [3][H][N]
  int quads;                    // d32 is in the quad layout (0: the caller's [3][H][N])
  float* d32;
  double* d64b;                 // second pair for closed loops (sampling of update t+1
  float* d32b;                  //   overlaps update t), or nullptr
  SearchState* st;
  double* cand_kappa;
  double* cand_v;
  RhsC<double>* cand_c64;       // per-slot rollout constants of the candidate
  RhsC<float>* cand_c32;
  int32_t* cand_ok;    // AND of the round's trajectory decisions
  int32_t* cand_dead;  // set once the candidate is known to fail
  int32_t* cand_ss;    // steady-state check passed
  unsigned long long* cand_min;
  uint32_t* recheck_list;
  uint32_t* recheck_jlast;      // per entry: the recheck runs steps 0..jlast
  uint32_t* recheck_count;
  DevStats* stats;
  uint8_t* P;                   // optional
  int recheck_blocks;
  int sms;                      // streaming multiprocessors of the device (> 0; launches
                                //   refuse a descriptor without it)
  int probe_steps;              // steps of a SEG_PROBE segment
  void* lane_state;             // LaneState<T>[m_cap * N] for probed rounds
  // parametric uncertainty: per-scenario parameter multipliers m[k * NPARAM
  // + p] of each scenario pair (nullptr when off)
  double* pmul;
  double* pmulb;
  ScenFold fold, foldb;         // the folded models of each pair's scenarios
  double punc_rho;
  uint32_t punc_mask;
  // host: the tensor maps of the two binary32 scenario arrays (the second
  // repeats the first until a second pair exists), or nullptr: the binary32
  // rings then use per-lane asynchronous copies
  const CUtensorMap* tmap;
  int tma;                      // RRG_TMA_*: which ring launches take the TMA
  int inject;                   // RRG_INJECT_* test switches (0 in normal use)
  int tma_pair_bps;             // resident blocks per SM of the paired TMA kernel (0: never paired)
  EqModel eq;
  // Only the largest admissible candidate counts (grid and k-section searches
  // with RRG_EXIT_CANDIDATE, whose candidates ascend with their slot): rows run
  // from the largest kappa down, and a candidate that every trajectory has
  // passed stops those below it.  2: the kernels' shared-memory limits are
  // set (top_down_pad).
  int top_down;
  // Top-down launches in two parts (launch_rollout): 1, the part held to one
  // candidate's warps, 2, the part that runs what it left; 0: one launch.
  int held;
  // Scenarios may have exponents of their own, which the binary64 power table does
  // not hold (pow then).
  int own_exponents;
};

// Binary64 rollouts on stored scenarios take four lanes per trajectory (Coop64)
// while that leaves every scheduler at most two warps (2 x 42 binary64 instructions
// a step against 110); 500 steps, one lane against four: 1.83 -> 0.96 ms with one
// warp a scheduler, 1.83 -> 1.40 with two, and a third would cost 2.0.  Where a
// torque takes pow, which every warp repeats however few of its lanes need it, at
// most one: 50 steps, one lane against four 0.89 -> 0.78 ms with one warp a
// scheduler, 0.89 -> 1.46 with two.
inline bool coop64_fits(const Launch& L, int rows) {
  const long long lone = static_cast<long long>((L.N + 31) / 32) * rows;  // warps, one lane per trajectory
  return L.m64.pw != nullptr && lone <= (L.own_exponents ? 1LL : 2LL) * L.sms;
}

// Folds the FC3 parameter vector into the constants the kernels use
// (binary64, then rounded once to binary32).  Only products and quotients
// occur, so no multiply-add can be fused and host and device agree bit for
// bit.  Called once per handle on the host and, under parametric
// uncertainty, once per trajectory on the device.
__host__ __device__ inline void fold_constants(const double* P, Fc3K<double>* k64,
                                               Fc3K<float>* k32) {
  Fc3K<double> K{};
  K.inv_p_atm = 1.0 / P[P_P_ATM];
  K.a_w = P[P_A_W];
  K.a_p = P[P_A_P];
  K.k_sm = P[P_K_SM];
  K.k_ca = P[P_K_CA];
  K.e = (P[P_GAMMA] - 1.0) / P[P_GAMMA];
  K.C_cp = P[P_C_P] * P[P_T_ATM] / P[P_ETA_CP];
  K.C_m = P[P_ETA_CM] * P[P_K_T] / P[P_R_CM];
  K.k_v = P[P_K_V];
  K.K_p = P[P_K_P];
  K.RT_Vca = P[P_R_A] * P[P_T_ST] / P[P_V_CA];
  K.RT_Vsm = P[P_R_A] * P[P_T_ST] / P[P_V_SM];
  K.inv_J = 1.0 / P[P_J_CP];
  K.pws = nullptr;
  *k64 = K;
  Fc3K<float> F{};
  F.inv_p_atm = static_cast<float>(K.inv_p_atm);
  F.a_w = static_cast<float>(K.a_w);
  F.a_p = static_cast<float>(K.a_p);
  F.k_sm = static_cast<float>(K.k_sm);
  F.k_ca = static_cast<float>(K.k_ca);
  F.e = static_cast<float>(K.e);
  F.C_cp = static_cast<float>(K.C_cp);
  F.C_m = static_cast<float>(K.C_m);
  F.k_v = static_cast<float>(K.k_v);
  F.K_p = static_cast<float>(K.K_p);
  F.RT_Vca = static_cast<float>(K.RT_Vca);
  F.RT_Vsm = static_cast<float>(K.RT_Vsm);
  F.inv_J = static_cast<float>(K.inv_J);
  F.pws = nullptr;
  *k32 = F;
}

// Constants of the closed loop at setpoint I (binary64; every operation
// rounded separately, so each call site computes the same bits).
__device__ __forceinline__ CandK<double> cand_consts(const double* __restrict__ P, double I) {
  CandK<double> C;
  C.W_o2 = __ddiv_rn(__dmul_rn(__dmul_rn(P[P_M_O2], P[P_N_CELL]), I), __dmul_rn(4.0, P[P_FARADAY]));
  const double W_ref = __ddiv_rn(__dmul_rn(P[P_LAM_REF], C.W_o2), P[P_X_O2]);
  const double v_ff = __dadd_rn(__dadd_rn(P[P_C0], __dmul_rn(P[P_C1], I)),
                                __dmul_rn(__dmul_rn(P[P_C2], I), I));
  C.V0 = __dadd_rn(v_ff, __dmul_rn(P[P_K_P], W_ref));
  C.y_scale = __ddiv_rn(__dmul_rn(P[P_X_O2], P[P_K_SM]), C.W_o2);
  return C;
}

__device__ __forceinline__ CandK<float> cand_round(const CandK<double>& C) {
  CandK<float> F;
  F.W_o2 = static_cast<float>(C.W_o2);
  F.V0 = static_cast<float>(C.V0);
  F.y_scale = static_cast<float>(C.y_scale);
  return F;
}

// Binary64 product and sum rounded on their own on host and device alike
// (the device compiler would otherwise fuse a product into a following add).
__host__ __device__ inline double mul_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ inline double add_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dadd_rn(a, b);
#else
  return a + b;
#endif
}

// L v (components ca, w, sm) of the linear part, each product and sum
// rounded on its own.
struct Vec3 { double a, w, s; };
__host__ __device__ inline Vec3 lin(const ModelC& m, const Vec3& v) {
  Vec3 r;
  r.a = add_rn(mul_rn(m.l_cs, v.s), -mul_rn(m.l_ca, v.a));
  r.w = add_rn(mul_rn(m.l_ws, v.s), -mul_rn(m.l_ww, v.w));
  r.s = add_rn(add_rn(mul_rn(m.l_sw, v.w), mul_rn(m.l_sa, v.a)), -mul_rn(m.l_ss, v.s));
  return r;
}
// u + c v
__host__ __device__ inline Vec3 axpy(double c, const Vec3& v, const Vec3& u) {
  return Vec3{add_rn(u.a, mul_rn(c, v.a)), add_rn(u.w, mul_rn(c, v.w)), add_rn(u.s, mul_rn(c, v.s))};
}
__host__ __device__ inline Vec3 scale(double c, const Vec3& v) {
  return Vec3{mul_rn(c, v.a), mul_rn(c, v.w), mul_rn(c, v.s)};
}

// Folds the model's constants for the rollout step of size h (rk4_step_fast),
// the same bits on the host and the device.
__host__ __device__ inline void fold_model(const Fc3K<double>& K, const double* P, double h,
                                           StepModel<double>* out) {
  ModelC m;
  m.l_cs = mul_rn(K.RT_Vca, K.k_sm);
  m.l_ca = add_rn(m.l_cs, mul_rn(K.RT_Vca, K.k_ca));
  const double e1 = mul_rn(mul_rn(K.C_m, K.K_p), K.inv_J);
  const double cj = mul_rn(K.C_m, K.inv_J);
  m.l_ww = add_rn(mul_rn(cj, K.k_v), mul_rn(e1, K.a_w));
  m.l_ws = mul_rn(e1, K.a_p);
  m.l_sa = mul_rn(K.RT_Vsm, K.k_sm);
  m.l_sw = mul_rn(K.RT_Vsm, K.a_w);
  m.l_ss = add_rn(mul_rn(K.RT_Vsm, K.a_p), m.l_sa);
  const double kw = mul_rn(P[P_M_O2], P[P_N_CELL]) / mul_rn(4.0, P[P_FARADAY]);  // W_o2 = kw v
  m.b_ca = mul_rn(K.RT_Vca, kw);
  m.d0 = mul_rn(cj, P[P_C0]);
  m.d1 = mul_rn(cj, add_rn(P[P_C1], mul_rn(K.K_p, mul_rn(P[P_LAM_REF], kw) / P[P_X_O2])));
  m.d2 = mul_rn(cj, P[P_C2]);
  m.ky = mul_rn(P[P_X_O2], P[P_K_SM]) / kw;
  m.p_atm = P[P_P_ATM];
  m.inv_p_atm = K.inv_p_atm;
  out->c = m;

  StepU<double>& U = out->U;
  StepPhi<double>& F = out->F;
  const double h2 = mul_rn(0.5, h), h6 = h / 6.0, ip = K.inv_p_atm;
  const double e3 = mul_rn(K.C_cp, K.inv_J);
  U.ip = ip;
  U.e = K.e;
  U.A = mul_rn(e3, K.a_w);
  U.B = mul_rn(mul_rn(e3, K.a_p), P[P_P_ATM]);
  F.h = h;
  F.h2 = h2;
  // the columns of M_2, M_3, M_4, R and of the combination that carries c
  Vec3 M2[3], M3[3], M4[3], R[3], Ph[3];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int j = 0; j < 3; ++j) {
    const Vec3 u{j == 0 ? 1.0 : 0.0, j == 1 ? 1.0 : 0.0, j == 2 ? 1.0 : 0.0};
    const Vec3 l1 = lin(m, u);
    M2[j] = axpy(h2, l1, u);
    const Vec3 l2 = lin(m, M2[j]);
    M3[j] = axpy(h2, l2, u);
    const Vec3 l3 = lin(m, M3[j]);
    M4[j] = axpy(h, l3, u);
    const Vec3 l4 = lin(m, M4[j]);
    R[j] = axpy(h6, axpy(2.0, l2, axpy(2.0, l3, axpy(1.0, l1, l4))), u);
    Ph[j] = scale(h6, axpy(2.0, M2[j], axpy(2.0, M3[j], axpy(1.0, u, M4[j]))));
  }
  U.x2a = mul_rn(ip, M2[0].s); U.x2w = mul_rn(ip, M2[1].s); U.x2s = mul_rn(ip, M2[2].s);
  U.w2w = M2[1].w; U.w2s = M2[2].w;
  U.x3a = mul_rn(ip, M3[0].s); U.x3w = mul_rn(ip, M3[1].s); U.x3s = mul_rn(ip, M3[2].s);
  U.w3a = M3[0].w; U.w3w = M3[1].w; U.w3s = M3[2].w;
  U.x4a = mul_rn(ip, M4[0].s); U.x4w = mul_rn(ip, M4[1].s); U.x4s = mul_rn(ip, M4[2].s);
  U.w4a = M4[0].w; U.w4w = M4[1].w; U.w4s = M4[2].w;
  U.faa = R[0].a; U.faw = R[1].a; U.fas = R[2].a;
  U.fsa = R[0].s; U.fsw = R[1].s; U.fss = R[2].s;
  U.fwa = R[0].w; U.fww = R[1].w; U.fws = R[2].w;
  F.aa = Ph[0].a; F.aw = Ph[1].a; F.as = Ph[2].a;
  F.sa = Ph[0].s; F.sw = Ph[1].s; F.ss = Ph[2].s;
  F.wa = Ph[0].w; F.ww = Ph[1].w; F.ws = Ph[2].w;
  // the torque's columns: k_i = L z_i + c - N_i e_w
  const Vec3 ew{0.0, 1.0, 0.0};
  const Vec3 le = lin(m, ew);
  // N_1: z_2 = -h2 e_w, z_3 = h2 L z_2, z_4 = h L z_3
  const Vec3 p2 = scale(-h2, ew), lp2 = scale(-h2, le);
  const Vec3 p3 = scale(h2, lp2), lp3 = lin(m, p3);
  const Vec3 p4 = scale(h, lp3), lp4 = lin(m, p4);
  const Vec3 f1 = scale(h6, axpy(2.0, lp2, axpy(2.0, lp3, axpy(-1.0, ew, lp4))));
  // N_2: z_3 = -h2 e_w, z_4 = h L z_3
  const Vec3 q4 = scale(h, lp2), lq4 = lin(m, q4);
  const Vec3 f2 = scale(h6, axpy(2.0, lp2, axpy(-2.0, ew, lq4)));
  // N_3: z_4 = -h e_w
  const Vec3 f3 = scale(h6, axpy(-2.0, ew, scale(-h, le)));
  U.w2n1 = p2.w;
  U.x3n1 = mul_rn(ip, p3.s);
  U.w3n1 = p3.w;
  U.w3n2 = p2.w;
  U.x4n1 = mul_rn(ip, p4.s);
  U.w4n1 = p4.w;
  U.x4n2 = mul_rn(ip, q4.s);
  U.w4n2 = q4.w;
  U.w4n3 = -h;
  U.fan1 = f1.a; U.fsn1 = f1.s; U.fwn1 = f1.w;
  U.fan2 = f2.a; U.fsn2 = f2.s; U.fwn2 = f2.w;
  U.fsn3 = f3.s; U.fwn3 = f3.w;
  U.fwn4 = -h6;
  out->pw = K.pws;
}

// The coefficients rounded once to binary32 (StepU and StepPhi hold nothing
// but T values), fss less 1 (add_sm).
__host__ __device__ inline void round_model(const StepModel<double>& m, StepModel<float>* out) {
  static_assert(sizeof(StepU<double>) == 2 * sizeof(StepU<float>) &&
                sizeof(StepPhi<double>) == 2 * sizeof(StepPhi<float>), "arrays of T");
  out->c = m.c;
  out->pw = nullptr;
  const double* u = &m.U.ip;
  float* uf = &out->U.ip;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (size_t i = 0; i < sizeof(StepU<float>) / sizeof(float); ++i) uf[i] = static_cast<float>(u[i]);
  out->U.fss = static_cast<float>(add_rn(m.U.fss, -1.0));
  const double* p = &m.F.h;
  float* pf = &out->F.h;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (size_t i = 0; i < sizeof(StepPhi<float>) / sizeof(float); ++i) pf[i] = static_cast<float>(p[i]);
}

// The steady-state threshold is y_min + eps_ss (y_c - y_min); a binary32
// solution (error about 1e-6) decides it unless it lies within 1e-4 of it.
inline void fold_eq(const double* P, double y_min, double eps_ss, double y_c, EqModel* E) {
  E->w1 = P[P_M_O2] * P[P_N_CELL] / (4.0 * P[P_FARADAY]);
  const double guess = P[P_LAM_REF] / P[P_X_O2];
  E->v0 = P[P_C0];
  E->v1 = P[P_C1] + P[P_K_P] * (guess * E->w1);
  E->v2 = P[P_C2];
  E->guess = static_cast<float>(guess);
  const double d = y_c - y_min, p = eps_ss * d;
  E->thr_ss = y_min + p;
  const double band = 1e-4 * (1.0 + std::fabs(E->thr_ss));
  const double hi = E->thr_ss + band, lo = E->thr_ss - band;
  E->y_pass = static_cast<float>(hi);
  if (static_cast<double>(E->y_pass) > hi) E->y_pass = std::nextafterf(E->y_pass, -INFINITY);
  E->y_fail = static_cast<float>(lo);
  if (static_cast<double>(E->y_fail) < lo) E->y_fail = std::nextafterf(E->y_fail, INFINITY);
}

// Candidate constants of the rollouts at setpoint v about the reference point
// q_r (gauge coordinates; binary32 values, or 0 for the gauge form), with the
// output bound y_min folded into the slack offset: the derivative at q_r
// without the torque, c = L q_r + b(v).  Every operation is spelled out in
// binary64, so each call site computes the same bits; 18 of them.
__device__ __forceinline__ RhsC<double> fold_cand(const ModelC& m, double v, const double q_r[3],
                                                  double y_min) {
  const double a = q_r[0], w = q_r[1], s = q_r[2];
  RhsC<double> R;
  R.c_ca = fma_rn(-m.b_ca, v, fma_rn(m.l_cs, s, __dmul_rn(-m.l_ca, a)));
  R.c_w = __dadd_rn(fma_rn(m.l_ws, s, __dmul_rn(-m.l_ww, w)), fma_rn(v, fma_rn(m.d2, v, m.d1), m.d0));
  R.c_sm = fma_rn(-m.l_ss, s, fma_rn(m.l_sw, w, __dmul_rn(m.l_sa, a)));
  R.x_r = fma_rn(s, m.inv_p_atm, 1.0);
  // 1 / v without the division's instructions, inside its range
  const unsigned ev = (static_cast<unsigned>(__double2hiint(v)) & 0x7fffffffu) >> 20;
  R.y_scale = (ev > 24u && ev < 2022u) ? __dmul_rn(m.ky, rcp_cubic(v)) : __ddiv_rn(m.ky, v);
  R.s_off = fma_rn(R.y_scale, __dsub_rn(s, a), -y_min);
  R.r_ca = a;
  R.r_w = w;
  R.r_sm = s;
  return R;
}
__device__ __forceinline__ RhsC<float> round_cand(const RhsC<double>& R) {
  return RhsC<float>{static_cast<float>(R.c_ca), static_cast<float>(R.c_w), static_cast<float>(R.c_sm),
                     static_cast<float>(R.x_r), static_cast<float>(R.y_scale), static_cast<float>(R.s_off),
                     static_cast<float>(R.r_ca), static_cast<float>(R.r_w), static_cast<float>(R.r_sm)};
}

// Table of the binary64 x^e - 1 (host; rrg_capi.cu); false, and an unusable
// table, for an exponent outside [-1, 1].
bool pow_table(double e, PowTable* S);

// ---- kernel launchers (rrg_kernels.cu) --------------------------------
// dual: write the pair (base + *t_dev) & 1 (closed loops with two pairs).
// In the binary32 modes only the binary32 copy is written.
cudaError_t launch_sample(const Launch& L, uint64_t seed, uint64_t base,
                          const unsigned long long* t_dev, const double* amp, bool dual = false,
                          cudaStream_t stream = nullptr);
// The folded models of a pair's scenarios (parametric uncertainty; nothing
// otherwise) from its multipliers: pair 0, or pair 1 (second), or by the parity
// of base + *t_dev (dual).  launch_sample runs it after its draw.
cudaError_t launch_scenario_fold(const Launch& L, bool second, uint64_t base = 0,
                                 const unsigned long long* t_dev = nullptr, bool dual = false,
                                 cudaStream_t stream = nullptr);
// Fills pair 0's binary64 array from its Philox counters if it was sampled
// lazily (no-op otherwise).
cudaError_t launch_materialize64(const Launch& L);
cudaError_t launch_round_scenarios(const Launch& L);
// Marks pair 0's binary64 array as holding its values.
cudaError_t launch_mark64(const Launch& L);
cudaError_t launch_fill(const Launch& L, double* a, size_t n, double v);
// buf_base >= 0: the update index is buf_base + *t_dev and selects the
// scenario pair by its parity; otherwise pair 0
cudaError_t launch_search_begin(const Launch& L, const double* d_x, const double* d_r,
                                const unsigned long long* t_dev, const double* d_v_prev,
                                long long buf_base = -1);
cudaError_t launch_search_next(const Launch& L, double* d_v_t, double* d_kappa,
                               int32_t* d_flags);
cudaError_t launch_search_mid(const Launch& L);
// Candidate set-up for the slots the last search kernel chose: one block per
// candidate (the binary64 equilibrium solves spread over the SMs).
cudaError_t launch_prepare(const Launch& L, int width);
// d_vp / d_r (optional): read v_prev and r on the device instead (a captured
// graph replayed with new inputs).
cudaError_t launch_eval_prepare(const Launch& L, const double* d_x, double v_prev, double r,
                                const double* d_kappas, int m, const double* d_vp = nullptr,
                                const double* d_r = nullptr);
cudaError_t launch_eval_finish(const Launch& L, int m, uint8_t* d_adm, double* d_min_slack);
// Tensor map of a binary32 scenario array in the quad layout for the TMA ring
// (boxes of 32 scenarios x one chunk of steps x 3 components); false when the
// driver refuses, and for more than kTmaMaxScenarios: a box starts at element
// four times its scenario, a signed 32-bit coordinate, which scenario 2^29 would
// overflow (the copy then raises an illegal instruction).  Half of that keeps
// every sum of a coordinate and a box away from the limit.
// tma_ring_prepare() sets the TMA kernels' shared-memory limit on the current
// device (once per device); false if the runtime refuses.
constexpr int kTmaMaxScenarios = 1 << 28;
bool encode_scenario_map(CUtensorMap* m, const float* d32, int N, int H);
bool tma_ring_prepare();
// Resident blocks per SM of the two-candidates-per-thread TMA kernel (after
// tma_ring_prepare on the current device; 0 if the runtime does not answer).
int tma_pair_blocks_per_sm(bool pu);
// Resident blocks per SM of the two-candidates-per-thread rollout kernel
// (queried from the runtime on the first call, then cached).
int pair_blocks_per_sm(bool pu);
// allow_pair: the round's rows are all full-horizon segments (no pipelined
// probe), so two candidates may share a thread (Launch::pair).
// kernels (may be null): receives how many kernels that took.
cudaError_t launch_rollout(const Launch& L, int m_launch, bool use_fp64, int early_exit,
                           bool recheck_classify, bool allow_pair = false, int* kernels = nullptr);
cudaError_t launch_recheck(const Launch& L, int early_exit);
cudaError_t launch_equilibrium(const Launch& L, double v, double* d_out4, int32_t* d_status);
cudaError_t launch_step_latency(const Launch& L, double v, int steps, double* d_out2, int32_t* d_status);
cudaError_t launch_plant(const Launch& L, const double* d_x, const double* d_v, uint64_t seed,
                         uint64_t base, const unsigned long long* t_dev, const double* amp_dev,
                         double* d_x_next);
cudaError_t launch_loop_end(const Launch& L, LoopState* ls, uint64_t seed, uint64_t t0,
                            const double* amp_dev, double* d_v_out, double* d_kappa_out,
                            int32_t* d_flags_out, double* d_x_out);
cudaError_t launch_loop_init(const Launch& L, LoopState* ls, const double* x0, double v0,
                             double* d_x_out);

// Discrete adjoint of the min-slack objective (rrg_adjoint.cu), for the m
// candidate slots the last candidate set-up prepared; layouts in the file.
constexpr int kAdjOutStride = 3 + 4 + RRG_NPARAM;
// argmin = false: the argmin pass is left to the reverse sweep (lane_min /
// lane_arg given to launch_adjoint_reverse), one launch fewer.
cudaError_t launch_adjoint_forward(const Launch& L, bool fp64, int m, int checkpoint, double* ckpt,
                                   double* lane_min, int* lane_arg, double* d_out,
                                   cudaEvent_t fwd_begin, cudaEvent_t fwd_end, bool argmin = true);
// The reverse sweeps read v_prev and r from the search state the candidate
// set-up wrote.  out_h, ss_h: pinned host copies of the slots' outputs and
// steady-state flags, written by the kernel (or null).
cudaError_t launch_adjoint_reverse(const Launch& L, bool fp64, int slot0, int count, int checkpoint,
                                   const double* ckpt, void* seg, double* d_out,
                                   const double* lane_min = nullptr, const int* lane_arg = nullptr, double* out_h = nullptr, int32_t* ss_h = nullptr);

// Binary32-vs-binary64 slack error of every trajectory of the m candidates
// the last eval_prepare + prepare set up (rrg_error.cu): per lane o = i N + k
// the largest |s32_j - s64_j| over j = 0..H and its step, both min slacks and
// the number of steps the band rule [-band, band) would decide wrongly and
// the largest ratio of a step's error to max(band, |s64_j|).  j_err, smin32,
// smin64, unsafe, ratio may be null.
cudaError_t launch_slack_error(const Launch& L, int m, float band, double* err, int32_t* j_err,
                               double* smin32, double* smin64, int32_t* unsafe, double* ratio);

// Configuration check shared with the handle-less entry point (rrg_capi.cu);
// on failure the message is readable with rrg_last_error(NULL).
int check_config(const rrg_config* c);
void set_thread_error(const char* msg);

// Number of search rounds each strategy enqueues (host-side schedule).
int search_round_count(const SearchCfg& c);
// Candidate count of round `round` of the schedule.
int search_round_width(const SearchCfg& c, int round);
// True when the first two rounds are pipelined (probe + continue).
bool search_pipelined(const SearchCfg& c, int horizon);
// Standard rounds enqueued after a pipelined pair (enough to finish the
// search from any level a wrong provisional outcome can send it back to),
// and the candidate width they need.
int search_extra_rounds(const SearchCfg& c);
int search_extra_width(const SearchCfg& c);

}  // namespace rrg
