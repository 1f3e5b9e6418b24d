// rrg_device.cuh -- device-side building blocks of the robust reference
// governor: the FC3 closed-loop right-hand side and output, the RK4 step,
// the Philox4x64-10 scenario generator and order-preserving keys for
// atomic minima.  Included by every translation unit with device code.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace rrg {

// a b + c rounded once; never simplified (x 0 + c is NaN for x = inf or NaN).
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// ---------------------------------------------------------------------------
// x^e - 1 in binary64 for x in [1, 2), from a table of kPowCells cells.
//
// A binary64 instruction takes a GB300 warp scheduler 64 cycles (measured: 2
// lanes per clock and SM, a lone warp's independent DFMAs no faster than its
// dependent ones), so what counts is their number.  With c the midpoint of
// x's cell and t = x / c - 1, |t| <= 2^-10,
//   x^e - 1 = (c^e - 1) + c^e sum_{n >= 1} binom(e, n) t^n,
// the terms from t^3 on are below 2^-34 c^e |binom(e, 3)|: formed in binary32
// (their rounding is below 2^-58) they cost no binary64 instruction, the term
// t^6 and later ones are below 2^-65.  Four binary64 instructions are left
// (t and three of Horner's rule) against 38 of one series over [1, 2].
// 1 / c is a binary32 value, so t is formed with one rounding.  Built on the
// host for one exponent (pow_table); a nullptr table (another exponent,
// or one outside [-1, 1]) and an x outside [1, 2) take pow.
constexpr int kPowCells = 512;
struct alignas(16) PowCell {
  double inv_c;       // 1 / c
  double a0, a1, a2;  // c^e - 1, c^e e, c^e binom(e, 2)
  float a3, a4, a5;   // c^e binom(e, n)
  float inv_cf;       // 1 / c
};
struct alignas(16) PowTable {
  PowCell cell[kPowCells];
  double e;           // the exponent the table is for (NaN: no table)
};

// A binary32 value widened without the binary64 pipe (0 becomes 2^-127, far
// below any rounding of its use).
__device__ __forceinline__ double widen_bits(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u);
  return __hiloint2double(static_cast<int>(hi), static_cast<int>(u << 29));
}

__device__ __forceinline__ double pow_m1_table(const PowTable* __restrict__ S, double x, double e) {
  const int hi = __double2hiint(x);
  if (S != nullptr && (hi >> 20) == 0x3ff) {
    const PowCell* __restrict__ c = S->cell + ((hi >> 11) & (kPowCells - 1));
    const double2 ia = __ldg(reinterpret_cast<const double2*>(c));
    const double2 a12 = __ldg(reinterpret_cast<const double2*>(c) + 1);
    const float4 f = __ldg(reinterpret_cast<const float4*>(c) + 2);
    const double t = fma_rn(x, ia.x, -1.0);
    // x truncated to binary32 is enough for the binary32 terms
    const uint32_t m = (static_cast<uint32_t>(hi) & 0xfffffu) << 3 |
                       static_cast<uint32_t>(__double2loint(x)) >> 29;
    const float tf = fma_rn(__uint_as_float(0x3f800000u | m), f.w, -1.0f);
    const double p3 = widen_bits(fma_rn(fma_rn(f.z, tf, f.y), tf, f.x));
    return fma_rn(t, fma_rn(t, fma_rn(t, p3, a12.y), a12.x), ia.y);
  }
  return pow(x, e) - 1.0;
}

// 1 / w in binary64: the hardware's approximate reciprocal (about 20 bits),
// refined by one cubic step of the Newton family, r + d (r + d r) with d =
// 1 - w r (error d^3): three binary64 instructions, within about one unit in
// the last place.
__device__ __forceinline__ double rcp_cubic(double w) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(w));
  const double d = fma_rn(-w, r, 1.0);
  return fma_rn(d, fma_rn(d, r, r), r);
}

// ---------------------------------------------------------------------------
// FC3 constants.  The state is kept in gauge coordinates
//   q = [p_ca - p_atm, w_cp, p_sm - p_atm]
// so that the pressure differences that set every flow (and the output) are
// formed from numbers of the size of the differences, not of ~1e5 Pa: in
// binary32 this keeps about 3 more significant bits in the slack.  All
// constants are folded once per handle in binary64 and rounded once.
template <typename T>
struct Fc3K {
  T inv_p_atm;   // 1 / p_atm
  T a_w, a_p;    // compressor map W_cp = a_w w - a_p q_sm
  T k_sm, k_ca;  // orifice and outlet coefficients
  T e;           // (gamma - 1) / gamma
  T C_cp;        // c_p T_atm / eta_cp
  T C_m;         // eta_cm k_t / R_cm
  T k_v;         // back-EMF constant
  T K_p;         // controller gain on the air-flow error
  T RT_Vca;      // R_a T_st / V_ca
  T RT_Vsm;      // R_a T_st / V_sm
  T inv_J;       // 1 / J_cp
  const PowTable* pws;   // binary64 x^e - 1 (device memory; nullptr: pow)
};

// Per-candidate constants (functions of the governed setpoint v = I only).
template <typename T>
struct CandK {
  T W_o2;     // O2 consumed, M_O2 n_cell I / (4 F)
  T V0;       // v_ff(I) + K_p W_ref(I): motor voltage at zero flow error
  T y_scale;  // x_O2 k_sm / W_o2: OER per pascal of p_sm - p_ca
};

// (1 + u)^e - 1, the compressor's isentropic temperature-ratio term: pow in
// binary64, the MUFU-based __powf in binary32.  (A degree-10 Chebyshev
// interpolant evaluated by Estrin's scheme was measured slower on GB300: a
// warp running one trajectory is issue-bound, and the polynomial costs more
// instructions than the two MUFU operations it would replace.)
template <typename T>
__device__ __forceinline__ T pow_e_m1(T e, T u, const PowTable* S);

template <>
__device__ __forceinline__ double pow_e_m1<double>(double e, double u, const PowTable* S) {
  return pow_m1_table(S, 1.0 + u, e);
}

template <>
__device__ __forceinline__ float pow_e_m1<float>(float e, float u, const PowTable*) {
  return __powf(1.0f + u, e) - 1.0f;
}

template <typename T> __device__ __forceinline__ T div_fast(T a, T b);
template <> __device__ __forceinline__ float div_fast<float>(float a, float b) { return __fdividef(a, b); }
template <> __device__ __forceinline__ double div_fast<double>(double a, double b) { return a / b; }

// dq/dt of the FC3 closed loop (mass balances of the cathode and supply
// manifold, torque balance of the compressor shaft under a feed-forward +
// proportional air-flow controller).
template <typename T>
__device__ __forceinline__ void fc3_rhs(const Fc3K<T>& K, const CandK<T>& C,
                                        T q_ca, T w, T q_sm,
                                        T& d_ca, T& d_w, T& d_sm) {
  const T W_cp = K.a_w * w - K.a_p * q_sm;
  const T W_sm = K.k_sm * (q_sm - q_ca);
  const T W_ca = K.k_ca * q_ca;
  const T pr_e = pow_e_m1<T>(K.e, q_sm * K.inv_p_atm, K.pws);
  const T tau_cp = div_fast<T>(K.C_cp * pr_e * W_cp, w);
  const T tau_cm = K.C_m * ((C.V0 - K.K_p * W_cp) - K.k_v * w);
  d_ca = K.RT_Vca * (W_sm - W_ca - C.W_o2);
  d_w = (tau_cm - tau_cp) * K.inv_J;
  d_sm = K.RT_Vsm * (W_cp - W_sm);
}

// Oxygen excess ratio y = h(x, v).
template <typename T>
__device__ __forceinline__ T fc3_output(const CandK<T>& C, T q_ca, T q_sm) {
  return C.y_scale * (q_sm - q_ca);
}

// ---------------------------------------------------------------------------
// The RK4 step of the rollouts, with the linear part of FC3 folded through the
// four stages (the equilibrium solve and the adjoint's reverse sweep keep the
// form above).
//
// In deviation coordinates z = q - q_r about a reference point q_r of the
// candidate (its binary32 equilibrium; 0 gives the gauge form) FC3 is linear
// but for one scalar in the speed's equation, the compressor's torque:
//   z' = L z + c - N(x, w) e_w,
//   N = (C_cp / J) W_cp (x^e - 1) / w = (x^e - 1) (A - B (x - 1) / w),
//   A = C_cp a_w / J, B = C_cp a_p p_atm / J
// (W_cp / w = a_w - a_p p_atm (x - 1) / w), x = p_sm / p_atm and w the speed.
// So every stage point and the step's result are fixed linear combinations of
// z, of c and of the stages' values N_1..N_4:
//   z_2 = M_2 z + (h/2) c - (h/2) N_1 e_w,   M_2 = I + (h/2) L
//   z_3 = M_3 z + ...,  M_3 = I + (h/2) L M_2;   M_4 = I + h L M_3
//   z+  = R z + ...,    R = I + (h/6) (L + 2 L M_2 + 2 L M_3 + L M_4)
// and a stage needs only its x and w, two rows of the combination.  The
// coefficients are products of the model's constants and the step size, formed
// in binary64 once per model and rounded once.
//
// Why: against right-hand sides evaluated stage by stage, a step on the TMA
// ring takes 90 binary32 instructions instead of 110 (4 torque terms of 7, 53
// multiply-adds, an addition, 3 loads, slack and bookkeeping), and its dependent chain
// shortens: x_{i+1} does not depend on N_i (the torque reaches the pressure one
// stage later), so the power's lg2 and ex2 of a stage overlap the stage
// before, and the chain through a stage is N_i -> w_{i+1} -> 1 / w -> N_{i+1}.
// Measured on GB300: one warp's chain 172 -> 145 cycles a step; launches that
// fill the SMs 2.3e11 -> 3.5e11 steps/s (nominal model, 114 cycles a step and
// scheduler: 90 issued, and lg2, rcp and ex2 hold their unit for 80).
// In binary64 49 multiply-adds and 4 torque terms of 12 instructions are left
// (pow_m1_table, rcp_cubic): 257 x 8 trajectories 10.8 -> 3.7 us a step.
//
// Near the reference every binary32 number is of the size of the deviation,
// not of the ~1e4 Pa gauge pressures, so the state's rounding shrinks with it;
// c and the reference are folded in binary64.
template <typename T>
struct StepU {  // one model's coefficients (per scenario under parametric uncertainty)
  T ip;         // 1 / p_atm
  T e, A, B;    // exponent and torque constants
  // stage 2..4: rows of x (already over p_atm) and w; nX: coefficient of N_X
  T x2a, x2w, x2s, w2w, w2s, w2n1;
  T x3a, x3w, x3s, x3n1, w3a, w3w, w3s, w3n1, w3n2;
  T x4a, x4w, x4s, x4n1, x4n2, w4a, w4w, w4s, w4n1, w4n2, w4n3;
  // the step's result: cathode pressure, manifold pressure (fss in binary32: less 1), speed
  T faa, faw, fas, fan1, fan2;
  T fsa, fsw, fss, fsn1, fsn2, fsn3;
  T fwa, fww, fws, fwn1, fwn2, fwn3, fwn4;
};

// What multiplies c in the combinations besides StepU's rows: the step sizes
// and the rows of (h/6) (I + 2 M_2 + 2 M_3 + M_4).
template <typename T>
struct StepPhi {
  T h, h2;
  T aa, aw, as, sa, sw, ss, wa, ww, ws;
};

template <typename T>
struct RhsC {            // constants of the candidate setpoint v (and the scenario's model)
  T c_ca, c_w, c_sm;     // the derivative at q_r without the torque: L q_r + b(v)
  T x_r;                 // 1 + sm_r / p_atm
  T y_scale;             // x_O2 k_sm / W_o2
  T s_off;               // slack at q_r: y_scale s_r - y_min
  T r_ca, r_w, r_sm;     // q_r (binary32 values, so both precisions share it)
};

// RhsC carried through the stages (formed once per trajectory): the constant
// of each row.
template <typename T>
struct StepC {
  T x1, x2, w2, x3, w3, x4, w4, fa, fw, fs;
  T y_scale, s_off, r_w;
};

template <typename T>
__device__ __forceinline__ StepC<T> step_consts(const StepU<T>& U, const StepPhi<T>& F, const RhsC<T>& C) {
  StepC<T> S;
  const T a = C.c_ca, w = C.c_w, s = C.c_sm;
  S.x1 = C.x_r;
  S.x2 = fma_rn(F.h2 * U.ip, s, C.x_r);
  S.w2 = fma_rn(F.h2, w, C.r_w);
  S.x3 = fma_rn(F.h2, fma_rn(U.x2a, a, fma_rn(U.x2w, w, U.x2s * s)), C.x_r);
  S.w3 = fma_rn(F.h2, fma_rn(U.w2w, w, U.w2s * s), C.r_w);
  S.x4 = fma_rn(F.h, fma_rn(U.x3a, a, fma_rn(U.x3w, w, U.x3s * s)), C.x_r);
  S.w4 = fma_rn(F.h, fma_rn(U.w3a, a, fma_rn(U.w3w, w, U.w3s * s)), C.r_w);
  S.fa = fma_rn(F.aa, a, fma_rn(F.aw, w, F.as * s));
  S.fs = fma_rn(F.sa, a, fma_rn(F.sw, w, F.ss * s));
  S.fw = fma_rn(F.wa, a, fma_rn(F.ww, w, F.ws * s));
  S.y_scale = C.y_scale;
  S.s_off = C.s_off;
  S.r_w = C.r_w;
  return S;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// N(x, w).  binary32: x^e by __powf, its - 1 fused with the product.
__device__ __forceinline__ float torque(const StepU<float>& U, const PowTable*, float x, float w) {
  const float p = __powf(x, U.e);
  const float t = fma_rn(-fma_rn(U.B, x, -U.B), rcp_approx(w), U.A);
  return fma_rn(p, t, -t);
}
__device__ __forceinline__ double torque(const StepU<double>& U, const PowTable* S, double x, double w) {
  const double t = fma_rn(-fma_rn(U.B, x, -U.B), rcp_cubic(w), U.A);
  return pow_m1_table(S, x, U.e) * t;
}

// The manifold pressure's result from its row's sum r: a binary64 row holds the
// pressure's own coefficient, a binary32 row that less 1, so its sum is the change
// over the step, and the pressure is added last.  Summed onto the pressure, each of
// the row's seven terms rounded at the pressure's magnitude, and the coefficient,
// close to 1, lost the digits of the change: the error against binary64 was 20-30 %
// above that of right-hand sides evaluated stage by stage.  One addition a step more
// gives, over updates of 1,024 scenarios x 2,000 steps (median trajectory, largest of
// 196,608): stage by stage 2.0e-7, 3.2e-6; summed onto the pressure 2.5e-7, 4.1e-6;
// here 1.9e-7, 2.5e-6; the cathode pressure's and the speed's rows so too 1.7e-7,
// 1.7e-6, for two more additions (16,384 x 16 x 1,000 steps: 730 us with none of
// them, 737 with this one, 746 with three).
__device__ __forceinline__ float add_sm(float s, float r) { return __fadd_rn(s, r); }
__device__ __forceinline__ double add_sm(double, double r) { return r; }

// One RK4 step followed by the disturbance (e_ca, e_w, e_sm) of Eq. 4, in
// place, on the deviation z = (q_ca, w, q_sm).  w_abs is the absolute speed
// r_w + w that the next step's first torque divides by: formed beside w from
// the same sum, so it never drifts from it by more than a rounding.  The
// newest N is always added last.  Every operation is spelled out, so each
// kernel that steps a trajectory gives the same bits.
// tq(x, w): the torque.
template <typename T, typename Torque>
__device__ __forceinline__ void rk4_step_with(const StepU<T>& U, const StepC<T>& C, T& q_ca, T& w, T& q_sm,
                                              T& w_abs, T e_ca, T e_w, T e_sm, const Torque& tq) {
  const T a = q_ca, z = w, s = q_sm;
  const T n1 = tq(fma_rn(U.ip, s, C.x1), w_abs);
  const T x2 = fma_rn(U.x2w, z, fma_rn(U.x2s, s, fma_rn(U.x2a, a, C.x2)));
  const T w2 = fma_rn(U.w2n1, n1, fma_rn(U.w2w, z, fma_rn(U.w2s, s, C.w2)));
  const T n2 = tq(x2, w2);
  const T x3 = fma_rn(U.x3n1, n1, fma_rn(U.x3w, z, fma_rn(U.x3s, s, fma_rn(U.x3a, a, C.x3))));
  const T w3 = fma_rn(U.w3n2, n2, fma_rn(U.w3n1, n1, fma_rn(U.w3w, z, fma_rn(U.w3s, s, fma_rn(U.w3a, a, C.w3)))));
  const T n3 = tq(x3, w3);
  const T x4 = fma_rn(U.x4n2, n2, fma_rn(U.x4n1, n1, fma_rn(U.x4w, z, fma_rn(U.x4s, s, fma_rn(U.x4a, a, C.x4)))));
  const T w4 = fma_rn(U.w4n3, n3, fma_rn(U.w4n2, n2, fma_rn(U.w4n1, n1,
               fma_rn(U.w4w, z, fma_rn(U.w4s, s, fma_rn(U.w4a, a, C.w4))))));
  const T n4 = tq(x4, w4);
  q_ca = fma_rn(U.fan2, n2, fma_rn(U.fan1, n1, fma_rn(U.faw, z, fma_rn(U.fas, s, fma_rn(U.faa, a, e_ca + C.fa)))));
  q_sm = add_sm(s, fma_rn(U.fsn3, n3, fma_rn(U.fsn2, n2, fma_rn(U.fsn1, n1,
         fma_rn(U.fsw, z, fma_rn(U.fss, s, fma_rn(U.fsa, a, e_sm + C.fs)))))));
  const T p = fma_rn(U.fwn3, n3, fma_rn(U.fwn2, n2, fma_rn(U.fwn1, n1,
              fma_rn(U.fww, z, fma_rn(U.fws, s, fma_rn(U.fwa, a, e_w + C.fw))))));
  w = fma_rn(U.fwn4, n4, p);
  w_abs = fma_rn(U.fwn4, n4, p + C.r_w);
}

// The same step with two binary32 multiply-adds per instruction (the same
// rounding as two fma_rn, on pairs in adjacent registers): the rows of x and
// w of a stage, and those of the two pressures, as pairs.  A packed
// multiply-add occupies its pipe for two cycles, so only issue slots are
// saved, and the coefficients must sit in registers.  Taken where they do
// anyway, in the parametric lanes on the TMA ring, which an issue-side
// conflict of three-register multiply-adds held back (16,384 x 16 x 1,000
// steps: 892 -> 850 us); the nominal lanes, whose coefficients are
// constant-bank operands, ran 14 % slower packed (741 -> 843 us), lone warps
// 6 %.
__device__ __forceinline__ uint64_t pk(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void upk(uint64_t p, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ void rk4_step_packed(const StepU<float>& U, const StepC<float>& C, float& q_ca,
                                                float& w, float& q_sm, float& w_abs, float e_ca, float e_w,
                                                float e_sm) {
  const auto tq = [&](float x, float speed) { return torque(U, nullptr, x, speed); };
  const float a = q_ca, z = w, s = q_sm;
  const uint64_t aa = pk(a, a), zz = pk(z, z), ss = pk(s, s);
  const float n1 = tq(fma_rn(U.ip, s, C.x1), w_abs);
  float x2, w2, x3, w3, x4, w4;
  upk(fma2(pk(U.x2w, U.w2w), zz, fma2(pk(U.x2s, U.w2s), ss, pk(fma_rn(U.x2a, a, C.x2), C.w2))), x2, w2);
  uint64_t p3 = fma2(pk(U.x3w, U.w3w), zz, fma2(pk(U.x3s, U.w3s), ss, fma2(pk(U.x3a, U.w3a), aa, pk(C.x3, C.w3))));
  uint64_t p4 = fma2(pk(U.x4w, U.w4w), zz, fma2(pk(U.x4s, U.w4s), ss, fma2(pk(U.x4a, U.w4a), aa, pk(C.x4, C.w4))));
  uint64_t pf = fma2(pk(U.faw, U.fsw), zz, fma2(pk(U.fas, U.fss), ss,
                fma2(pk(U.faa, U.fsa), aa, add2(pk(e_ca, e_sm), pk(C.fa, C.fs)))));
  float p = fma_rn(U.fww, z, fma_rn(U.fws, s, fma_rn(U.fwa, a, e_w + C.fw)));
  w2 = fma_rn(U.w2n1, n1, w2);
  const uint64_t nn1 = pk(n1, n1);
  p3 = fma2(pk(U.x3n1, U.w3n1), nn1, p3);
  p4 = fma2(pk(U.x4n1, U.w4n1), nn1, p4);
  pf = fma2(pk(U.fan1, U.fsn1), nn1, pf);
  p = fma_rn(U.fwn1, n1, p);
  const float n2 = tq(x2, w2);
  upk(p3, x3, w3);
  w3 = fma_rn(U.w3n2, n2, w3);
  const uint64_t nn2 = pk(n2, n2);
  p4 = fma2(pk(U.x4n2, U.w4n2), nn2, p4);
  pf = fma2(pk(U.fan2, U.fsn2), nn2, pf);
  p = fma_rn(U.fwn2, n2, p);
  const float n3 = tq(x3, w3);
  upk(p4, x4, w4);
  w4 = fma_rn(U.w4n3, n3, w4);
  upk(pf, q_ca, q_sm);
  q_sm = add_sm(s, fma_rn(U.fsn3, n3, q_sm));
  p = fma_rn(U.fwn3, n3, p);
  const float n4 = tq(x4, w4);
  w = fma_rn(U.fwn4, n4, p);
  w_abs = fma_rn(U.fwn4, n4, p + C.r_w);
}

template <typename T>
__device__ __forceinline__ void rk4_step_fast(const StepU<T>& U, const PowTable* pw, const StepC<T>& C,
                                              T& q_ca, T& w, T& q_sm, T& w_abs, T e_ca, T e_w, T e_sm) {
  rk4_step_with(U, C, q_ca, w, q_sm, w_abs, e_ca, e_w, e_sm,
                   [&](T x, T speed) { return torque(U, pw, x, speed); });
}

// ---------------------------------------------------------------------------
// Philox4x64-10, written from Salmon et al., "Parallel random numbers: as easy
// as 1, 2, 3" (SC'11): per round two 64x64 -> 128-bit products, words
// permuted and xored with the key; the key advances by a Weyl sequence.
struct U64x4 { uint64_t w[4]; };

__device__ __forceinline__ U64x4 philox4x64_10(uint64_t c0, uint64_t c1, uint64_t c2,
                                               uint64_t c3, uint64_t k0, uint64_t k1) {
  constexpr uint64_t kM0 = 0xD2E7470EE14C6C93ull, kM1 = 0xCA5A826395121157ull;
  constexpr uint64_t kW0 = 0x9E3779B97F4A7C15ull, kW1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) { k0 += kW0; k1 += kW1; }
    const uint64_t hi0 = __umul64hi(kM0, c0), lo0 = kM0 * c0;
    const uint64_t hi1 = __umul64hi(kM1, c2), lo1 = kM1 * c2;
    const uint64_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
  }
  U64x4 o;
  o.w[0] = c0; o.w[1] = c1; o.w[2] = c2; o.w[3] = c3;
  return o;
}

// 64 x 64 -> 128 bit product.
__device__ __forceinline__ void mul128(uint64_t m, uint64_t x, uint64_t& hi, uint64_t& lo) {
  const unsigned __int128 p = static_cast<unsigned __int128>(m) * x;
  hi = static_cast<uint64_t>(p >> 64);
  lo = static_cast<uint64_t>(p);
}

// Philox blocks at the counters (j, k0 + i kstep, upd, 0), key (seed, 0), for the
// KT scenarios i of a thread and one step j after the other: step(j, sink) calls
// sink(i, w0, w1, w2).  The scenario enters through word 1 and the step through
// word 0, so of the twenty products of a block one depends on the scenario
// alone (formed once per thread) and three on the step alone (shared by the
// thread's scenarios; callers keep j the same for every thread of a block, so
// they may run on the uniform path): 15 + 3 / KT are left per block.
//
// The generator is bound by the integer pipes: a 64-bit product is four wide
// multiply-adds at two cycles each and about as many additions, and the
// scheduler's multiply and logic pipes are each half busy.  Measured (16,384 x
// 5,000 binary32 draws): one block per (j, k) with its index division 892 us,
// this form 720 us with KT = 1, 700 with 2, 716 with 4.
template <int KT>
struct PhiloxCols {
  static constexpr uint64_t kM0 = 0xD2E7470EE14C6C93ull, kM1 = 0xCA5A826395121157ull;
  static constexpr uint64_t kW0 = 0x9E3779B97F4A7C15ull, kW1 = 0xBB67AE8584CAA73Bull;
  uint64_t seed, u_lo, b_hi[KT], b_lo[KT];

  __device__ __forceinline__ PhiloxCols(uint64_t k0, uint64_t kstep, uint64_t upd, uint64_t seed_) : seed(seed_) {
    uint64_t u_hi;  // round 0 of the update index
    mul128(kM1, upd, u_hi, u_lo);
#pragma unroll
    for (int i = 0; i < KT; ++i)  // rounds 0 and 1 of the scenario
      mul128(kM0, u_hi ^ (k0 + static_cast<uint64_t>(i) * kstep) ^ seed, b_hi[i], b_lo[i]);
  }

  template <typename Sink>
  __device__ __forceinline__ void step(int j, const Sink& sink) const {
    uint64_t a_hi, a_lo, c_hi, c_lo, e_hi, e_lo;  // rounds 0, 1 and 2 of the step
    mul128(kM0, static_cast<uint64_t>(j), a_hi, a_lo);
    mul128(kM1, a_hi, c_hi, c_lo);
    mul128(kM0, c_hi ^ u_lo ^ (seed + kW0), e_hi, e_lo);
#pragma unroll
    for (int i = 0; i < KT; ++i) {
      uint64_t ka = seed + 2 * kW0, kb = 2 * kW1, h, l;
      mul128(kM1, b_hi[i] ^ a_lo ^ kW1, h, l);  // round 2's other product
      uint64_t c0 = h ^ c_lo ^ ka, c1 = l, c2 = e_hi ^ b_lo[i] ^ kb, c3 = e_lo;
#pragma unroll
      for (int r = 3; r < 10; ++r) {
        ka += kW0;
        kb += kW1;
        uint64_t h0, l0, h1, l1;
        mul128(kM0, c0, h0, l0);
        mul128(kM1, c2, h1, l1);
        c0 = h1 ^ c1 ^ ka;
        c1 = l1;
        c2 = h0 ^ c3 ^ kb;
        c3 = l0;
      }
      sink(i, c0, c1, c2);
    }
  }
};

// ---------------------------------------------------------------------------
// The handles' binary32 scenario arrays hold four consecutive steps of a
// scenario side by side: [3 components][quads of steps][N scenarios][4 steps],
// H rounded up to whole quads.  A lane then reads four steps of a component
// with one 16-byte load (a warp: 512 consecutive bytes), from global memory or
// from a chunk that the TMA brought, where [3][H][N] took one load (and its
// share of the address arithmetic) per step and component; and every row is a
// multiple of 16 bytes whatever N.
__host__ __device__ inline size_t quad_rows(int H) { return (static_cast<size_t>(H) + 3) / 4; }
__host__ __device__ inline size_t quad_elems(int H, int N) { return 12 * quad_rows(H) * static_cast<size_t>(N); }
__host__ __device__ inline size_t quad_index(int c, int j, int k, int H, int N) {
  return ((c * quad_rows(H) + static_cast<size_t>(j >> 2)) * N + k) * 4 + (j & 3);
}

// a (2u - 1) with u the top 53 bits of w scaled to [0, 1).  2u - 1 equals
// t 2^-52 exactly for the integer t = (w >> 11) - 2^52, and a 2^-52 is exact,
// so (a 2^-52) t rounds the same real number once: one conversion and one
// binary64 multiply instead of four operations on GB300's narrow FP64 pipe.
// (For a below 2^-960, a 2^-52 would lose bits to underflow; such tiny
// half-ranges take the four-operation form.)
__device__ __forceinline__ double uniform_sym(uint64_t w, double a) {
  if (a < 0x1.0p-960) {
    const double u = __dmul_rn(static_cast<double>(w >> 11), 0x1.0p-53);
    return __dmul_rn(a, __dsub_rn(__dmul_rn(2.0, u), 1.0));
  }
  const long long t = static_cast<long long>(w >> 11) - (1ll << 52);
  return __dmul_rn(__ll2double_rn(t), __dmul_rn(a, 0x1.0p-52));
}

// a (2u - 1) in binary32 from the top 24 bits of w, with a_scaled = a 2^-23:
// RN32((w >> 40) - 2^23) a 2^-23).  Within a 2^-23 plus one binary32 rounding
// of the binary64 value above, and without binary64 arithmetic.
__device__ __forceinline__ float uniform_sym32(uint64_t w, float a_scaled) {
  const int t = static_cast<int>(w >> 40) - (1 << 23);
  return __fmul_rn(__int2float_rn(t), a_scaled);
}

// ---------------------------------------------------------------------------
// Order-preserving 64-bit key of a double (for atomicMin); NaN must be mapped
// by the caller.
__device__ __forceinline__ unsigned long long dkey(double x) {
  const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x));
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double dunkey(unsigned long long k) {
  return (k >> 63) ? __longlong_as_double(static_cast<long long>(k & 0x7FFFFFFFFFFFFFFFull))
                   : __longlong_as_double(static_cast<long long>(~k));
}

// Eq. 2 evaluated as written, without fused multiply-add.
__device__ __forceinline__ double governed(double v_prev, double r, double kappa) {
  return __dadd_rn(v_prev, __dmul_rn(kappa, __dsub_rn(r, v_prev)));
}

}  // namespace rrg
