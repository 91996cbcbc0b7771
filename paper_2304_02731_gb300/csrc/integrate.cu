// Trajectory integrator: Hamilton's equations (Sec. 2, Eqs. 3-4) in Jacobi
// coordinates, one trajectory per thread, Dormand-Prince 5(4) with a
// per-lane adaptive step (Sec. 3.2: SciPy's solve_ivp RK45 step control).
// Large all-Morse batches run here until their queue is empty; what is left,
// and every other batch, runs the same arithmetic with several lanes per
// trajectory (integrate_grp.cu; launch_stages below).
//
// GB300 design:
//  * The state (12 doubles) and the stage derivatives live in registers;
//    global memory is touched only to load a lane and to store it back.
//  * Runge-Kutta-Nystrom form.  Since d(rho)/dt = P/mu depends on P only,
//    every stage position of the classical method can be written with the
//    stage accelerations alone:
//        rho_s = rho + h c_s v + h^2 sum_q (A^2)_{sq} a_q ,   v = P/mu,
//    and the 5th-order update and the embedded error likewise use b^T A and
//    e^T A.  This is algebraically the same method as the 12-dimensional
//    Dormand-Prince step, with 6 (not 12) stored values per stage.
//  * The three pair distances of the last stage (FSAL, the new state) are
//    reused by the stop test, so the test costs no extra square roots.
//  * Step acceptance is a select, not a branch: all lanes of a warp run the
//    same instruction stream; only retirement diverges.
//  * Persistent mode: a finished lane takes the next trajectory index from a
//    device counter, with one atomicAdd per warp for all lanes that need
//    work (ballot + popc), so warps stay full until the queue drains.
//  * GB300 issues one warp-wide FP64 instruction per 64 to 76 cycles per SM
//    sub-partition (1/64 of the FP32 rate), so the kernel is bound by the
//    number of FP64-pipe instructions per step, and by their form: products
//    and sums are DFMAs on registers (regop.cuh), which took the 200,000-lane
//    sweep sample from 1.01 to 1.08 G attempts/s.  Everything that does not
//    need 53-bit arithmetic runs on the integer / FP32 pipes: the step-size
//    controller's error norm (magnitudes taken from the doubles' exponent and
//    leading mantissa bits, ratios in FP32), the stop tests (integer compares
//    of non-negative doubles) and the minimum-step test (exponent compare).
//  * Each pair force takes 1/sqrt(s) and e^x (elem64.cuh), 3 FP64
//    instructions each: the reciprocal square root is an FP32 hardware
//    estimate finished in FP64; the exponential is Tang's table method (a
//    2048-entry table of 2^(j/2048) in shared memory, the table index
//    rounded in FP32, the quadratic and cubic terms in float-float).
//  * Stages 6 and 7 (c = 1) share rho + h v, and the tableau entries that are
//    zero in exact arithmetic are skipped at compile time.
//  * Linear combinations that do not need an FP64 result run as float-float
//    compensated dot products on the FP32 / integer pipes (ff.cuh): the
//    acceleration corrections of stages 4-6 (one DADD each onto the FP64
//    base) and the embedded error estimate.  The new state (stage 7, v_n+1)
//    keeps its FP64 sums.
#include <cuda_runtime.h>
#include <cstdint>
#include <utility>

#include "qcams_device.cuh"
#include "qcams_internal.h"
#include "dp5_tableau.cuh"
#include "elem64.cuh"
#include "ff.cuh"
#include "step_ctrl.cuh"
#include "pair_force.cuh"

namespace qcams {
namespace {

// Coefficients in the constant bank, indexed at compile time.  A DFMA with a
// constant-bank operand takes 76 cycles instead of 64 (regop.cuh), so only the
// few products formed once per step read it directly; the weights b, which
// multiply every component, are staged in shared memory for register loads.
__constant__ RknTab kT = make_rkn_tab();

// The coefficients of the float-float sums as float pairs.
__constant__ RknTabFF kTff = make_rkn_tab_ff();

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------------------
// Accelerations a = (dP1/dt / mu12, dP2/dt / mu123) at Jacobi positions x,
// and the squared pair distances (AB, BC, CA).
//   r_AB = rho1,  r_BC = rho2 - cB rho1,  r_CA = rho2 + cA rho1
//   dV/drho1 = g_AB r_AB - cB g_BC r_BC + cA g_CA r_CA,
//   dV/drho2 = g_BC r_BC + g_CA r_CA,          g = V'(r)/r.
// ---------------------------------------------------------------------------
template <bool MORSE>
__device__ __forceinline__ void accel(const DevSys& S, const double* __restrict__ T,
                                      const double* x, double* a, double* s2, const OpReg& op) {
  const double rab0 = x[0], rab1 = x[1], rab2 = x[2];
  const double rbc0 = fma(-S.cB, x[0], x[3]), rbc1 = fma(-S.cB, x[1], x[4]),
               rbc2 = fma(-S.cB, x[2], x[5]);
  const double rca0 = fma(S.cA, x[0], x[3]), rca1 = fma(S.cA, x[1], x[4]),
               rca2 = fma(S.cA, x[2], x[5]);
  s2[0] = fma(rab0, rab0, fma(rab1, rab1, op.mul(rab2, rab2)));
  s2[1] = fma(rbc0, rbc0, fma(rbc1, rbc1, op.mul(rbc2, rbc2)));
  s2[2] = fma(rca0, rca0, fma(rca1, rca1, op.mul(rca2, rca2)));
  const double u0 = pair_u<MORSE>(S.pair[0], s2[0], T, op);
  const double u1 = pair_u<MORSE>(S.pair[1], s2[1], T, op);
  const double u2 = pair_u<MORSE>(S.pair[2], s2[2], T, op);
  const double f0 = op.mul(MORSE ? S.kf_morse[0] : S.kf[0], u0);
  const double f1 = op.mul(MORSE ? S.kf_morse[1] : S.kf[1], u1);
  const double f2 = op.mul(MORSE ? S.kf_morse[2] : S.kf[2], u2);
  const double h1 = op.mul(MORSE ? S.kf_morse[3] : S.kf[3], u1);
  const double h2 = op.mul(MORSE ? S.kf_morse[4] : S.kf[4], u2);
  a[0] = fma(f0, rab0, fma(f1, rbc0, op.mul(f2, rca0)));
  a[1] = fma(f0, rab1, fma(f1, rbc1, op.mul(f2, rca1)));
  a[2] = fma(f0, rab2, fma(f1, rbc2, op.mul(f2, rca2)));
  a[3] = fma(h1, rbc0, op.mul(h2, rca0));
  a[4] = fma(h1, rbc1, op.mul(h2, rca1));
  a[5] = fma(h1, rbc2, op.mul(h2, rca2));
}

// Position of stage s (1-based, s >= 2) from base = rho + h c_s v.
// The stage's coefficients h^2 (A^2)_{sq} are formed once per stage rather
// than scaling each component's sum by h^2 (6 multiplies); entries that are
// zero in exact arithmetic are skipped (stage 2 has no acceleration term).
template <int s>
__device__ __forceinline__ void stage_x(const double* base, const double (*acc)[6], double hh,
                                        double* x, const OpReg& op) {
  double w[s > 2 ? s - 2 : 1];
#pragma unroll
  for (int q = 1; q <= s - 2; ++q) w[q - 1] = dpA2Zero(s, q) ? 0.0 : op.mul(hh, kT.a2[s][q]);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double xi = base[i];
#pragma unroll
    for (int q = 1; q <= s - 2; ++q)
      if (!dpA2Zero(s, q)) xi = fma(w[q - 1], acc[q - 1][i], xi);
    x[i] = xi;
  }
}
// The same for stages 2 and 3 (c_s < 1), forming rho + h c_s v per component.
template <int s>
__device__ __forceinline__ void stage_x(const double* rho, const double* vel, const double (*acc)[6],
                                        double h, double hh, double* x, const OpReg& op) {
  static_assert(s == 2 || s == 3, "stages 4-6 use stage_x_ff, 7 the FP64 form");
  const double hc = op.mul(h, dpC(s));
  double base[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) base[i] = fma(hc, vel[i], rho[i]);
  stage_x<s>(base, acc, hh, x, op);
}

// Position of stage s = 4, 5, 6: base + h^2 sum_q (A^2)_{sq} a_q, the sum
// as a float-float compensated dot product (FP32 / integer pipes) added to
// the FP64 base with one DADD.  Its error, ~1e-13 h^2 |a|, reaches the step's
// result through the stage force only, damped by (h omega)^3 below the FP64
// rounding of the result; the 5th-order position (stage 7) and velocity
// keep FP64 sums.
template <int s>
__device__ __forceinline__ void stage_x_ff(const double* base, const double (*acc)[6], float hhh,
                                           float hhl, double* x, const OpReg& op) {
  static_assert(s >= 4 && s <= 6, "stages 4-6");
  float wh[s - 2], wl[s - 2];
#pragma unroll
  for (int q = 1; q <= s - 2; ++q) {
    const FFc c = kTff.a2[s][q];
    wh[q - 1] = __fmul_rn(hhh, c.hi);
    wl[q - 1] = fmaf(hhh, c.hi, -wh[q - 1]) + fmaf(hhh, c.lo, hhl * c.hi);
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    float sm, cm, ah, al;
    split_ff(acc[0][i], ah, al);
    ff_dot_first(sm, cm, wh[0], wl[0], ah, al);
#pragma unroll
    for (int q = 2; q <= s - 2; ++q) {
      split_ff(acc[q - 1][i], ah, al);
      ff_dot_acc(sm, cm, wh[q - 1], wl[q - 1], ah, al);
    }
    x[i] = op.add(base[i], ff_to_double(sm, cm));
  }
}

// One Dormand-Prince step of size h from (rho, vel) with acc[0] = a(rho).
// On return acc[1..6] hold the stage accelerations, xn / vn the 5th-order
// solution (acc[6] = a(xn), FSAL), er / ev the embedded error estimates of
// positions and velocities divided by h^2 and h (the error norm applies
// those factors in FP32), s2 the squared pair distances at xn.
//
// The error estimates are sums of ~1e-9 |a| from terms of ~0.05 |a|; the
// FP32 norm needs them to about 20 bits, so they are float-float
// compensated dot products (relative error ~1e-6 where the norm is near 1,
// the level of the norm's own 20-bit magnitudes) rather than FP64 sums.
template <bool MORSE>
__device__ __forceinline__ void dp_step(const DevSys& S, const double* __restrict__ T,
                                        const double* rho, const double* vel, double (*acc)[6],
                                        double h, double* xn, double* vn, float* er, float* ev,
                                        double* s2, const OpReg& op, const double* sB) {
  const double hh = op.mul(h, h);
  float hhh, hhl;
  split_ff(hh, hhh, hhl);
  double x[6];
  stage_x<2>(rho, vel, acc, h, hh, x, op);
  accel<MORSE>(S, T, x, acc[1], s2, op);
  stage_x<3>(rho, vel, acc, h, hh, x, op);
  accel<MORSE>(S, T, x, acc[2], s2, op);
  double base[6];
  const double hc4 = op.mul(h, dpC(4)), hc5 = op.mul(h, dpC(5));
#pragma unroll
  for (int i = 0; i < 6; ++i) base[i] = fma(hc4, vel[i], rho[i]);
  stage_x_ff<4>(base, acc, hhh, hhl, x, op);
  accel<MORSE>(S, T, x, acc[3], s2, op);
#pragma unroll
  for (int i = 0; i < 6; ++i) base[i] = fma(hc5, vel[i], rho[i]);
  stage_x_ff<5>(base, acc, hhh, hhl, x, op);
  accel<MORSE>(S, T, x, acc[4], s2, op);
#pragma unroll
  for (int i = 0; i < 6; ++i) base[i] = fma(h, vel[i], rho[i]);   // c_6 = c_7 = 1
  stage_x_ff<6>(base, acc, hhh, hhl, x, op);
  accel<MORSE>(S, T, x, acc[5], s2, op);
  stage_x<7>(base, acc, hh, xn, op);
  accel<MORSE>(S, T, xn, acc[6], s2, op);
  // the weights b_q as register operands
  double bq[7];
#pragma unroll
  for (int q = 1; q <= 6; ++q) bq[q] = static_cast<const volatile double*>(sB)[q];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double vb = op.mul(bq[1], acc[0][i]);
#pragma unroll
    for (int q = 3; q <= 6; ++q) vb = fma(bq[q], acc[q - 1][i], vb);
    vn[i] = fma(h, vb, vel[i]);
    // (e^T A)_2 = e_2 = 0 and (e^T A)_7 = 0: a_2 never enters, a_7 only ev
    float es, ec, rs, rc, ah, al;
    split_ff(acc[0][i], ah, al);
    ff_dot_first(es, ec, kTff.e[1].hi, kTff.e[1].lo, ah, al);
    ff_dot_first(rs, rc, kTff.ea[1].hi, kTff.ea[1].lo, ah, al);
#pragma unroll
    for (int q = 3; q <= 7; ++q) {
      split_ff(acc[q - 1][i], ah, al);
      ff_dot_acc(es, ec, kTff.e[q].hi, kTff.e[q].lo, ah, al);
      if (!dpEAZero(q)) ff_dot_acc(rs, rc, kTff.ea[q].hi, kTff.ea[q].lo, ah, al);
    }
    ev[i] = es + ec;
    er[i] = rs + rc;
  }
}

// Lane registers.
struct LaneState {
  double rho[6], vel[6];
  double acc[7][6];
  double t, h, tmax;
  int nacc, nrej, calls;   // calls = accepted + rejected in this launch
  int status;
  int sid;
  float atv[2];            // atol / mu of the two velocity blocks (FP32)
  bool rejected;           // the current step attempt follows a rejection
};

// Starting step (Hairer, Norsett & Wanner, Solving ODEs I, Sec. II.4), as
// used by SciPy's solve_ivp; error-estimator order 4, exponent 1/5.  Run once
// per trajectory, in FP64.
template <bool MORSE>
__device__ double initial_step(const DevSys& S, const double* __restrict__ T, const LaneState& L,
                               double rtol, double atol, const OpReg& op) {
  double atv[2] = {atol * S.inv_mu12, atol * S.inv_mu123};
  double d0 = 0.0, d1 = 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double scr = atol + fabs(L.rho[i]) * rtol;
    double scv = atv[i / 3] + fabs(L.vel[i]) * rtol;
    double q0 = L.rho[i] / scr, q1 = L.vel[i] / scv;
    d0 += q0 * q0 + q1 * q1;
    double p0 = L.vel[i] / scr, p1 = L.acc[0][i] / scv;
    d1 += p0 * p0 + p1 * p1;
  }
  d0 = sqrt(d0 / 12.0);
  d1 = sqrt(d1 / 12.0);
  double h0 = (d0 < 1e-5 || d1 < 1e-5) ? 1e-6 : 0.01 * d0 / d1;
  double x1[6], a1[6], s2[3];
#pragma unroll
  for (int i = 0; i < 6; ++i) x1[i] = fma(h0, L.vel[i], L.rho[i]);
  accel<MORSE>(S, T, x1, a1, s2, op);
  double d2 = 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double scr = atol + fabs(L.rho[i]) * rtol;
    double scv = atv[i / 3] + fabs(L.vel[i]) * rtol;
    double p0 = h0 * L.acc[0][i] / scr, p1 = (a1[i] - L.acc[0][i]) / scv;
    d2 += p0 * p0 + p1 * p1;
  }
  d2 = sqrt(d2 / 12.0) / h0;
  double h1 = (d1 <= 1e-15 && d2 <= 1e-15) ? fmax(1e-6, h0 * 1e-3)
                                           : pow(0.01 / fmax(d1, d2), 0.2);
  return fmin(100.0 * h0, h1);
}

__device__ __forceinline__ bool runnable(int st) {
  return st == QCAMS_LANE_READY || st == QCAMS_LANE_RUNNING;
}

// Load lane i; returns false if it is not runnable.  Computes acc[0] and,
// if no step size is stored yet, the starting step.
template <bool MORSE>
__device__ bool lane_load(const SysSet& sys, const IntegParams& ip, const double* __restrict__ T,
                          const DevBatch& B, int64_t i, LaneState& L,
                          unsigned long long& rhs_count, const OpReg& op) {
  L.status = B.status[i];
  if (!runnable(L.status)) return false;
  L.sid = B.sys_id[i];
  if (L.sid < 0 || L.sid >= sys.n) {
    B.status[i] = QCAMS_LANE_INVALID;
    return false;
  }
  const DevSys& S = sys.s[L.sid];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    L.rho[k] = B.y[k][i];
    L.rho[3 + k] = B.y[3 + k][i];
    L.vel[k] = B.y[6 + k][i] * S.inv_mu12;
    L.vel[3 + k] = B.y[9 + k][i] * S.inv_mu123;
  }
  L.t = B.t[i];
  L.h = B.h[i];
  L.tmax = ip.t_stop * B.t_scale[i];
  L.nacc = B.nsteps[i];
  L.nrej = B.nrej[i];
  L.calls = 0;
  L.rejected = false;
  L.status = QCAMS_LANE_RUNNING;
  L.atv[0] = (float)(ip.atol * S.inv_mu12);
  L.atv[1] = (float)(ip.atol * S.inv_mu123);
  double s2[3];
  accel<MORSE>(S, T, L.rho, L.acc[0], s2, op);
  rhs_count += 1;
  if (!(L.h > 0.0)) {
    L.h = initial_step<MORSE>(S, T, L, ip.rtol, ip.atol, op);
    rhs_count += 1;
  }
  return true;
}

template <bool MORSE>
__device__ void lane_store(const SysSet& sys, const DevBatch& B, int64_t i, const LaneState& L,
                           bool handoff = false) {
  const DevSys& S = sys.s[L.sid];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    B.y[k][i] = L.rho[k];
    B.y[3 + k][i] = L.rho[3 + k];
    B.y[6 + k][i] = handoff ? L.vel[k] : L.vel[k] * S.mu12;
    B.y[9 + k][i] = handoff ? L.vel[3 + k] : L.vel[3 + k] * S.mu123;
  }
  B.t[i] = L.t;
  B.h[i] = L.h;
  B.status[i] = static_cast<uint8_t>(
      handoff ? kHandoff | (L.rejected ? kHandoffRejected : 0) : L.status);
  B.nsteps[i] = L.nacc;
  B.nrej[i] = L.nrej;
}

// One adaptive step attempt with SciPy's RK45 rules: RMS error norm with
// scale atol + rtol max(|y_n|, |y_n+1|); accept iff norm < 1; new step
// h * clamp(0.9 norm^(-1/5), 0.2, 10), with no growth on the attempt that
// follows a rejection.  After an accepted step the stop rules are applied
// (Sec. 3.1: r_stop while separating, or t >= t_max).
//
// Only the step itself (stages, 5th-order update) is FP64; the error vector
// comes as FP32 from float-float sums.  The norm is formed in FP32 from
// 20-bit magnitudes of the state and scale terms (relative error < 1e-6,
// irrelevant to a step-size controller); accept / reject is a select, so
// the warp does not diverge.  The minimum step is checked by exponents: h
// fails below 8-16 ulp(t).
__device__ __forceinline__ void lane_attempt(const SysSet& sys, const IntegParams& ip,
                                             const double* __restrict__ T, LaneState& L,
                                             const OpReg& op, const double* sB) {
  const DevSys& S = sys.s[L.sid];
  {
    const int eh = (__double2hiint(L.h) >> 20) & 0x7ff;
    const int et = (__double2hiint(L.t) >> 20) & 0x7ff;
    if (et - eh >= 49 || eh == 0) {
      L.status = QCAMS_LANE_FAIL_HMIN;
      return;
    }
  }
  double xn[6], vn[6], s2[3];
  float er[6], ev[6];
  dp_step<true>(S, T, L.rho, L.vel, L.acc, L.h, xn, vn, er, ev, s2, op, sB);
  unsigned bad = 0, ignore = 0;
  float sum = 0.f;
  const float rt = ip.rtol_f, at = ip.atol_f;
  const float atv0 = L.atv[0], atv1 = L.atv[1];
  const float hf = mag_f(L.h, ignore), hhf = hf * hf;   // h > 0
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const float scr = fmaf(rt, fmaxf(mag_f(L.rho[i], ignore), mag_f(xn[i], ignore)), at);
    const float qr = err_mag(er[i], bad) * hhf * rcp_approx(scr);
    sum = fmaf(qr, qr, sum);
    const float scv = fmaf(rt, fmaxf(mag_f(L.vel[i], ignore), mag_f(vn[i], ignore)),
                           i < 3 ? atv0 : atv1);
    const float qv = err_mag(ev[i], bad) * hf * rcp_approx(scv);
    sum = fmaf(qv, qv, sum);
  }
  const float en2 = sum * (1.0f / 12.0f);
  L.calls += 1;
  if (bad) {
    L.status = QCAMS_LANE_FAIL_NAN;
    return;
  }
  // en^(-1/5) = en2^(-1/10)
  const float fac = 0.9f * pow_m01(en2);
  const bool accept = en2 < 1.0f;
  float fa = (en2 == 0.0f) ? 10.0f : fminf(10.0f, fac);
  fa = L.rejected ? fminf(1.0f, fa) : fa;
  const float f = accept ? fa : fmaxf(0.2f, fac);
  const double tn = L.t + L.h;
  L.t = accept ? tn : L.t;
  L.h = L.h * static_cast<double>(f);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    L.rho[i] = accept ? xn[i] : L.rho[i];
    L.vel[i] = accept ? vn[i] : L.vel[i];
    L.acc[0][i] = accept ? L.acc[6][i] : L.acc[0][i];
  }
  L.nacc += accept ? 1 : 0;
  L.nrej += accept ? 0 : 1;
  L.rejected = !accept;
  // stop rules on the accepted state (integer / FP32 compares)
  const long long smax = max(dbits(s2[0]), max(dbits(s2[1]), dbits(s2[2])));
  const float radial = fmaf(signed_f(L.rho[3]), signed_f(L.vel[3]),
                            fmaf(signed_f(L.rho[4]), signed_f(L.vel[4]),
                                 signed_f(L.rho[5]) * signed_f(L.vel[5])));
  int st = L.status;
  st = (accept && dbits(L.t) >= dbits(L.tmax)) ? QCAMS_LANE_DONE_TMAX : st;
  st = (accept && smax > dbits(ip.r_stop2) && radial > 0.0f) ? QCAMS_LANE_DONE_RSTOP : st;
  st = (st == QCAMS_LANE_RUNNING && (long long)(L.nacc + L.nrej) >= ip.max_steps)
           ? QCAMS_LANE_FAIL_MAXSTEPS : st;
  L.status = st;
}

__device__ __forceinline__ void flush_counters(unsigned long long rhs, unsigned long long steps,
                                               unsigned long long* counters) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rhs += __shfl_xor_sync(FULL, rhs, o);
    steps += __shfl_xor_sync(FULL, steps, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&counters[0], rhs);
    atomicAdd(&counters[1], steps);
  }
}

// Persistent refill-queue launch: each warp pops trajectory indices for all
// of its idle lanes with one atomicAdd (ballot + popc + shuffle).  With
// q.keep > 0 the lanes that are left when the queue is empty are handed on
// (StageQueue).
template <int BLOCK, int MINB>
__global__ void __launch_bounds__(BLOCK, MINB)
    k_integrate_persistent(SysSet sys, IntegParams ip, DevBatch B, unsigned long long* counters,
                           StageQueue q) {
  __shared__ double sT[kExpTableSize], sK[kOpRegs], sB[8];
  op_reg_fill(sK);
  if (threadIdx.x < 8) sB[threadIdx.x] = kT.b[threadIdx.x];
  load_exp_table(sT);   // ends with a barrier
  OpReg op;
  op.load(sK);
  const unsigned lane = threadIdx.x & 31u;
  unsigned long long rhs = 0, steps = 0;
  LaneState L;
  int64_t idx = -1;
  bool have = false, exhausted = false;
  for (;;) {
    const bool need = !have && !exhausted;
    const unsigned want = __ballot_sync(FULL, need);
    if (want) {
      const int leader = __ffs(want) - 1;
      unsigned long long base = 0;
      if ((int)lane == leader) base = atomicAdd(q.head, (unsigned long long)__popc(want));
      base = __shfl_sync(FULL, base, leader);
      bool skip = false;   // took a lane that does not run
      if (need) {
        const int64_t k = (int64_t)(base + __popc(want & ((1u << lane) - 1u)));
        if (k >= B.n) {
          exhausted = true;
        } else {
          idx = q.list_in ? q.list_in[k] : k;
          have = lane_load<true>(sys, ip, sT, B, idx, L, rhs, op);
          skip = !have;
        }
      }
      const unsigned gone = __ballot_sync(FULL, skip);
      if (gone && lane == 0) atomicAdd(q.retired, (unsigned long long)__popc(gone));
    }
    if (__all_sync(FULL, exhausted && !have)) break;
    if (q.keep > 0 && stage_over(q, B.n, lane)) {
      const unsigned pass = __ballot_sync(FULL, have);
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd(q.n_out, (unsigned long long)__popc(pass));
      at = __shfl_sync(FULL, at, 0);
      if (have) {
        rhs += 6ull * L.calls;
        steps += L.calls;
        lane_store<true>(sys, B, idx, L, true);
        q.list_out[at + __popc(pass & ((1u << lane) - 1u))] = idx;
      }
      break;
    }
    if (have) lane_attempt(sys, ip, sT, L, op, sB);
    const bool done = have && L.status != QCAMS_LANE_RUNNING;
    const unsigned ended = __ballot_sync(FULL, done);
    if (ended) {
      if (done) {
        rhs += 6ull * L.calls;
        steps += L.calls;
        lane_store<true>(sys, B, idx, L);
        have = false;
      }
      if (lane == 0) atomicAdd(q.retired, (unsigned long long)__popc(ended));
    }
  }
  flush_counters(rhs, steps, counters);
}

// Starting step of every runnable lane that has none yet (h = 0), for the
// lane-group stages: two right-hand sides a lane, once per trajectory.
template <bool MORSE>
__global__ void __launch_bounds__(128) k_start_step(SysSet sys, IntegParams ip, DevBatch B,
                                                    unsigned long long* counters) {
  __shared__ double sT[kExpTableSize], sK[kOpRegs], sB[8];
  op_reg_fill(sK);
  if (threadIdx.x < 8) sB[threadIdx.x] = kT.b[threadIdx.x];
  load_exp_table(sT);   // ends with a barrier
  OpReg op;
  op.load(sK);
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  unsigned long long rhs = 0;
  if (i < B.n && runnable(B.status[i]) && !(B.h[i] > 0.0)) {
    LaneState L;
    unsigned long long all = 0;
    if (lane_load<MORSE>(sys, ip, sT, B, i, L, all, op)) {
      B.h[i] = L.h;
      rhs = 1;
    }
  }
  flush_counters(rhs, 0, counters);
}

// Queue order of a run: lanes by falling t_scale = R / v_rel, the flight time
// of an undeflected collision.  Slow collisions take the most steps and form
// the long-lived complexes; a long trajectory that is taken last runs alone
// at the end.  A counting sort over kOrderBuckets buckets (the leading float
// bits of t_scale, 16 to the octave): the order within a bucket is free, and
// results do not depend on the order at all.  Lanes that already come that way
// (a sweep of rising energies) keep their own order, since neighbours of equal
// length finish together: 221,184 of them took 0.35 % more when shuffled.
// It reads t_scale three times and writes and reads a list entry, 40 bytes a
// lane, of which 8 come from DRAM (1.6 M lanes: the list stays in L2): with it 200,000
// mixed lanes at scattered energies take 612 ms instead of 763 (FP64), and
// 1,000,000 labelling lanes 28.6 ms instead of 38.4 (FP32).
constexpr int kOrderBuckets = 4096, kOrderBlock = 1024, kOrderChunk = 4096;

__device__ __forceinline__ int order_bucket(const DevBatch& B, int64_t i) {
  return (int)((__float_as_uint((float)B.t_scale[i]) >> 19) & (kOrderBuckets - 1));
}

// Bucket counts; count[kOrderBuckets] becomes 1 if a lane has a slower one
// next to it or half a batch behind it, by more than four buckets (a quarter
// of an octave): the vibrational phase moves R, and so t_scale, by up to ten
// percent among the lanes of a cell.
__global__ void __launch_bounds__(kOrderBlock) k_order_count(DevBatch B, unsigned* count) {
  __shared__ unsigned h[kOrderBuckets];
  const int64_t half = B.n / 2;
  bool mixed = false;
  for (int k = threadIdx.x; k < kOrderBuckets; k += kOrderBlock) h[k] = 0u;
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)kOrderBlock + threadIdx.x; i < B.n;
       i += (int64_t)gridDim.x * kOrderBlock) {
    const int k = order_bucket(B, i);
    mixed |= i + 1 < B.n && k + 4 < order_bucket(B, i + 1);
    mixed |= i + half < B.n && k + 4 < order_bucket(B, i + half);
    atomicAdd(&h[k], 1u);
  }
  if (mixed) count[kOrderBuckets] = 1u;
  __syncthreads();
  for (int k = threadIdx.x; k < kOrderBuckets; k += kOrderBlock)
    if (h[k]) atomicAdd(&count[k], h[k]);
}

// Counts to first positions, highest bucket first; *total = n.
__global__ void __launch_bounds__(kOrderBlock) k_order_scan(unsigned* count, int64_t n,
                                                            unsigned long long* total) {
  __shared__ unsigned ws[32];
  constexpr int PER = kOrderBuckets / kOrderBlock;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  unsigned mine[PER], sum = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    mine[k] = count[kOrderBuckets - 1 - (PER * t + k)];
    sum += mine[k];
  }
  unsigned v = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(FULL, v, o);
    if (lane >= o) v += u;
  }
  if (lane == 31) ws[warp] = v;
  __syncthreads();
  unsigned before = v - sum;
  for (int w = 0; w < warp; ++w) before += ws[w];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    count[kOrderBuckets - 1 - (PER * t + k)] = before;
    before += mine[k];
  }
  if (t == 0) *total = (unsigned long long)n;
}

// Places one chunk of lanes: its bucket counts, one range of the list per
// bucket, then the lanes.
__global__ void __launch_bounds__(kOrderBlock) k_order_place(DevBatch B, unsigned* next,
                                                             long long* list) {
  __shared__ unsigned h[kOrderBuckets];
  const int64_t base = (int64_t)blockIdx.x * kOrderChunk;
  if (next[kOrderBuckets] == 0u) {   // in order as they come
    for (int64_t i = base + threadIdx.x; i < base + kOrderChunk && i < B.n; i += kOrderBlock)
      list[i] = i;
    return;
  }
  for (int k = threadIdx.x; k < kOrderBuckets; k += kOrderBlock) h[k] = 0u;
  __syncthreads();
  int bucket[kOrderChunk / kOrderBlock];
  unsigned at[kOrderChunk / kOrderBlock];
#pragma unroll
  for (int k = 0; k < kOrderChunk / kOrderBlock; ++k) {
    const int64_t i = base + k * kOrderBlock + threadIdx.x;
    bucket[k] = i < B.n ? order_bucket(B, i) : -1;
    if (bucket[k] >= 0) at[k] = atomicAdd(&h[bucket[k]], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < kOrderBuckets; k += kOrderBlock)
    if (h[k]) h[k] = atomicAdd(&next[k], h[k]);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kOrderChunk / kOrderBlock; ++k)
    if (bucket[k] >= 0) list[h[bucket[k]] + at[k]] = base + k * kOrderBlock + threadIdx.x;
}

// Fixed-step mode: exactly max_steps steps of size h_fixed, no control and
// no stop test (used to check the integrator against the reference steps).
template <bool MORSE>
__global__ void __launch_bounds__(128) k_integrate_fixed(SysSet sys, IntegParams ip, DevBatch B,
                                                         unsigned long long* counters) {
  __shared__ double sT[kExpTableSize], sK[kOpRegs], sB[8];
  op_reg_fill(sK);
  if (threadIdx.x < 8) sB[threadIdx.x] = kT.b[threadIdx.x];
  load_exp_table(sT);   // ends with a barrier
  OpReg op;
  op.load(sK);
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  unsigned long long rhs = 0, steps = 0;
  if (i < B.n) {
    int st = B.status[i];
    const int sid = B.sys_id[i];
    if (runnable(st) && (sid < 0 || sid >= sys.n)) B.status[i] = QCAMS_LANE_INVALID;
    if (runnable(st) && sid >= 0 && sid < sys.n) {
      LaneState L;
      L.sid = sid;
      const DevSys& S = sys.s[L.sid];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        L.rho[k] = B.y[k][i];
        L.rho[3 + k] = B.y[3 + k][i];
        L.vel[k] = B.y[6 + k][i] * S.inv_mu12;
        L.vel[3 + k] = B.y[9 + k][i] * S.inv_mu123;
      }
      double s2[3];
      accel<MORSE>(S, sT, L.rho, L.acc[0], s2, op);
      double t = B.t[i];
      const double h = ip.h_fixed;
      for (long long it = 0; it < ip.max_steps; ++it) {
        double xn[6], vn[6];
        float er[6], ev[6];
        dp_step<MORSE>(S, sT, L.rho, L.vel, L.acc, h, xn, vn, er, ev, s2, op, sB);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          L.rho[q] = xn[q];
          L.vel[q] = vn[q];
          L.acc[0][q] = L.acc[6][q];
        }
        t += h;
      }
      L.t = t;
      L.h = h;
      L.status = QCAMS_LANE_RUNNING;
      L.nacc = B.nsteps[i] + (int)ip.max_steps;
      L.nrej = B.nrej[i];
      lane_store<MORSE>(sys, B, i, L);
      rhs = 1 + 6ull * ip.max_steps;
      steps = ip.max_steps;
    }
  }
  flush_counters(rhs, steps, counters);
}

__global__ void k_exp_check(const double* x, double* mine, double* ref, long long n) {
  __shared__ double sT[kExpTableSize];
  load_exp_table(sT);
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  mine[i] = texp(x[i], sT);
  ref[i] = exp(x[i]);
}

// The integrator's pair-force elementary functions on n squared distances s
// of one Morse pair (alpha = c0, alpha re = c1): 1/sqrt(s), the exponent's
// argument x = c1 - c0 r and e^x, exactly as the force law forms them.
__global__ void k_force_math_check(const double* s, double c0, double c1, float c0f, float c1f,
                                   double* ri_out, double* x_out, double* e_out, long long n) {
  __shared__ double sT[kExpTableSize];
  load_exp_table(sT);
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float rf;
  const double si = s[i];
  const double ri = rsqrt_seeded(si, rf);
  const double x = fma(-c0, si * ri, c1);
  ri_out[i] = ri;
  x_out[i] = x;
  e_out[i] = texp_hint(x, fmaf(-c0f, rf, c1f), sT);
}

// The integrator's float-float dot product on n rows of m <= 8 terms:
// out[i] = sum_q w[q] a[i m + q] formed as in the stage corrections (both
// operands split into float pairs, Dot2 accumulation, rebuilt as a double)
// and out_f[i] = the same sum rounded to FP32 as the error estimate takes it.
__global__ void k_ff_dot_check(const double* a, const double* w, int m, double* out,
                               float* out_f, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float s = 0.0f, c = 0.0f;
  for (int q = 0; q < m; ++q) {
    float wh, wl, ah, al;
    split_ff(w[q], wh, wl);
    split_ff(a[i * m + q], ah, al);
    if (q == 0)
      ff_dot_first(s, c, wh, wl, ah, al);
    else
      ff_dot_acc(s, c, wh, wl, ah, al);
  }
  out[i] = ff_to_double(s, c);
  out_f[i] = s + c;
}

bool all_morse(const SysSet& s) {
  for (int k = 0; k < s.n; ++k)
    for (int p = 0; p < 3; ++p)
      if (s.s[k].pair[p].kind != QCAMS_MORSE) return false;
  return true;
}

// Launch-shape variants: threads per block and the resident blocks per SM
// each kernel is compiled for (__launch_bounds__ minimum, which caps the
// registers per thread).  At ~190 registers, 64-thread blocks fit 5 per SM
// (10 warps) where 128-thread blocks fit 2 (8 warps); the autotuner measures.
struct Variant {
  int block, minb;
};
constexpr Variant kVariants[] = {{128, 1}, {64, 1}, {128, 3}, {64, 6}, {64, 7}, {256, 1}};
constexpr int kNumVariants = sizeof(kVariants) / sizeof(kVariants[0]);

int find_variant(int block, int minb) {
  if (block <= 0) block = 128;
  if (minb <= 0) minb = 1;
  for (int v = 0; v < kNumVariants; ++v)
    if (kVariants[v].block == block && kVariants[v].minb == minb) return v;
  return -1;
}

template <int BLOCK, int MINB>
cudaError_t launch_shape(const SysSet& sys, const IntegParams& ip, const DevBatch& b, int sm_count,
                         unsigned long long* counters, const StageQueue& q, cudaStream_t st) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, k_integrate_persistent<BLOCK, MINB>, BLOCK, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  long long grid = (long long)per_sm * sm_count;
  const long long need = (b.n + BLOCK - 1) / BLOCK;
  if (grid > need) grid = need;
  if (grid < 1) grid = 1;
  k_integrate_persistent<BLOCK, MINB><<<(unsigned)grid, BLOCK, 0, st>>>(sys, ip, b, counters, q);
  return cudaGetLastError();
}

cudaError_t launch_variant(int v, const SysSet& sys, const IntegParams& ip, const DevBatch& b,
                           int sm_count, unsigned long long* counters, const StageQueue& q,
                           cudaStream_t st) {
  switch (v) {
    case 0: return launch_shape<128, 1>(sys, ip, b, sm_count, counters, q, st);
    case 1: return launch_shape<64, 1>(sys, ip, b, sm_count, counters, q, st);
    case 2: return launch_shape<128, 3>(sys, ip, b, sm_count, counters, q, st);
    case 3: return launch_shape<64, 6>(sys, ip, b, sm_count, counters, q, st);
    case 4: return launch_shape<64, 7>(sys, ip, b, sm_count, counters, q, st);
    case 5: return launch_shape<256, 1>(sys, ip, b, sm_count, counters, q, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_exp_check(const double* x, double* mine, double* ref, long long n,
                             cudaStream_t st) {
  k_exp_check<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, mine, ref, n);
  return cudaGetLastError();
}

cudaError_t launch_force_math_check(const double* s, double c0, double c1, double* ri,
                                    double* x, double* e, long long n, cudaStream_t st) {
  k_force_math_check<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(s, c0, c1, (float)c0,
                                                                  (float)c1, ri, x, e, n);
  return cudaGetLastError();
}

cudaError_t launch_ff_dot_check(const double* a, const double* w, int m, double* out,
                               float* out_f, long long n, cudaStream_t st) {
  k_ff_dot_check<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, w, m, out, out_f, n);
  return cudaGetLastError();
}

cudaError_t launch_integrate_shape(const SysSet& sys, const IntegParams& ip, const DevBatch& b,
                                   int block, int blocks_per_sm, Ctx& ctx, cudaStream_t st) {
  const int v = find_variant(block, blocks_per_sm);
  if (v < 0 || !all_morse(sys)) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(ctx.counters, 0, kCounters * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  StageQueue q;
  q.head = ctx.counters + 4;
  q.retired = ctx.counters + 5;
  return launch_variant(v, sys, ip, b, ctx.sm_count, ctx.counters, q, st);
}

cudaError_t launch_queue_order(const DevBatch& b, long long* list, unsigned* scratch,
                               unsigned long long* n_out, cudaStream_t st) {
  static_assert(8 * kOrderMinLanes >= 4 * (kOrderBuckets + 1), "counts fit in jprime");
  cudaError_t e = cudaMemsetAsync(scratch, 0, (kOrderBuckets + 1) * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  const int64_t chunks = (b.n + kOrderChunk - 1) / kOrderChunk;
  k_order_count<<<(unsigned)(chunks < 304 ? chunks : 304), kOrderBlock, 0, st>>>(b, scratch);
  k_order_scan<<<1, kOrderBlock, 0, st>>>(scratch, b.n, n_out);
  k_order_place<<<(unsigned)chunks, kOrderBlock, 0, st>>>(b, scratch, list);
  return cudaGetLastError();
}

// The lane lists live in vprime and jprime, which the product analysis writes
// for every lane after the run.  A caller may have pointed several outputs at
// one buffer, and the order's counts are 32 bits wide: then there are no
// lists, the first stage runs to the end, and lanes are taken as they come.
bool lists_usable(const DevBatch& b) {
  if (b.n >= (int64_t)1 << 32) return false;
  const uintptr_t v = (uintptr_t)b.vprime, j = (uintptr_t)b.jprime, len = 8 * (uintptr_t)b.n;
  if (!v || !j || (v & 7) || (j & 7)) return false;
  auto apart = [&](const void* p, size_t size) {
    const uintptr_t a = (uintptr_t)p, e = a + size * (uintptr_t)b.n;
    return !a || ((e <= v || a >= v + len) && (e <= j || a >= j + len));
  };
  for (int k = 0; k < 12; ++k)
    if (!apart(b.y[k], 8)) return false;
  return (v + len <= j || j + len <= v) && apart(b.t, 8) && apart(b.h, 8) &&
         apart(b.t_scale, 8) && apart(b.E0, 8) && apart(b.Ecol, 8) && apart(b.status, 1) &&
         apart(b.nsteps, 4) && apart(b.nrej, 4) && apart(b.sys_id, 4);
}

namespace {

// FP64 adaptive run of modes 0 and 1 in stages.  A stage runs until its
// source is used up and at most keep_per_sm trajectories per SM are
// unfinished, then hands those on (StageQueue): near its end a batch has few
// long trajectories scattered over its warps, each warp-wide FP64
// instruction costs a sub-partition 64 cycles however many lanes it serves,
// and packing the survivors into fewer warps, with more lanes each, shortens
// their steps.  Every stage forms the same bits, so the path a trajectory
// takes does not show in its results.  Where the lines lie (GB300, 152 SMs):
//  * The one-thread kernel only for all-Morse batches of at least 512
//    trajectories per SM (77,824), which fill it twice over: there it runs
//    1.08 G attempts/s against 1.06 of the three-lane queue (200,000 sweep
//    lanes); in the generic form the queue is ahead, 0.84 against 0.75, and
//    below that size the one-thread kernel has idle sub-partitions (0.54
//    against 0.97 at 12,096 lanes).  It hands on as soon as its source is
//    empty: its own capacity is 256 per SM.
//  * Three lanes per trajectory hold 120 trajectories per SM; at 80 and at 20
//    per SM (2 warps and half a warp per sub-partition) the survivors are
//    packed again, the last time with six lanes each (6.7 instead of 8.8 us a
//    step when each sub-partition has one warp).
// 12,288 sweep lanes take 460 ms this way, 572 ms with three lanes to the
// end, 660 ms without packing and 1,250 ms in the one-thread kernel alone;
// 200,000 mixed lanes 612 ms (763 without the queue order) against 1,440 ms.
struct Stage {
  int lanes;         // lanes per trajectory (1: the persistent kernel)
  int keep_per_sm;   // hands on at this many trajectories per SM (0: none)
};
constexpr Stage kStages[] = {{1, 256}, {3, 80}, {3, 20}, {6, 0}};
constexpr int kNumStages = sizeof(kStages) / sizeof(kStages[0]);
constexpr int kOneThreadMinPerSm = 512;
// Batches that the first stage cannot hold at once (three lanes: 120 per SM)
// are taken in the order of launch_queue_order.
constexpr int kOrderMinPerSm = 120;
static_assert(4 + 4 * kNumStages <= kCounters, "a counter block per stage");

// The stages that a batch of n lanes takes.
struct StagePlan {
  bool order = false;          // takes the queue order
  int n = 0;                   // stages, from first to last:
  int stage[kNumStages];       // index into kStages
  int64_t bound[kNumStages];   // the most trajectories it can meet
  int64_t keep[kNumStages];    // hands on at this many (0: runs to the end)
};
StagePlan plan_stages(bool morse, bool lists, int64_t n, int64_t sms) {
  StagePlan p;
  p.order = lists && n > kOrderMinPerSm * sms && n >= kOrderMinLanes;
  int64_t bound = n;
  for (int s = 0; s < kNumStages; ++s) {
    const int64_t keep = kStages[s].keep_per_sm * sms;
    if (kStages[s].lanes == 1 ? !(morse && lists && n >= kOneThreadMinPerSm * sms) : bound <= keep)
      continue;
    p.stage[p.n] = s;
    p.bound[p.n] = bound;
    p.keep[p.n] = lists ? keep : 0;
    if (p.keep[p.n++] == 0) break;
    bound = keep < bound ? keep : bound;
  }
  return p;
}

template <bool MORSE>
cudaError_t launch_stages(const SysSet& sys, const DevShape* shapes, const IntegParams& ip,
                          const DevBatch& b, int variant, Ctx& ctx, cudaStream_t st) {
  const StagePlan plan = plan_stages(MORSE, lists_usable(b), b.n, ctx.sm_count);
  StageQueue q;
  long long* list[2] = {reinterpret_cast<long long*>(b.vprime),
                        reinterpret_cast<long long*>(b.jprime)};
  if (plan.order) {   // slowest collisions first
    cudaError_t e = launch_queue_order(b, list[0], reinterpret_cast<unsigned*>(b.jprime),
                                       ctx.counters + 3, st);
    if (e != cudaSuccess) return e;
    q.list_in = list[0];
    q.n_in = ctx.counters + 3;
    std::swap(list[0], list[1]);
  }
  for (int k = 0; k < plan.n; ++k) {
    const int lanes = kStages[plan.stage[k]].lanes;
    unsigned long long* c = ctx.counters + 4 + 4 * plan.stage[k];
    q.head = c;
    q.retired = c + 1;
    q.n_out = c + 2;
    q.list_out = list[0];
    q.keep = plan.keep[k];
    cudaError_t e = cudaSuccess;
    if (lanes == 1) {
      e = launch_variant(variant, sys, ip, b, ctx.sm_count, ctx.counters, q, st);
    } else {
      if (k == 0) {
        k_start_step<MORSE>
            <<<(unsigned)((b.n + 127) / 128), 128, 0, st>>>(sys, ip, b, ctx.counters);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess)
        e = launch_integrate_queue(sys, shapes, ip, b, lanes, plan.bound[k], ctx.sm_count,
                                   ctx.counters, q, st, MORSE);
    }
    if (e != cudaSuccess) return e;
    q.list_in = q.list_out;
    q.n_in = q.n_out;
    q.handed_on = true;
    std::swap(list[0], list[1]);
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_integrate(const SysSet& sys, const DevShape* shapes, const IntegParams& ip,
                             const DevBatch& b, int precision, int persistent, int block,
                             int blocks_per_sm, Ctx& ctx, cudaStream_t st) {
  if (b.n == 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(ctx.counters, 0, kCounters * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  const bool morse = all_morse(sys);
  if (precision == 32) return launch_integrate32(sys, shapes, ip, b, persistent, ctx, st, morse);
  if (ip.fixed_step) {
    const unsigned grid = (unsigned)((b.n + 127) / 128);
    if (morse) k_integrate_fixed<true><<<grid, 128, 0, st>>>(sys, ip, b, ctx.counters);
    else k_integrate_fixed<false><<<grid, 128, 0, st>>>(sys, ip, b, ctx.counters);
    return cudaGetLastError();
  }
  if (persistent == 2 || persistent == 3)
    return launch_integrate_grouped(sys, shapes, ip, b, persistent == 2 ? 3 : 6, ctx.counters, st,
                                    morse);
  const int v = find_variant(block, blocks_per_sm);
  if (v < 0) return cudaErrorInvalidValue;
  return morse ? launch_stages<true>(sys, shapes, ip, b, v, ctx, st)
               : launch_stages<false>(sys, shapes, ip, b, v, ctx, st);
}

int integrate_plan(const SysSet& sys, const IntegParams& ip, int precision, int persistent,
                   int64_t n, int sm_count, int lanes[8], int* n_stages) {
  *n_stages = 1;
  lanes[0] = 1;
  if (n == 0) return *n_stages = 0;
  const bool morse = all_morse(sys);
  if (precision == 32) return integrate32_queue(morse, sys.n == 1, persistent, n, sm_count) ? 4 : 1;
  if (ip.fixed_step) return 1;
  if (persistent >= 2) {
    lanes[0] = persistent == 2 ? 3 : 6;
    return 1;
  }
  const StagePlan p = plan_stages(morse, true, n, sm_count);
  static_assert(kNumStages <= 8, "room in lanes");
  *n_stages = p.n;
  for (int k = 0; k < p.n; ++k) lanes[k] = kStages[p.stage[k]].lanes;
  return (p.order ? 3 : 0) + (lanes[0] == 1 ? 0 : 1) + p.n;
}

int integrate_variant_count() { return kNumVariants; }

void integrate_variant_shape(int v, int* block, int* minb) {
  *block = kVariants[v].block;
  *minb = kVariants[v].minb;
}

bool integrate_shape_supported(int block, int blocks_per_sm) {
  return find_variant(block, blocks_per_sm) >= 0;
}

cudaError_t integrate_variant_info(int v, int* regs, int* blocks_per_sm) {
  cudaFuncAttributes a;
  cudaError_t e = cudaErrorInvalidValue;
#define QCAMS_INFO(B, N)                                              \
  e = cudaFuncGetAttributes(&a, k_integrate_persistent<B, N>);        \
  if (e == cudaSuccess)                                               \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(                \
        blocks_per_sm, k_integrate_persistent<B, N>, B, 0)
  switch (v) {
    case 0: QCAMS_INFO(128, 1); break;
    case 1: QCAMS_INFO(64, 1); break;
    case 2: QCAMS_INFO(128, 3); break;
    case 3: QCAMS_INFO(64, 6); break;
    case 4: QCAMS_INFO(64, 7); break;
    case 5: QCAMS_INFO(256, 1); break;
    default: break;
  }
#undef QCAMS_INFO
  if (e == cudaSuccess) *regs = a.numRegs;
  return e;
}

bool integrate_all_morse(const SysSet& sys) { return all_morse(sys); }

}  // namespace qcams
