// FP64 trajectory integrator with three or six lanes per trajectory.
//
// The same method as integrate.cu (Hamilton's equations in Jacobi
// coordinates, Sec. 2 Eqs. 3-4; Dormand-Prince 5(4) in Runge-Kutta-Nystrom
// form with SciPy's RK45 step control, Sec. 3.2; the stop rules of
// Sec. 3.1).  GB300 issues a warp-wide FP64 instruction in 64 cycles per SM
// sub-partition however many of its lanes are active, so what a trajectory's
// step takes is its chain of warp-wide FP64 instructions, 516 in the
// one-thread-per-trajectory kernel.  Here a group of G lanes carries one
// trajectory: each lane holds 6 / G of the six position components (and
// the matching velocities and stage accelerations) and evaluates the force
// of pair c mod 3 (AB, BC, CA) of its lane index c.
//   G = 3: lane j holds component j of both Jacobi vectors; a step takes
//          177 warp-wide FP64 instructions (Morse), 10 trajectories a warp.
//   G = 6: lane c holds one component (c < 3: rho1, else rho2), the two
//          halves of the group evaluate the three pair forces twice; 140
//          instructions a step, 5 trajectories a warp.
// The group exchanges pair-vector components, the pair force factors, the
// step's scalar coefficients (each lane forms every G-th) and the error
// norm's terms by warp shuffles.
//
// Two kernels: k_integrate_grp (launch modes 2 and 3) keeps its trajectories
// from start to end and sums squared distances and norms in its own lane
// order; k_integrate_queue (SEQ; the stages of modes 0 and 1) sums them in
// the one-thread kernel's order, so that its results are that kernel's bit
// for bit, and refills its groups from a queue.  Saturated, three lanes cost
// 17.7 FP64 instructions per trajectory and step against 16.1, but finer
// grain and three times the warps make up for it (figures at launch_stages
// in integrate.cu).
//
// Every quantity the step control and the stop rules decide on (error norm,
// largest pair distance, radial velocity, collapse) is reduced in the same
// order in all lanes of a group, so they take identical decisions.
// The lanes left over at the end of a warp repeat the first lanes of its
// last group and store nothing; a lane whose trajectory is done or absent
// keeps executing the warp's instructions (FP64 costs the same either way)
// with its state frozen, so every shuffle runs on the full warp.
#include <cuda_runtime.h>

#include "qcams_device.cuh"
#include "qcams_internal.h"
#include "dp5_tableau.cuh"
#include "elem64.cuh"
#include "ff.cuh"
#include "step_ctrl.cuh"
#include "pair_force.cuh"

namespace qcams {
namespace {

__constant__ RknTab kT3 = make_rkn_tab();
__constant__ RknTabFF kTff3 = make_rkn_tab_ff();

// Tableau entries staged in shared memory by load_coefs: the step's nine
// scalar coefficients (lanes index them by their place in the group), then
// the weights b_1 .. b_6.
constexpr int kCoefs = 15;
__device__ __forceinline__ void load_coefs(double* c) {
  if (threadIdx.x < 4) c[threadIdx.x] = dpC(2 + threadIdx.x);
  if (threadIdx.x == 4) c[4] = kT3.a2[3][1];
  if (threadIdx.x == 5) c[5] = kT3.a2[7][1];
  if (threadIdx.x >= 6 && threadIdx.x < 9) c[threadIdx.x] = kT3.a2[7][threadIdx.x - 3];
  if (threadIdx.x >= 9 && threadIdx.x < 15) c[threadIdx.x] = kT3.b[threadIdx.x - 8];
}

constexpr unsigned FULL = 0xffffffffu;
constexpr int kGrpBlock = 32;   // one warp per block: small batches spread over the SMs
constexpr int kQueueBlock = 128;

// A lane's place in its group and the constants of its pair.
template <int G>
struct Grp {
  static constexpr int K = 6 / G;          // position components per lane
  static constexpr int PER_WARP = 32 / G;  // trajectories per warp
  int c;        // lane index in the group, 0 .. G-1
  int j;        // pair index c mod 3 (0 = AB, 1 = BC, 2 = CA)
  int base;     // lane of group index 0
  DevPair q;    // pair j of the trajectory's system
  double kf;    // dP1-force factor of pair j (f_j = kf u_j)
  double cA, cB;   // the system's Jacobi coefficients
  double kh;    // dP2-force factor of pair j (h_1, h_2; pair AB: unused); with
                // G = 6 the upper half holds it in kf
  const double* coef;   // the step's nine tableau entries, in shared memory
  // global position component (0-2: rho1, 3-5: rho2) of local component k
  __device__ __forceinline__ int comp(int k) const { return G == 3 ? (k == 0 ? j : 3 + j) : c; }
};

// Sum over the group of a per-lane value, in lane order (identical in all
// lanes of the group).
template <int G, typename V>
__device__ __forceinline__ V grp_sum(V v, int base) {
  V s = __shfl_sync(FULL, v, base);
#pragma unroll
  for (int k = 1; k < G; ++k) s += __shfl_sync(FULL, v, base + k);
  return s;
}
template <int G>
__device__ __forceinline__ unsigned grp_or(unsigned v, int base) {
  unsigned s = 0;
#pragma unroll
  for (int k = 0; k < G; ++k) s |= __shfl_sync(FULL, v, base + k);
  return s;
}
template <int G>
__device__ __forceinline__ long long grp_max(long long v, int base) {
  long long s = __shfl_sync(FULL, v, base);
#pragma unroll
  for (int k = 1; k < G; ++k) s = max(s, __shfl_sync(FULL, v, base + k));
  return s;
}

// The error norm's sum over the six components as the one-thread kernel
// forms it: position then velocity term of component 0, 1, .. 5.
template <int G>
__device__ __forceinline__ float grp_norm_seq(const float* qr, const float* qv, int base) {
  float sum = 0.0f;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const int src = base + (G == 3 ? i % 3 : i), k = G == 3 ? i / 3 : 0;
    const float a = __shfl_sync(FULL, qr[k], src), b = __shfl_sync(FULL, qv[k], src);
    sum = fmaf(b, b, fmaf(a, a, sum));
  }
  return sum;
}

// u = V'(r)/r of the lane's pair at squared distance s: pair_u's formulas.
// The lanes of a warp hold different pairs, so the
// generic form is one sequence for the Morse, Buckingham and (12,6) / (8,6)
// Lennard-Jones kinds with selected operands instead of a branch per kind.
template <bool MORSE, bool SEQ>
__device__ __forceinline__ double pair_u_grp(const DevPair& q, double s,
                                             const double* __restrict__ T,
                                             const OpReg& op) {
  float rf;
  const double ri = rsqrt_seeded(s, rf, op);
  if (MORSE) {
    const double as = op.mul(q.c0, s);
    const double x = texp_hint(fma(-as, ri, q.c1), fmaf(-q.ef0, rf, q.ef1), T, op);
    return op.mul(fma(-x, x, x), ri);
  }
  const bool isM = q.kind == QCAMS_MORSE, isB = q.kind == QCAMS_BUCK;
  const bool isL = !isM && !isB, general = isL && !(q.n == 6 && (q.m == 12 || q.m == 8));
  double x = 1.0;
  if (!isL) {
    const double as = op.mul(isB ? q.c1 : q.c0, s);
    x = texp_hint(fma(-as, ri, isB ? q.lc2 : q.c1), fmaf(-q.ef0, rf, q.ef1), T, op);
  }
  const double ri2 = op.mul(ri, ri), ri4 = op.mul(ri2, ri2);
  const double ri6 = op.mul(ri4, ri2);
  const double hb = isL && q.m == 12 ? ri6 : ri4, hh = op.mul(hb, hb);
  // Morse c2/r, Buckingham A B e^{-B r}/r, Lennard-Jones m Cm/r^m
  const double A = op.mul(isB ? x : q.c2, isL ? hh : ri);
  const double B = fma(isM ? -x : q.c3, isM ? x : (isL ? ri6 : hh), isM ? x : -A);
  const double C = op.mul(B, isM ? A : ri2);
  double u = isB ? B : C;
  if (general) u = SEQ ? lj_u(q, ri, op) : pot_g(q, ri, s * ri);
  return u;
}

// The lane's acceleration components (dP1/dt / mu12 or dP2/dt / mu123 for
// its position components x) and the squared distance of pair j.  The pair
// vectors are those of accel() in integrate.cu:
//   r_AB = rho1,  r_BC = rho2 - cB rho1,  r_CA = rho2 + cA rho1.
// Each lane forms component j of the three pair vectors (with G = 6, from
// its own component and its partner's across the two halves), gathers
// components j+1, j+2 of pair j's vector from the lanes holding them in its
// half (each sender choosing the pair its receiver needs), forms the
// squared distance with one multiply and two FMAs, evaluates
// u_j = V'(r_j)/r_j, and the group exchanges f_j = kf u_j and h_j = kh u_j.
template <bool MORSE, int G, bool SEQ>
__device__ __forceinline__ void accel_grp(const Grp<G>& L,
                                          const double* __restrict__ T, const double* x,
                                          double* a, double& s_own,
                                          const OpReg& op) {
  double x1, x2;
  if (G == 3) {
    x1 = x[0];
    x2 = x[1];
  } else {
    const double other = __shfl_sync(FULL, x[0], L.base + (L.c + 3) % 6);
    x1 = L.c < 3 ? x[0] : other;
    x2 = L.c < 3 ? other : x[0];
  }
  const double rab = x1, rbc = fma(-L.cB, x1, x2), rca = fma(L.cA, x1, x2);
  const int half = L.base + (L.c - L.j);   // lane of component 0 in this lane's half
  double rk[2];
#pragma unroll
  for (int r = 1; r <= 2; ++r) {
    // in round r a lane receives from the lane of component (j + r) mod 3,
    // which sends its component of pair (its j - r) mod 3: the receiver's pair
    const int want = (L.j + 3 - r) % 3;
    const double v = want == 0 ? rab : (want == 1 ? rbc : rca);
    rk[r - 1] = __shfl_sync(FULL, v, half + (L.j + r) % 3);
  }
  const double rj = L.j == 0 ? rab : (L.j == 1 ? rbc : rca);
  // SEQ: the squares summed in the one-thread kernel's component order
  const double c0 = !SEQ || L.j == 0 ? rj : (L.j == 1 ? rk[1] : rk[0]);
  const double c1 = !SEQ || L.j == 0 ? rk[0] : (L.j == 1 ? rj : rk[1]);
  const double c2 = !SEQ || L.j == 0 ? rk[1] : (L.j == 1 ? rk[0] : rj);
  const double s = fma(c0, c0, fma(c1, c1, op.mul(c2, c2)));
  s_own = s;
  const double u = pair_u_grp<MORSE, SEQ>(L.q, s, T, op);
  if (G == 3) {
    const double f = op.mul(L.kf, u), h = op.mul(L.kh, u);
    const double f0 = __shfl_sync(FULL, f, L.base), f1 = __shfl_sync(FULL, f, L.base + 1),
                 f2 = __shfl_sync(FULL, f, L.base + 2);
    const double h1 = __shfl_sync(FULL, h, L.base + 1), h2 = __shfl_sync(FULL, h, L.base + 2);
    a[0] = fma(f0, rab, fma(f1, rbc, op.mul(f2, rca)));
    a[1] = fma(h1, rbc, op.mul(h2, rca));
  } else {
    // the lower half forms the f_j, the upper one the h_j: each half needs its own
    const double f = op.mul(L.kf, u);
    const double f0 = __shfl_sync(FULL, f, half), f1 = __shfl_sync(FULL, f, half + 1),
                 f2 = __shfl_sync(FULL, f, half + 2);
    a[0] = fma(L.c < 3 ? f0 : 0.0, rab, fma(f1, rbc, op.mul(f2, rca)));
  }
}

// The step's scalar coefficients (as integrate.cu's stage_x forms them):
// h c_2 .. h c_5, then h^2 (A^2)_{31} and h^2 (A^2)_{7q}, q = 1, 3, 4, 5;
// (A^2)_{32} and (A^2)_{72} are zero.  They are the same for every lane of a
// trajectory, so lane j forms every G-th of them and the group exchanges
// the results.
constexpr int kSteps = 9;
static_assert(dpA2Zero(7, 2) && !dpA2Zero(7, 1) && !dpA2Zero(7, 3) && !dpA2Zero(7, 4) &&
              !dpA2Zero(7, 5) && !dpA2Zero(3, 1), "the nonzero entries of stages 3 and 7");
template <int G>
__device__ __forceinline__ void step_coeffs(const Grp<G>& L, double h, double hh, double* w,
                                            const OpReg& op) {
  double mine[(kSteps + G - 1) / G];
#pragma unroll
  for (int r = 0; r < (kSteps + G - 1) / G; ++r) {
    const int k = min(r * G + L.c, kSteps - 1);
    mine[r] = op.mul(k < 4 ? h : hh, L.coef[k]);
  }
#pragma unroll
  for (int k = 0; k < kSteps; ++k) w[k] = __shfl_sync(FULL, mine[k / G], L.base + k % G);
}

// Stages 4-6: the acceleration correction as a float-float dot product
// added to the FP64 base with one DADD.
template <int s, int K>
__device__ __forceinline__ void stage_xk_ff(const double* base, const double (*acc)[K], float hhh,
                                            float hhl, double* x, const OpReg& op) {
  float wh[s - 2], wl[s - 2];
#pragma unroll
  for (int q = 1; q <= s - 2; ++q) {
    const FFc c = kTff3.a2[s][q];
    wh[q - 1] = __fmul_rn(hhh, c.hi);
    wl[q - 1] = fmaf(hhh, c.hi, -wh[q - 1]) + fmaf(hhh, c.lo, hhl * c.hi);
  }
#pragma unroll
  for (int i = 0; i < K; ++i) {
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

// One Dormand-Prince step of size h for the lane's components, with
// acc[0] = a(rho).  On return acc[1..6] hold the stage accelerations, xn /
// vn the 5th-order solution, er / ev the embedded error estimates divided by
// h^2 and h, s_own the squared distance of pair j at xn (per component the
// arithmetic of integrate.cu's dp_step).
template <bool MORSE, int G, bool SEQ>
__device__ __forceinline__ void dp_step_grp(const Grp<G>& L,
                                            const double* __restrict__ T, const double* rho,
                                            const double* vel, double (*acc)[Grp<G>::K],
                                            double h, double* xn, double* vn, float* er,
                                            float* ev, double& s_own,
                                            const OpReg& op) {
  constexpr int K = Grp<G>::K;
  const double hh = op.mul(h, h);
  double w[kSteps];
  step_coeffs<G>(L, h, hh, w, op);
  float hhh, hhl;
  split_ff(hh, hhh, hhl);
  double x[K], base[K];
#pragma unroll
  for (int i = 0; i < K; ++i) base[i] = fma(w[0], vel[i], rho[i]);
  accel_grp<MORSE, G, SEQ>(L, T, base, acc[1], s_own, op);
#pragma unroll
  for (int i = 0; i < K; ++i) base[i] = fma(w[1], vel[i], rho[i]);
#pragma unroll
  for (int i = 0; i < K; ++i) x[i] = fma(w[4], acc[0][i], base[i]);
  accel_grp<MORSE, G, SEQ>(L, T, x, acc[2], s_own, op);
#pragma unroll
  for (int i = 0; i < K; ++i) base[i] = fma(w[2], vel[i], rho[i]);
  stage_xk_ff<4, K>(base, acc, hhh, hhl, x, op);
  accel_grp<MORSE, G, SEQ>(L, T, x, acc[3], s_own, op);
#pragma unroll
  for (int i = 0; i < K; ++i) base[i] = fma(w[3], vel[i], rho[i]);
  stage_xk_ff<5, K>(base, acc, hhh, hhl, x, op);
  accel_grp<MORSE, G, SEQ>(L, T, x, acc[4], s_own, op);
#pragma unroll
  for (int i = 0; i < K; ++i) base[i] = fma(h, vel[i], rho[i]);   // c_6 = c_7 = 1
  stage_xk_ff<6, K>(base, acc, hhh, hhl, x, op);
  accel_grp<MORSE, G, SEQ>(L, T, x, acc[5], s_own, op);
#pragma unroll
  for (int i = 0; i < K; ++i)
    xn[i] = fma(w[8], acc[4][i],
                fma(w[7], acc[3][i], fma(w[6], acc[2][i], fma(w[5], acc[0][i], base[i]))));
  accel_grp<MORSE, G, SEQ>(L, T, xn, acc[6], s_own, op);
  // the weights b_q as register operands
  double bq[7];
#pragma unroll
  for (int q = 1; q <= 6; ++q) bq[q] = static_cast<const volatile double*>(L.coef)[8 + q];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    double vb = op.mul(bq[1], acc[0][i]);
#pragma unroll
    for (int q = 3; q <= 6; ++q) vb = fma(bq[q], acc[q - 1][i], vb);
    vn[i] = fma(h, vb, vel[i]);
    // (e^T A)_2 = e_2 = 0 and (e^T A)_7 = 0: a_2 never enters, a_7 only ev
    float es, ec, rs, rc, ah, al;
    split_ff(acc[0][i], ah, al);
    ff_dot_first(es, ec, kTff3.e[1].hi, kTff3.e[1].lo, ah, al);
    ff_dot_first(rs, rc, kTff3.ea[1].hi, kTff3.ea[1].lo, ah, al);
#pragma unroll
    for (int q = 3; q <= 7; ++q) {
      split_ff(acc[q - 1][i], ah, al);
      ff_dot_acc(es, ec, kTff3.e[q].hi, kTff3.e[q].lo, ah, al);
      if (!dpEAZero(q)) ff_dot_acc(rs, rc, kTff3.ea[q].hi, kTff3.ea[q].lo, ah, al);
    }
    ev[i] = es + ec;
    er[i] = rs + rc;
  }
}

// A trajectory's state in one lane of its group: the lane's K position
// components, their velocities P / mu and stage accelerations; the scalars
// are the same in all lanes of the group.
template <int K>
struct GrpLane {
  double rho[K], vel[K];
  double acc[7][K];
  double t, h, tmax;
  float atv[K];            // atol / mu of each component (FP32)
  int nacc, nrej, calls, status;
  bool rejected;
};

__device__ __forceinline__ bool runnable(int st) {
  return st == QCAMS_LANE_READY || st == QCAMS_LANE_RUNNING;
}

// Starting step (Hairer, Norsett & Wanner, Solving ODEs I, Sec. II.4, as
// SciPy's solve_ivp takes it), the norms summed over the group.
template <bool MORSE, int G>
__device__ double initial_step_grp(const Grp<G>& L, const double* __restrict__ T,
                                   const GrpLane<Grp<G>::K>& X, const double* inv_mu, double rtol, double atol,
                                   const OpReg& op) {
  constexpr int K = Grp<G>::K;
  double d0 = 0.0, d1 = 0.0;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const double scr = atol + fabs(X.rho[i]) * rtol;
    const double scv = atol * inv_mu[i] + fabs(X.vel[i]) * rtol;
    const double q0 = X.rho[i] / scr, q1 = X.vel[i] / scv;
    d0 += q0 * q0 + q1 * q1;
    const double p0 = X.vel[i] / scr, p1 = X.acc[0][i] / scv;
    d1 += p0 * p0 + p1 * p1;
  }
  d0 = sqrt(grp_sum<G>(d0, L.base) / 12.0);
  d1 = sqrt(grp_sum<G>(d1, L.base) / 12.0);
  const double h0 = (d0 < 1e-5 || d1 < 1e-5) ? 1e-6 : 0.01 * d0 / d1;
  double x1[K], a1[K], s_dummy;
#pragma unroll
  for (int i = 0; i < K; ++i) x1[i] = fma(h0, X.vel[i], X.rho[i]);
  accel_grp<MORSE, G, false>(L, T, x1, a1, s_dummy, op);
  double d2 = 0.0;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const double scr = atol + fabs(X.rho[i]) * rtol;
    const double scv = atol * inv_mu[i] + fabs(X.vel[i]) * rtol;
    const double p0 = h0 * X.acc[0][i] / scr, p1 = (a1[i] - X.acc[0][i]) / scv;
    d2 += p0 * p0 + p1 * p1;
  }
  d2 = sqrt(grp_sum<G>(d2, L.base) / 12.0) / h0;
  const double h1 = (d1 <= 1e-15 && d2 <= 1e-15) ? fmax(1e-6, h0 * 1e-3)
                                                 : pow(0.01 / fmax(d1, d2), 0.2);
  return fmin(100.0 * h0, h1);
}

// One adaptive step attempt with SciPy's RK45 rules, as integrate.cu's
// lane_attempt: RMS error norm with scale atol + rtol max(|y_n|, |y_n+1|)
// (FP32, from 20-bit magnitudes), accept iff norm < 1, new step
// h clamp(0.9 norm^(-1/5), 0.2, 10) with no growth right after a rejection,
// then the stop rules on the accepted state (Sec. 3.1).  Lanes whose
// trajectory is not running execute it with their state frozen.
template <bool MORSE, int G, bool SEQ>
__device__ __forceinline__ void attempt_grp(const Grp<G>& L,
                                            const DevShape* shapes, int sid,
                                            const IntegParams& ip, const double* __restrict__ T,
                                            GrpLane<Grp<G>::K>& X, const OpReg& op) {
  constexpr int K = Grp<G>::K;
  bool go = X.status == QCAMS_LANE_RUNNING;
  {
    const int eh = (__double2hiint(X.h) >> 20) & 0x7ff;
    const int et = (__double2hiint(X.t) >> 20) & 0x7ff;
    const bool fail_h = go && (et - eh >= 49 || eh == 0);
    X.status = fail_h ? QCAMS_LANE_FAIL_HMIN : X.status;
    go = go && !fail_h;
  }
  double xn[K], vn[K], s_new;
  float er[K], ev[K];
  dp_step_grp<MORSE, G, SEQ>(L, T, X.rho, X.vel, X.acc, X.h, xn, vn, er, ev, s_new, op);
  unsigned bad = 0, ignore = 0;
  float part = 0.f, qrs[K], qvs[K];
  const float rt = ip.rtol_f, at = ip.atol_f;
  const float hf = mag_f(X.h, ignore), hhf = hf * hf;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const float scr = fmaf(rt, fmaxf(mag_f(X.rho[i], ignore), mag_f(xn[i], ignore)), at);
    const float qr = err_mag(er[i], bad) * hhf * rcp_approx(scr);
    part = fmaf(qr, qr, part);
    qrs[i] = qr;
    const float scv = fmaf(rt, fmaxf(mag_f(X.vel[i], ignore), mag_f(vn[i], ignore)), X.atv[i]);
    const float qv = err_mag(ev[i], bad) * hf * rcp_approx(scv);
    part = fmaf(qv, qv, part);
    qvs[i] = qv;
  }
  const float en2 =
      (SEQ ? grp_norm_seq<G>(qrs, qvs, L.base) : grp_sum<G>(part, L.base)) * (1.0f / 12.0f);
  bad = grp_or<G>(bad, L.base);
  X.calls += go ? 1 : 0;
  X.status = (go && bad) ? QCAMS_LANE_FAIL_NAN : X.status;
  go = go && !bad;
  const float fac = 0.9f * pow_m01(en2);
  const bool accept = go && en2 < 1.0f;
  float fa = (en2 == 0.0f) ? 10.0f : fminf(10.0f, fac);
  fa = X.rejected ? fminf(1.0f, fa) : fa;
  const float f = accept ? fa : fmaxf(0.2f, fac);
  const double tn = X.t + X.h;
  X.t = accept ? tn : X.t;
  X.h = go ? X.h * static_cast<double>(f) : X.h;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    X.rho[i] = accept ? xn[i] : X.rho[i];
    X.vel[i] = accept ? vn[i] : X.vel[i];
    X.acc[0][i] = accept ? X.acc[6][i] : X.acc[0][i];
  }
  X.nacc += accept ? 1 : 0;
  X.nrej += (go && !accept) ? 1 : 0;
  X.rejected = go ? !accept : X.rejected;
  // stop rules on the accepted state, reduced over the group
  const long long smax = grp_max<G>(dbits(s_new), L.base);
  float radial;   // rho2 . P2 / mu123
  if (SEQ) {
    // the rho2 components are the last of each lane (G = 3) or lanes 3-5
    const float r = signed_f(X.rho[K - 1]), v = signed_f(X.vel[K - 1]);
    constexpr int at = G == 3 ? 0 : 3;
    float ra[3], va[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      ra[i] = __shfl_sync(FULL, r, L.base + at + i);
      va[i] = __shfl_sync(FULL, v, L.base + at + i);
    }
    radial = fmaf(ra[0], va[0], fmaf(ra[1], va[1], ra[2] * va[2]));
  } else {
    float rad = 0.0f;   // from the lane's rho2 components
#pragma unroll
    for (int i = 0; i < K; ++i)
      rad += L.comp(i) >= 3 ? signed_f(X.rho[i]) * signed_f(X.vel[i]) : 0.0f;
    radial = grp_sum<G>(rad, L.base);
  }
  unsigned collapse = 0;
  if (!MORSE)
    collapse = (L.q.kind == QCAMS_BUCK && dbits(s_new) < dbits(shapes[sid * 3 + L.j].r_b2)) ? 1u : 0u;
  collapse = grp_or<G>(collapse, L.base);
  int st = X.status;
  st = (accept && dbits(X.t) >= dbits(X.tmax)) ? QCAMS_LANE_DONE_TMAX : st;
  st = (accept && smax > dbits(ip.r_stop2) && radial > 0.0f) ? QCAMS_LANE_DONE_RSTOP : st;
  st = (accept && collapse) ? QCAMS_LANE_FAIL_COLLAPSE : st;
  st = (go && st == QCAMS_LANE_RUNNING && (long long)(X.nacc + X.nrej) >= ip.max_steps)
           ? QCAMS_LANE_FAIL_MAXSTEPS : st;
  X.status = st;
}

// One warp per block, 32 / G trajectories per warp (lanes G k .. G k + G - 1
// for trajectory (32 / G) w + k of warp w), no refill: every lane runs
// until the last trajectory of its warp is done.
template <bool MORSE, int G>
__global__ void __launch_bounds__(kGrpBlock) k_integrate_grp(SysSet sys, const DevShape* shapes,
                                                             IntegParams ip, DevBatch B,
                                                             unsigned long long* counters) {
  constexpr int K = Grp<G>::K, PER_WARP = Grp<G>::PER_WARP;
  __shared__ double sT[kExpTableSize], sC[kCoefs], sK[kOpRegs];
  op_reg_fill(sK);
  load_coefs(sC);
  load_exp_table(sT);   // ends with a barrier
  OpReg op;
  op.load(sK);
  const int lane = threadIdx.x & 31;
  const int used = PER_WARP * G;   // lanes of whole groups; the rest mirror the last group
  Grp<G> L;
  L.c = lane < used ? lane % G : lane - used;
  L.base = lane < used ? lane - L.c : used - G;
  L.j = L.c % 3;
  L.coef = sC;
  const int64_t i =
      ((int64_t)blockIdx.x * (kGrpBlock / 32) + (threadIdx.x >> 5)) * PER_WARP + L.base / G;
  const bool owner = lane < used && i < B.n;   // stores its components
  const int64_t ir = i < B.n ? i : B.n - 1;    // lanes past the batch mirror its last trajectory
  const int status0 = B.status[ir];
  int sid = B.sys_id[ir];
  const bool sid_ok = sid >= 0 && sid < sys.n;
  if (owner && L.c == 0 && runnable(status0) && !sid_ok) B.status[i] = QCAMS_LANE_INVALID;
  const bool active = owner && runnable(status0) && sid_ok;
  if (!sid_ok) sid = 0;   // keep the frozen lanes' arithmetic defined
  const DevSys& S = sys.s[sid];
  L.q = S.pair[L.j];
            L.cA = S.cA;
            L.cB = S.cB;
  L.kf = MORSE ? S.kf_morse[L.j] : S.kf[L.j];
  L.kh = L.j == 0 ? L.kf : (MORSE ? S.kf_morse[2 + L.j] : S.kf[2 + L.j]);
  if (G == 6 && L.c >= 3) L.kf = L.kh;

  GrpLane<K> X;
  double inv_mu[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int cg = L.comp(k);
    inv_mu[k] = cg < 3 ? S.inv_mu12 : S.inv_mu123;
    X.atv[k] = (float)(ip.atol * inv_mu[k]);
    X.rho[k] = B.y[cg][ir];
    X.vel[k] = B.y[6 + cg][ir] * inv_mu[k];
  }
  X.t = B.t[ir];
  X.h = B.h[ir];
  X.tmax = ip.t_stop * B.t_scale[ir];
  X.nacc = B.nsteps[ir];
  X.nrej = B.nrej[ir];
  X.calls = 0;
  X.rejected = false;
  X.status = active ? QCAMS_LANE_RUNNING : QCAMS_LANE_INVALID;
  double s_dummy;
  accel_grp<MORSE, G, false>(L, sT, X.rho, X.acc[0], s_dummy, op);
  unsigned long long rhs = active ? 1 : 0, steps = 0;
  const bool need_h = active && !(X.h > 0.0);
  if (__any_sync(FULL, need_h)) {
    const double h0 = initial_step_grp<MORSE, G>(L, sT, X, inv_mu, ip.rtol, ip.atol, op);
    X.h = need_h ? h0 : X.h;
    rhs += need_h ? 1 : 0;
  }
  while (__any_sync(FULL, X.status == QCAMS_LANE_RUNNING))
    attempt_grp<MORSE, G, false>(L, shapes, sid, ip, sT, X, op);
  if (active) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int cg = L.comp(k);
      B.y[cg][i] = X.rho[k];
      B.y[6 + cg][i] = X.vel[k] * (cg < 3 ? S.mu12 : S.mu123);
    }
    if (L.c == 0) {
      B.t[i] = X.t;
      B.h[i] = X.h;
      B.status[i] = static_cast<uint8_t>(X.status);
      B.nsteps[i] = X.nacc;
      B.nrej[i] = X.nrej;
    }
  }
  // counters per trajectory, from its group-index-0 lane
  rhs = (active && L.c == 0) ? rhs + 6ull * X.calls : 0;
  steps = (active && L.c == 0) ? (unsigned long long)X.calls : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rhs += __shfl_xor_sync(FULL, rhs, o);
    steps += __shfl_xor_sync(FULL, steps, o);
  }
  if (lane == 0) {
    atomicAdd(&counters[0], rhs);
    atomicAdd(&counters[1], steps);
  }
}

// Load trajectory idx into its group's lanes: a start (positions and
// momenta) or a resumed one (velocities in y[6..11], flags in the status).
template <bool MORSE, int G>
__device__ __forceinline__ void group_load(const SysSet& sys, const IntegParams& ip,
                                           const DevBatch& B, int64_t idx, int st, bool resumed, int sid,
                                           Grp<G>& L, GrpLane<Grp<G>::K>& X) {
  const DevSys& S = sys.s[sid];
  L.q = S.pair[L.j];
  L.cA = S.cA;
  L.cB = S.cB;
  L.kf = MORSE ? S.kf_morse[L.j] : S.kf[L.j];
  L.kh = L.j == 0 ? L.kf : (MORSE ? S.kf_morse[2 + L.j] : S.kf[2 + L.j]);
  if (G == 6 && L.c >= 3) L.kf = L.kh;
#pragma unroll
  for (int k = 0; k < Grp<G>::K; ++k) {
    const int cg = L.comp(k);
    const double inv_mu = cg < 3 ? S.inv_mu12 : S.inv_mu123, v = B.y[6 + cg][idx];
    X.atv[k] = (float)(ip.atol * inv_mu);
    X.rho[k] = B.y[cg][idx];
    X.vel[k] = resumed ? v : v * inv_mu;
  }
  X.t = B.t[idx];
  X.h = B.h[idx];
  X.tmax = ip.t_stop * B.t_scale[idx];
  X.nacc = B.nsteps[idx];
  X.nrej = B.nrej[idx];
  X.calls = 0;
  X.rejected = resumed && (st & kHandoffRejected);
  X.status = QCAMS_LANE_RUNNING;
}

// Store a trajectory: finished (momenta, its final status) or, with handoff,
// as it stands between two attempts.
template <int G>
__device__ __forceinline__ void group_store(const DevSys& S, const DevBatch& B, int64_t idx,
                                            const Grp<G>& L, const GrpLane<Grp<G>::K>& X,
                                            bool handoff) {
#pragma unroll
  for (int k = 0; k < Grp<G>::K; ++k) {
    const int cg = L.comp(k);
    B.y[cg][idx] = X.rho[k];
    B.y[6 + cg][idx] = handoff ? X.vel[k] : X.vel[k] * (cg < 3 ? S.mu12 : S.mu123);
  }
  if (L.c == 0) {
    B.t[idx] = X.t;
    B.h[idx] = X.h;
    B.status[idx] = static_cast<uint8_t>(
        handoff ? kHandoff | (X.rejected ? kHandoffRejected : 0) : X.status);
    B.nsteps[idx] = X.nacc;
    B.nrej[idx] = X.nrej;
  }
}

// The one-thread kernels' trajectories, bit for bit, with G lanes each and a
// refill queue: a group that is done takes the next trajectory of its source
// (all lanes, or the list an earlier stage handed on), with one atomicAdd
// per warp for all groups that need work.  Once the source is used up and at
// most `keep` trajectories are unfinished, every warp stores its own to the
// output list and ends (stage_queue in qcams_internal.h).
template <bool MORSE, int G>
__global__ void __launch_bounds__(kQueueBlock, G == 3 ? 3 : 4)
    k_integrate_queue(SysSet sys, const DevShape* shapes, IntegParams ip, DevBatch B,
                      unsigned long long* counters, StageQueue q) {
  constexpr int K = Grp<G>::K, PER_WARP = Grp<G>::PER_WARP;
  const int64_t n = q.list_in ? (int64_t)*q.n_in : B.n;
  // nothing left for this block (every block takes at least its first batch)
  if ((int64_t)blockIdx.x * (PER_WARP * (kQueueBlock / 32)) >= n) return;
  __shared__ double sT[kExpTableSize], sC[kCoefs], sK[kOpRegs];
  op_reg_fill(sK);
  load_coefs(sC);
  load_exp_table(sT);   // ends with a barrier
  OpReg op;
  op.load(sK);
  const int lane = threadIdx.x & 31;
  const int used = PER_WARP * G;   // lanes of whole groups; the rest mirror the last group
  Grp<G> L;
  L.c = lane < used ? lane % G : lane - used;
  L.base = lane < used ? lane - L.c : used - G;
  L.j = L.c % 3;
  L.coef = sC;
  const bool owner = lane < used, first = owner && L.c == 0;
  int64_t idx = 0;
  int sid = 0;
  bool have = false, exhausted = false;
  GrpLane<K> X;
  L.q = sys.s[0].pair[L.j];
  L.kf = L.kh = L.cA = L.cB = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {   // an absent trajectory's lanes hold defined values
    X.atv[k] = 0.0f;
    X.rho[k] = 1.0;
    X.vel[k] = X.acc[0][k] = 0.0;
  }
  X.t = X.h = X.tmax = 0.0;
  X.nacc = X.nrej = X.calls = 0;
  X.rejected = false;
  X.status = QCAMS_LANE_INVALID;
  unsigned long long rhs = 0, steps = 0;
  for (;;) {
    // one bit per group that needs work
    const unsigned want = __ballot_sync(FULL, first && !have && !exhausted);
    if (want) {
      const int leader = __ffs(want) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(q.head, (unsigned long long)__popc(want));
      base = __shfl_sync(FULL, base, leader);
      bool fresh = false, started = false, skip = false;
      int st = 0;
      if (!have && !exhausted) {
        const int64_t k = (int64_t)(base + __popc(want & ((1u << L.base) - 1u)));
        if (k >= n) {
          exhausted = true;
        } else {
          idx = q.list_in ? q.list_in[k] : k;
          st = B.status[idx];
          started = q.handed_on && (st & kHandoff);
          const int s_in = B.sys_id[idx];
          const bool run = started || runnable(st), ok = s_in >= 0 && s_in < sys.n;
          fresh = run && ok;
          skip = !fresh;
          if (fresh) sid = s_in;
          if (!(run && !ok)) st = fresh ? st : -1;
          else st = -2;   // runnable, but no such system
        }
      }
      __syncwarp();   // every lane has read its status
      if (first && st == -2) B.status[idx] = QCAMS_LANE_INVALID;
      const unsigned gone = __ballot_sync(FULL, first && skip);
      if (gone && lane == 0) atomicAdd(q.retired, (unsigned long long)__popc(gone));
      if (fresh) {
        group_load<MORSE, G>(sys, ip, B, idx, st, started, sid, L, X);
        have = true;
      }
      if (__any_sync(FULL, fresh)) {
        // acc[0] is the force at rho of a running trajectory too (FSAL), so
        // the whole warp forms it again
        double s_dummy;
        accel_grp<MORSE, G, true>(L, sT, X.rho, X.acc[0], s_dummy, op);
        rhs += (fresh && !started && first) ? 1 : 0;
      }
    }
    if (!__any_sync(FULL, have)) {
      if (__all_sync(FULL, exhausted)) break;
      continue;
    }
    if (q.keep > 0 && stage_over(q, n, lane)) {
      const unsigned pass = __ballot_sync(FULL, first && have);
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd(q.n_out, (unsigned long long)__popc(pass));
      at = __shfl_sync(FULL, at, 0);
      if (have && owner) {
        group_store<G>(sys.s[sid], B, idx, L, X, true);
        if (first) {
          q.list_out[at + __popc(pass & ((1u << lane) - 1u))] = idx;
          rhs += 6ull * X.calls;
          steps += X.calls;
        }
      }
      break;
    }
    attempt_grp<MORSE, G, true>(L, shapes, sid, ip, sT, X, op);
    const bool done = have && X.status != QCAMS_LANE_RUNNING;
    const unsigned ended = __ballot_sync(FULL, first && done);
    if (ended) {
      if (done && owner) {
        group_store<G>(sys.s[sid], B, idx, L, X, false);
        rhs += first ? 6ull * X.calls : 0;
        steps += first ? X.calls : 0;
      }
      have = have && !done;
      if (lane == 0) atomicAdd(q.retired, (unsigned long long)__popc(ended));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rhs += __shfl_xor_sync(FULL, rhs, o);
    steps += __shfl_xor_sync(FULL, steps, o);
  }
  if (lane == 0) {
    atomicAdd(&counters[0], rhs);
    atomicAdd(&counters[1], steps);
  }
}

template <int G>
cudaError_t launch_grp(const SysSet& sys, const DevShape* shapes, const IntegParams& ip,
                       const DevBatch& b, unsigned long long* counters, cudaStream_t st,
                       bool all_morse) {
  const long long warps = (b.n + Grp<G>::PER_WARP - 1) / Grp<G>::PER_WARP;
  const unsigned grid = (unsigned)((warps + kGrpBlock / 32 - 1) / (kGrpBlock / 32));
  if (all_morse)
    k_integrate_grp<true, G><<<grid, kGrpBlock, 0, st>>>(sys, shapes, ip, b, counters);
  else
    k_integrate_grp<false, G><<<grid, kGrpBlock, 0, st>>>(sys, shapes, ip, b, counters);
  return cudaGetLastError();
}

template <bool MORSE, int G>
cudaError_t launch_queue(const SysSet& sys, const DevShape* shapes, const IntegParams& ip,
                         const DevBatch& b, int64_t n_max, int sm_count,
                         unsigned long long* counters, const StageQueue& q, cudaStream_t st) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, k_integrate_queue<MORSE, G>, kQueueBlock, 0);
  if (e != cudaSuccess) return e;
  constexpr int per_block = Grp<G>::PER_WARP * (kQueueBlock / 32);
  const long long need = (n_max + per_block - 1) / per_block;
  long long grid = (long long)(per_sm < 1 ? 1 : per_sm) * sm_count;
  if (grid > need) grid = need;
  k_integrate_queue<MORSE, G>
      <<<(unsigned)grid, kQueueBlock, 0, st>>>(sys, shapes, ip, b, counters, q);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_integrate_queue(const SysSet& sys, const DevShape* shapes,
                                   const IntegParams& ip, const DevBatch& b, int lanes,
                                   int64_t n_max, int sm_count, unsigned long long* counters,
                                   const StageQueue& q, cudaStream_t st, bool all_morse) {
  if (lanes == 3)
    return all_morse ? launch_queue<true, 3>(sys, shapes, ip, b, n_max, sm_count, counters, q, st)
                     : launch_queue<false, 3>(sys, shapes, ip, b, n_max, sm_count, counters, q, st);
  return all_morse ? launch_queue<true, 6>(sys, shapes, ip, b, n_max, sm_count, counters, q, st)
                   : launch_queue<false, 6>(sys, shapes, ip, b, n_max, sm_count, counters, q, st);
}

cudaError_t grouped_func_info(int lanes, bool all_morse, int* regs, int* blocks_per_sm) {
  cudaFuncAttributes a;
  cudaError_t e = cudaErrorInvalidValue;
#define QCAMS_GRP_INFO(M, G)                                                               \
  e = cudaFuncGetAttributes(&a, k_integrate_grp<M, G>);                                    \
  if (e == cudaSuccess)                                                                    \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_integrate_grp<M, G>, \
                                                      kGrpBlock, 0)
  if (lanes == 3) {
    if (all_morse) { QCAMS_GRP_INFO(true, 3); } else { QCAMS_GRP_INFO(false, 3); }
  } else if (lanes == 6) {
    if (all_morse) { QCAMS_GRP_INFO(true, 6); } else { QCAMS_GRP_INFO(false, 6); }
  }
#undef QCAMS_GRP_INFO
  if (e == cudaSuccess) *regs = a.numRegs;
  return e;
}

cudaError_t queue_func_info(bool all_morse, int* regs, int* blocks_per_sm) {
  cudaFuncAttributes a;
  cudaError_t e = all_morse ? cudaFuncGetAttributes(&a, k_integrate_queue<true, 3>)
                            : cudaFuncGetAttributes(&a, k_integrate_queue<false, 3>);
  if (e != cudaSuccess) return e;
  *regs = a.numRegs;
  return all_morse ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                         blocks_per_sm, k_integrate_queue<true, 3>, kQueueBlock, 0)
                   : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                         blocks_per_sm, k_integrate_queue<false, 3>, kQueueBlock, 0);
}

cudaError_t launch_integrate_grouped(const SysSet& sys, const DevShape* shapes,
                                     const IntegParams& ip, const DevBatch& b, int lanes,
                                     unsigned long long* counters, cudaStream_t st,
                                     bool all_morse) {
  if (b.n == 0) return cudaSuccess;
  if (lanes == 3) return launch_grp<3>(sys, shapes, ip, b, counters, st, all_morse);
  if (lanes == 6) return launch_grp<6>(sys, shapes, ip, b, counters, st, all_morse);
  return cudaErrorInvalidValue;
}

}  // namespace qcams
