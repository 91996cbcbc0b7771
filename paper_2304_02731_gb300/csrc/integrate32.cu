// FP32 trajectory integrator with compensated (Kahan) state updates.
//
// Same method as the FP64 integrator (Hamilton's equations in Jacobi
// coordinates, Sec. 2 Eqs. 3-4; Dormand-Prince 5(4) with SciPy's RK45 step
// control, Sec. 3.2; stop rules of Sec. 3.1) in single precision, for the
// FP32 study of the sweep.  GB300 runs FP32 at 64x its FP64 rate, so this
// path trades accuracy (tolerances ~1e-6) for throughput.
//
//  * Stages, forces and the error norm are FP32 (the hardware 1/sqrt and
//    2^x of x log2 e, relative error below 2 + 1.2 |x| ulp; the
//    exponentials of the force law have |x| < 2 where the force matters and
//    up to ~35 only for pairs far apart, whose forces are negligible).
//  * Each step adds a small increment to a large state (|rho| ~ 30 bohr,
//    increments ~1e-2), so plain FP32 accumulation would lose ~1e-7 |y| per
//    step.  Positions and velocities are therefore kept as Kahan pairs
//    (value, compensation): y_true = y - c, and every update y += d folds the
//    rounding error of the previous updates back in (Kahan, CACM 8 (1965) 40).
//  * Time is FP64 (one add per step).  Initial conditions, the level table,
//    the energy bookkeeping and the product analysis stay FP64: the kernel
//    loads the FP64 state as (float, compensation) and stores y - c in FP64.
#include <cuda_runtime.h>

#include <cstring>

#include "dp5_tableau.cuh"
#include "qcams_device.cuh"
#include "qcams_internal.h"

namespace qcams {
namespace {

struct RknTabF {
  float a2[8][8], c[8], b[8], e[8], ea[8];
};
__host__ __device__ constexpr RknTabF make_rkn_tab_f() {
  RknTabF f{};
  for (int s = 1; s <= 7; ++s) {
    f.c[s] = (float)dpC(s);
    f.b[s] = (float)dpB(s);
    f.e[s] = (float)dpE(s);
    f.ea[s] = dpEAZero(s) ? 0.0f : (float)dpEA(s);
    for (int q = 1; q <= 7; ++q) f.a2[s][q] = dpA2Zero(s, q) ? 0.0f : (float)dpA2(s, q);
  }
  return f;
}

constexpr unsigned FULL = 0xffffffffu;

// Approximate reciprocal (one MUFU instruction, about 1 ulp): the error norm
// needs only a few significant bits, and the scales it divides by are
// positive and far from the FP32 range limits (atol > 0).
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 2^x (one MUFU instruction, relative error about 2^-22): the force law's
// exponentials e^y are taken as 2^(y log2 e) with the constants of y
// pre-scaled by log2 e on the host, so no multiply precedes the MUFU.
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 1/sqrt(s) (one MUFU instruction, about 1 ulp).  Flush-to-zero: s is a
// squared pair distance, subnormal only for pairs closer than 1e-19 bohr,
// where the lane fails on the infinite force it gets.
__device__ __forceinline__ float rsqrt_approx(float s) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s));
  return r;
}

// x^(-1/10) for the step-size factor, as 2^(-log2(x) / 10) (two MUFU
// instructions and a multiply).  x = 0 or subnormal gives +inf, which the
// controller caps at the maximum growth factor as it does for a zero norm.
__device__ __forceinline__ float pow_m01(float x) {
  float l, r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(-0.1f * l));
  return r;
}

// Two FP32 values in one aligned register pair, with the packed multiply-add,
// multiply and add of sm_100: one instruction for two IEEE operations (each
// half rounds as the scalar instruction does).
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo_of(F2 a) {
  float l, h;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(l), "=f"(h) : "l"(a.v));
  return l;
}
__device__ __forceinline__ float hi_of(F2 a) {
  float l, h;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(l), "=f"(h) : "l"(a.v));
  return h;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 dup(float a) { return f2(a, a); }
// a - b: b's sign flips inside the (exact) product with -1
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, F2{0xbf800000bf800000ull}, a); }
// The six components of a pair of Jacobi vectors are held as (0, 1), (3, 4)
// and (2, 5): the pair vectors rho2 - cB rho1 and rho2 + cA rho1 then take
// one packed and one scalar multiply-add each.
struct V6 {
  F2 a, b, c;
};
__device__ __forceinline__ void get6(const V6& v, float* x) {
  x[0] = lo_of(v.a);
  x[1] = hi_of(v.a);
  x[2] = lo_of(v.c);
  x[3] = lo_of(v.b);
  x[4] = hi_of(v.b);
  x[5] = hi_of(v.c);
}
__device__ __forceinline__ V6 put6(const float* x) {
  return V6{f2(x[0], x[1]), f2(x[3], x[4]), f2(x[2], x[5])};
}
__device__ __forceinline__ V6 fma6(F2 w, const V6& x, const V6& y) {
  return V6{fma2(w, x.a, y.a), fma2(w, x.b, y.b), fma2(w, x.c, y.c)};
}
__device__ __forceinline__ V6 mul6(F2 w, const V6& x) {
  return V6{mul2(w, x.a), mul2(w, x.b), mul2(w, x.c)};
}
__device__ __forceinline__ V6 add6(const V6& x, const V6& y) {
  return V6{add2(x.a, y.a), add2(x.b, y.b), add2(x.c, y.c)};
}
__device__ __forceinline__ V6 sub6(const V6& x, const V6& y) {
  return V6{sub2(x.a, y.a), sub2(x.b, y.b), sub2(x.c, y.c)};
}
__device__ __forceinline__ F2 sel2(bool p, F2 a, F2 b) { return F2{p ? a.v : b.v}; }
__device__ __forceinline__ V6 sel6(bool p, const V6& x, const V6& y) {
  return V6{sel2(p, x.a, y.a), sel2(p, x.b, y.b), sel2(p, x.c, y.c)};
}

// The Runge-Kutta-Nystrom coefficients, each in both halves of a pair.
struct RknTab2 {
  F2 a2[8][8], b[8], e[8], ea[8];
};
constexpr F2 both(float x) {
  const unsigned long long u = __builtin_bit_cast(unsigned, x);
  return F2{u << 32 | u};
}
constexpr RknTab2 make_rkn_tab2() {
  RknTab2 t{};
  const RknTabF f = make_rkn_tab_f();
  for (int s = 1; s <= 7; ++s) {
    t.b[s] = both(f.b[s]);
    t.e[s] = both(f.e[s]);
    t.ea[s] = both(f.ea[s]);
    for (int q = 1; q <= 7; ++q) t.a2[s][q] = both(f.a2[s][q]);
  }
  return t;
}
__constant__ RknTab2 kT2 = make_rkn_tab2();

// FP32 copies of the per-system constants (built on the host, so the kernel
// never converts doubles in its inner loop).
struct PairF {
  int kind, m, n, pad;
  float c0, c1, c2, c3, c4;
  float l0, l1;   // exponent constants times log2 e: Morse c0, c1; Buckingham
                  // ln(A B) (l0) and B (l1), so that 2^(l0 - l1 r) = A B e^{-B r}
};
struct SysF {
  float cA, cB, inv_mu12, inv_mu123, mu12, mu123;
  float kf[5], kf_morse[5];
  double mu12d, mu123d;
  PairF pair[3];
  // packed operands: (-cB, -cB), (cA, cA); of the pairs BC and CA the Morse
  // exponent's -l0 and l1 and the force coefficients (f1, f2) and (h1, h2)
  F2 ncB, cA2, nl0, l1, f12, h12;
};
struct SysSetF {
  SysF s[QCAMS_MAX_SYS];
  int n, pad;
};

__device__ __forceinline__ float ipowf_(float x, int n) {
  float r = 1.0f;
  while (n) {
    if (n & 1) r *= x;
    x *= x;
    n >>= 1;
  }
  return r;
}

// u = V'(r)/r (generic) or x (1 - x)/r (all-Morse kernels: the factor
// 2 alpha De is folded into kf_morse)
template <bool MORSE>
__device__ __forceinline__ float pair_u(const PairF& q, float s) {
  const float ri = rsqrt_approx(s);
  const float r = s * ri;
  if (MORSE) {
    const float x = ex2_approx(fmaf(-q.l0, r, q.l1));   // e^{-alpha (r - re)}
    return fmaf(-x, x, x) * ri;
  }
  if (q.kind == QCAMS_MORSE) {   // a Morse pair of a mixed system: V'/r = 2 alpha De x (1 - x) / r
    const float x = ex2_approx(fmaf(-q.l0, r, q.l1));
    return q.c2 * fmaf(-x, x, x) * ri;
  }
  const float ri2 = ri * ri;
  if (q.kind == QCAMS_LJ) {
    if (q.n == 6 && (q.m == 12 || q.m == 8)) {   // shared powers of 1/r^2
      const float ri4 = ri2 * ri2, ri6 = ri4 * ri2;
      const float h = q.m == 12 ? ri6 : ri4;
      return fmaf(q.c3, ri6, -q.c2 * (h * h)) * ri2;
    }
    return (q.c3 * ipowf_(ri, q.n) - q.c2 * ipowf_(ri, q.m)) * ri2;
  }
  // Buckingham: 6 C6 / r^8 - A B e^{-B r} / r
  const float ri4 = ri2 * ri2;
  return fmaf(q.c3, ri4 * ri4, -(ex2_approx(fmaf(-q.l1, r, q.l0)) * ri));
}

template <bool MORSE>
__device__ __forceinline__ void accel(const SysF& S, const V6& x, V6& a, float* s2) {
  const F2 bc = fma2(S.ncB, x.a, x.b), ca = fma2(S.cA2, x.a, x.b);
  const float x0 = lo_of(x.a), x1 = hi_of(x.a), x2 = lo_of(x.c);
  const float rbc0 = lo_of(bc), rbc1 = hi_of(bc), rbc2 = fmaf(-S.cB, x2, hi_of(x.c));
  const float rca0 = lo_of(ca), rca1 = hi_of(ca), rca2 = fmaf(S.cA, x2, hi_of(x.c));
  s2[0] = fmaf(x0, x0, fmaf(x1, x1, x2 * x2));
  s2[1] = fmaf(rbc0, rbc0, fmaf(rbc1, rbc1, rbc2 * rbc2));
  s2[2] = fmaf(rca0, rca0, fmaf(rca1, rca1, rca2 * rca2));
  float f0, f1, f2_, h1, h2;
  const float u0 = pair_u<MORSE>(S.pair[0], s2[0]);
  if (MORSE) {
    f0 = S.kf_morse[0] * u0;
    // pairs BC and CA packed (pair_u's operations)
    const float i1 = rsqrt_approx(s2[1]), i2 = rsqrt_approx(s2[2]);
    const F2 ri = f2(i1, i2), arg = fma2(S.nl0, mul2(f2(s2[1], s2[2]), ri), S.l1);
    const float e1 = ex2_approx(lo_of(arg)), e2 = ex2_approx(hi_of(arg));
    const F2 u = mul2(f2(fmaf(-e1, e1, e1), fmaf(-e2, e2, e2)), ri);
    const F2 f = mul2(S.f12, u), h = mul2(S.h12, u);
    f1 = lo_of(f);
    f2_ = hi_of(f);
    h1 = lo_of(h);
    h2 = hi_of(h);
  } else {
    const float u1 = pair_u<MORSE>(S.pair[1], s2[1]), u2 = pair_u<MORSE>(S.pair[2], s2[2]);
    f0 = S.kf[0] * u0;
    f1 = S.kf[1] * u1;
    f2_ = S.kf[2] * u2;
    h1 = S.kf[3] * u1;
    h2 = S.kf[4] * u2;
  }
  a.a = f2(fmaf(f0, x0, fmaf(f1, rbc0, f2_ * rca0)), fmaf(f0, x1, fmaf(f1, rbc1, f2_ * rca1)));
  a.b = f2(fmaf(h1, rbc0, h2 * rca0), fmaf(h1, rbc1, h2 * rca1));
  a.c = f2(fmaf(f0, x2, fmaf(f1, rbc2, f2_ * rca2)), fmaf(h1, rbc2, h2 * rca2));
}

struct Lane32 {
  V6 rho, vel;       // state (true value = state - compensation)
  V6 ncrho, ncvel;   // Kahan compensations, negated
  V6 acc[7];
  double t, tmax;
  float h;
  float atv[2];
  float rb2[3];           // Buckingham collapse radii squared (0 for other kinds)
  int nacc, nrej, calls, status, sid;
  bool rejected;
};

// atol + rtol max(|a|, |b|), halves apart.
__device__ __forceinline__ F2 scale2(F2 rt, F2 at, F2 a, F2 b) {
  return fma2(rt, f2(fmaxf(fabsf(lo_of(a)), fabsf(lo_of(b))), fmaxf(fabsf(hi_of(a)), fabsf(hi_of(b)))),
              at);
}
__device__ __forceinline__ F2 rcp2(F2 a) { return f2(rcp_approx(lo_of(a)), rcp_approx(hi_of(a))); }

// One adaptive attempt (SciPy RK45 rules, as in the FP64 integrator), all
// stages in FP32; the accepted increments are added with compensation.
// ONE: the batch has a single system, so its constants are read with a
// compile-time index (constant-bank operands, no per-lane indexed loads).
// Every linear combination of 6-vectors runs in packed instructions: 628
// instructions a step instead of 787, which bound the kernel by issue (79 %
// of the rate); it now waits on the FMA pipes' bursts and on latency with 16
// warps per SM (issue 69 %, FMA pipes 68 %).  The full sweep: 117.6 -> 110.7
// ms.
template <bool MORSE, bool ONE>
__device__ __forceinline__ void attempt(const SysSetF& sys, const IntegParams& ip, Lane32& L) {
  const SysF& S = sys.s[ONE ? 0 : L.sid];
  {
    const int eh = (__float_as_int(L.h) >> 23) & 0xff;
    const int et = (__double2hiint(L.t) >> 20) & 0x7ff;
    if ((et - 1023) - (eh - 127) >= 49 || eh == 0) {
      L.status = QCAMS_LANE_FAIL_HMIN;
      return;
    }
  }
  const float h = L.h, hh = h * h;
  const F2 h2 = dup(h), hh2 = dup(hh);
  V6 x;
  float s2[3];
#define QCAMS_STAGE(sIdx)                                                            \
  {                                                                                  \
    x = fma6(dup(h * (float)dpC(sIdx)), L.vel, L.rho); /* folded: c_6 = 1 */         \
    _Pragma("unroll") for (int q = 1; q <= (sIdx) - 2; ++q)                          \
        if (!dpA2Zero(sIdx, q)) x = fma6(mul2(hh2, kT2.a2[sIdx][q]), L.acc[q - 1], x); \
    accel<MORSE>(S, x, L.acc[(sIdx) - 1], s2);                                       \
  }
  QCAMS_STAGE(2)   // (A^2)_{2q} = 0, no acceleration term
  QCAMS_STAGE(3)
  QCAMS_STAGE(4)
  QCAMS_STAGE(5)
  QCAMS_STAGE(6)
#undef QCAMS_STAGE
  // stage 7 = the new state: increment d = h v + h^2 sum (b^T A)_q a_q,
  // compensated sum x7 = rho + (d - c)
  V6 sum{F2{0}, F2{0}, F2{0}};
#pragma unroll
  for (int q = 1; q <= 5; ++q)
    if (!dpA2Zero(7, q)) sum = fma6(kT2.a2[7][q], L.acc[q - 1], sum);
  const V6 yr = add6(fma6(hh2, sum, mul6(h2, L.vel)), L.ncrho);
  x = add6(L.rho, yr);
  accel<MORSE>(S, x, L.acc[6], s2);
  V6 vb = mul6(kT2.b[1], L.acc[0]);
#pragma unroll
  for (int q = 3; q <= 6; ++q) vb = fma6(kT2.b[q], L.acc[q - 1], vb);
  V6 ev = mul6(kT2.e[1], L.acc[0]);     // velocity error / h
#pragma unroll
  for (int q = 3; q <= 7; ++q) ev = fma6(kT2.e[q], L.acc[q - 1], ev);
  V6 er = mul6(kT2.ea[1], L.acc[0]);    // position error / h^2
#pragma unroll
  for (int q = 2; q <= 6; ++q)
    if (!dpEAZero(q)) er = fma6(kT2.ea[q], L.acc[q - 1], er);
  const V6 yv = fma6(h2, vb, L.ncvel);  // h vb - c
  const V6 vn = add6(L.vel, yv);
  // the factors h and h^2 multiply the two partial sums of squares once
  const F2 rt = dup(ip.rtol_f), at = dup(ip.atol_f);
  const V6 qr{mul2(er.a, rcp2(scale2(rt, at, L.rho.a, x.a))),
              mul2(er.b, rcp2(scale2(rt, at, L.rho.b, x.b))),
              mul2(er.c, rcp2(scale2(rt, at, L.rho.c, x.c)))};
  const V6 qv{mul2(ev.a, rcp2(scale2(rt, dup(L.atv[0]), L.vel.a, vn.a))),
              mul2(ev.b, rcp2(scale2(rt, dup(L.atv[1]), L.vel.b, vn.b))),
              mul2(ev.c, rcp2(scale2(rt, f2(L.atv[0], L.atv[1]), L.vel.c, vn.c)))};
  float sum_r = 0.0f, sum_v = 0.0f, tr[6], tv[6];
  get6(qr, tr);
  get6(qv, tv);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    sum_r = fmaf(tr[i], tr[i], sum_r);
    sum_v = fmaf(tv[i], tv[i], sum_v);
  }
  const float en2 = fmaf(hh, sum_v, (hh * hh) * sum_r) * (1.0f / 12.0f);
  L.calls += 1;
  if (!(en2 == en2)) {   // NaN fails the lane; an overflowing norm just rejects
    L.status = QCAMS_LANE_FAIL_NAN;
    return;
  }
  const float fac = 0.9f * pow_m01(en2);
  const bool accept = en2 < 1.0f;
  float fa = (en2 == 0.0f) ? 10.0f : fminf(10.0f, fac);
  fa = L.rejected ? fminf(1.0f, fa) : fa;
  const float f = accept ? fa : fmaxf(0.2f, fac);
  const double tn = L.t + (double)L.h;
  L.t = accept ? tn : L.t;
  L.h = L.h * f;
  // new compensation (x - rho) - y, negated
  L.ncrho = sel6(accept, sub6(yr, sub6(x, L.rho)), L.ncrho);
  L.ncvel = sel6(accept, sub6(yv, sub6(vn, L.vel)), L.ncvel);
  L.rho = sel6(accept, x, L.rho);
  L.vel = sel6(accept, vn, L.vel);
  L.acc[0] = sel6(accept, L.acc[6], L.acc[0]);
  L.nacc += accept ? 1 : 0;
  L.nrej += accept ? 0 : 1;
  L.rejected = !accept;
  const float smax = fmaxf(s2[0], fmaxf(s2[1], s2[2]));
  const float radial = fmaf(lo_of(L.rho.b), lo_of(L.vel.b),
                            fmaf(hi_of(L.rho.b), hi_of(L.vel.b), hi_of(L.rho.c) * hi_of(L.vel.c)));
  bool collapse = false;
  if (!MORSE) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
      collapse |= s2[k] < L.rb2[k];
  }
  int st = L.status;
  st = (accept && __double_as_longlong(L.t) >= __double_as_longlong(L.tmax))
           ? QCAMS_LANE_DONE_TMAX : st;
  st = (accept && smax > (float)ip.r_stop2 && radial > 0.0f) ? QCAMS_LANE_DONE_RSTOP : st;
  st = (accept && collapse) ? QCAMS_LANE_FAIL_COLLAPSE : st;
  st = (st == QCAMS_LANE_RUNNING && (long long)(L.nacc + L.nrej) >= ip.max_steps)
           ? QCAMS_LANE_FAIL_MAXSTEPS : st;
  L.status = st;
}

// Starting step (Hairer, Norsett & Wanner), in FP32.  The multiply-adds are
// written out, so that the sums round the same in every kernel.
__device__ __forceinline__ float add_squares(float s, float a, float b) {
  return __fadd_rn(s, fmaf(a, a, __fmul_rn(b, b)));
}
template <bool MORSE>
__device__ float initial_step(const SysF& S, const Lane32& L, float rtol, float atol) {
  float d0 = 0.f, d1 = 0.f, rho[6], vel[6], acc0[6];
  get6(L.rho, rho);
  get6(L.vel, vel);
  get6(L.acc[0], acc0);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const float scr = fmaf(fabsf(rho[i]), rtol, atol);
    const float scv = fmaf(fabsf(vel[i]), rtol, L.atv[i / 3]);
    const float q0 = rho[i] / scr, q1 = vel[i] / scv;
    d0 = add_squares(d0, q0, q1);
    const float p0 = vel[i] / scr, p1 = acc0[i] / scv;
    d1 = add_squares(d1, p0, p1);
  }
  d0 = sqrtf(d0 / 12.f);
  d1 = sqrtf(d1 / 12.f);
  const float h0 = (d0 < 1e-5f || d1 < 1e-5f) ? 1e-6f : 0.01f * d0 / d1;
  float x1[6], a1[6], s2[3];
#pragma unroll
  for (int i = 0; i < 6; ++i) x1[i] = fmaf(h0, vel[i], rho[i]);
  V6 av;
  accel<MORSE>(S, put6(x1), av, s2);
  get6(av, a1);
  float d2 = 0.f;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const float scr = fmaf(fabsf(rho[i]), rtol, atol);
    const float scv = fmaf(fabsf(vel[i]), rtol, L.atv[i / 3]);
    const float p0 = h0 * acc0[i] / scr, p1 = (a1[i] - acc0[i]) / scv;
    d2 = add_squares(d2, p0, p1);
  }
  d2 = sqrtf(d2 / 12.f) / h0;
  const float h1 = (d1 <= 1e-15f && d2 <= 1e-15f) ? fmaxf(1e-6f, h0 * 1e-3f)
                                                 : powf(0.01f / fmaxf(d1, d2), 0.2f);
  return fminf(100.f * h0, h1);
}

__device__ __forceinline__ bool runnable(int st) {
  return st == QCAMS_LANE_READY || st == QCAMS_LANE_RUNNING;
}

template <bool MORSE, bool ONE>
__device__ bool load(const SysSetF& sys, const DevShape* shapes, const IntegParams& ip,
                     const DevBatch& B, int64_t i, Lane32& L, unsigned long long& rhs) {
  L.status = B.status[i];
  if (!runnable(L.status)) return false;
  L.sid = B.sys_id[i];
  if (L.sid < 0 || L.sid >= sys.n) {
    B.status[i] = QCAMS_LANE_INVALID;
    return false;
  }
  const SysF& S = sys.s[ONE ? 0 : L.sid];
  float rho[6], vel[6], nr[6], nv[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double r = B.y[k][i];
    const double v = B.y[6 + k][i] * (k < 3 ? 1.0 / S.mu12d : 1.0 / S.mu123d);
    rho[k] = (float)r;
    nr[k] = -(float)((double)rho[k] - r);
    vel[k] = (float)v;
    nv[k] = -(float)((double)vel[k] - v);
  }
  L.rho = put6(rho);
  L.vel = put6(vel);
  L.ncrho = put6(nr);
  L.ncvel = put6(nv);
  L.t = B.t[i];
  L.h = (float)B.h[i];
  L.tmax = ip.t_stop * B.t_scale[i];
  L.nacc = B.nsteps[i];
  L.nrej = B.nrej[i];
  L.calls = 0;
  L.rejected = false;
  L.status = QCAMS_LANE_RUNNING;
  L.atv[0] = ip.atol_f * S.inv_mu12;
  L.atv[1] = ip.atol_f * S.inv_mu123;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    L.rb2[k] = (!MORSE && S.pair[k].kind == QCAMS_BUCK) ? (float)shapes[L.sid * 3 + k].r_b2 : 0.0f;
  float s2[3];
  accel<MORSE>(S, L.rho, L.acc[0], s2);
  rhs += 1;
  if (!(L.h > 0.0f)) {
    L.h = initial_step<MORSE>(S, L, ip.rtol_f, ip.atol_f);
    rhs += 1;
  }
  return true;
}

template <bool ONE>
__device__ void store(const SysSetF& sys, const DevBatch& B, int64_t i, const Lane32& L) {
  const SysF& S = sys.s[ONE ? 0 : L.sid];
  float rho[6], vel[6], nr[6], nv[6];
  get6(L.rho, rho);
  get6(L.vel, vel);
  get6(L.ncrho, nr);
  get6(L.ncvel, nv);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    B.y[k][i] = (double)rho[k] + (double)nr[k];
    B.y[6 + k][i] = ((double)vel[k] + (double)nv[k]) * (k < 3 ? S.mu12d : S.mu123d);
  }
  B.t[i] = L.t;
  B.h[i] = (double)L.h;
  B.status[i] = (uint8_t)L.status;
  B.nsteps[i] = L.nacc;
  B.nrej[i] = L.nrej;
}

__device__ __forceinline__ void flush(unsigned long long rhs, unsigned long long steps,
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

template <bool MORSE, bool ONE>
__global__ void __launch_bounds__(128) k_integrate32_plain(SysSetF sys, const DevShape* shapes,
                                                           IntegParams ip, DevBatch B,
                                                           unsigned long long* counters) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  unsigned long long rhs = 0, steps = 0;
  Lane32 L;
  if (i < B.n && load<MORSE, ONE>(sys, shapes, ip, B, i, L, rhs)) {
    while (L.status == QCAMS_LANE_RUNNING) attempt<MORSE, ONE>(sys, ip, L);
    rhs += 6ull * L.calls;
    steps += L.calls;
    store<ONE>(sys, B, i, L);
  }
  flush(rhs, steps, counters);
}

// The resident blocks per SM cap the registers: the all-Morse kernel takes
// 121, four blocks of 128 threads (five, at 96 registers, spill and run the
// sweep in 115.8 ms against 110.7; with several systems the four-block cap
// costs 32 bytes of spills: 1 M lanes of two systems 38.4 ms, of one 36.6);
// the generic one 120 or, with five blocks and 100 bytes of spills, 96: 35.8
// against 37.9 ms for 1 M lanes.
template <bool MORSE, bool ONE>
__global__ void __launch_bounds__(128, MORSE ? 4 : 5)
    k_integrate32_persistent(SysSetF sys, const DevShape* shapes, IntegParams ip, DevBatch B,
                             unsigned long long* counters, const long long* list) {
  const unsigned lane = threadIdx.x & 31u;
  unsigned long long rhs = 0, steps = 0;
  Lane32 L;
  int64_t idx = -1;
  bool have = false, exhausted = false;
  for (;;) {
    const bool need = !have && !exhausted;
    const unsigned want = __ballot_sync(FULL, need);
    if (want) {
      const int leader = __ffs(want) - 1;
      unsigned long long base = 0;
      if ((int)lane == leader) base = atomicAdd(&counters[2], (unsigned long long)__popc(want));
      base = __shfl_sync(FULL, base, leader);
      if (need) {
        const int64_t k = (int64_t)(base + __popc(want & ((1u << lane) - 1u)));
        if (k >= B.n) exhausted = true;
        else {
          idx = list ? list[k] : k;
          have = load<MORSE, ONE>(sys, shapes, ip, B, idx, L, rhs);
        }
      }
    }
    if (__all_sync(FULL, exhausted && !have)) break;
    if (have) {
      attempt<MORSE, ONE>(sys, ip, L);
      if (L.status != QCAMS_LANE_RUNNING) {
        rhs += 6ull * L.calls;
        steps += L.calls;
        store<ONE>(sys, B, idx, L);
        have = false;
      }
    }
  }
  flush(rhs, steps, counters);
}

SysSetF to_float(const SysSet& in) {
  SysSetF o{};
  o.n = in.n;
  for (int s = 0; s < in.n; ++s) {
    const DevSys& d = in.s[s];
    SysF& f = o.s[s];
    f.cA = (float)d.cA;
    f.cB = (float)d.cB;
    f.inv_mu12 = (float)d.inv_mu12;
    f.inv_mu123 = (float)d.inv_mu123;
    f.mu12 = (float)d.mu12;
    f.mu123 = (float)d.mu123;
    f.mu12d = d.mu12;
    f.mu123d = d.mu123;
    for (int k = 0; k < 5; ++k) {
      f.kf[k] = (float)d.kf[k];
      f.kf_morse[k] = (float)d.kf_morse[k];
    }
    for (int p = 0; p < 3; ++p) {
      const DevPair& q = d.pair[p];
      PairF& g = f.pair[p];
      g.kind = q.kind;
      g.m = q.m;
      g.n = q.n;
      g.c0 = (float)q.c0;
      g.c1 = (float)q.c1;
      g.c2 = (float)q.c2;
      g.c3 = (float)q.c3;
      g.c4 = (float)q.c4;
      const double log2e = 1.4426950408889634;
      g.l0 = (float)((q.kind == QCAMS_BUCK ? q.lc2 : q.c0) * log2e);
      g.l1 = (float)(q.c1 * log2e);
    }
    auto pack = [](float lo, float hi) {
      unsigned a, b;
      std::memcpy(&a, &lo, 4);
      std::memcpy(&b, &hi, 4);
      return F2{(unsigned long long)b << 32 | a};
    };
    f.ncB = pack(-f.cB, -f.cB);
    f.cA2 = pack(f.cA, f.cA);
    f.nl0 = pack(-f.pair[1].l0, -f.pair[2].l0);
    f.l1 = pack(f.pair[1].l1, f.pair[2].l1);
    f.f12 = pack(f.kf_morse[1], f.kf_morse[2]);
    f.h12 = pack(f.kf_morse[3], f.kf_morse[4]);
  }
  return o;
}

template <bool MORSE, bool ONE>
cudaError_t launch32_persistent(const SysSetF& sf, const DevShape* shapes, const IntegParams& ip,
                                const DevBatch& b, Ctx& ctx, cudaStream_t st) {
  const int block = 128;
  cudaError_t e = cudaMemsetAsync(ctx.counters + 2, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, k_integrate32_persistent<MORSE, ONE>, block, 0);
  if (e != cudaSuccess) return e;
  const long long* list = nullptr;
  // the slowest collisions first (figures at launch_queue_order)
  if (b.n >= kOrderMinLanes && lists_usable(b)) {
    long long* order = reinterpret_cast<long long*>(b.vprime);
    e = launch_queue_order(b, order, reinterpret_cast<unsigned*>(b.jprime), ctx.counters + 3, st);
    if (e != cudaSuccess) return e;
    list = order;
  }
  long long grid = (long long)(per_sm < 1 ? 1 : per_sm) * ctx.sm_count;
  const long long need_blocks = (b.n + block - 1) / block;
  if (grid > need_blocks) grid = need_blocks;
  if (grid < 1) grid = 1;
  k_integrate32_persistent<MORSE, ONE><<<(unsigned)grid, block, 0, st>>>(sf, shapes, ip, b,
                                                                        ctx.counters, list);
  return cudaGetLastError();
}

// Whether a batch runs in the refill queue (mode 1).
//
// The queue pays once a batch is several times what the GPU holds (384 to
// 640 lanes per SM): below, there is little to refill, its attempts are
// slower than those of one thread per lane, and its slowest lanes, taken
// first, share warps and SMs.  Milliseconds, queue / one thread each:
//   sweep, all energies       60,000 16.2 / 9.2, 125,000 21.0 / 12.9,
//                             260,000 22.0 / 20.1, 300,000 21.3 / 22.4
//   three generic systems     125,000 20.2 / 16.3, 260,000 25.2 / 22.7,
//                             300,000 22.9 / 23.9
//   LJ(12,6), one system      100,000 13.3 / 12.1, 125,000 12.8 / 13.6,
//                             150,000 13.6 / 13.0, 175,000 12.7 / 14.3
bool queue_pays(bool morse, bool one, int persistent, int64_t n, int64_t sms) {
  return persistent && n > (!morse && one ? 1024 : 1792) * sms;
}

template <bool MORSE, bool ONE>
cudaError_t launch32(const SysSetF& sf, const DevShape* shapes, const IntegParams& ip,
                     const DevBatch& b, int persistent, Ctx& ctx, cudaStream_t st) {
  if (queue_pays(MORSE, ONE, persistent, b.n, ctx.sm_count))
    return launch32_persistent<MORSE, ONE>(sf, shapes, ip, b, ctx, st);
  const unsigned grid = (unsigned)((b.n + 127) / 128);
  k_integrate32_plain<MORSE, ONE><<<grid, 128, 0, st>>>(sf, shapes, ip, b, ctx.counters);
  return cudaGetLastError();
}

}  // namespace

bool integrate32_queue(bool all_morse, bool one, int persistent, int64_t n, int sm_count) {
  return queue_pays(all_morse, one, persistent, n, sm_count);
}

cudaError_t launch_integrate32(const SysSet& sys, const DevShape* shapes, const IntegParams& ip,
                               const DevBatch& b, int persistent, Ctx& ctx, cudaStream_t st,
                               bool all_morse) {
  const SysSetF sf = to_float(sys);
  const bool one = sys.n == 1;
  if (all_morse)
    return one ? launch32<true, true>(sf, shapes, ip, b, persistent, ctx, st)
               : launch32<true, false>(sf, shapes, ip, b, persistent, ctx, st);
  return one ? launch32<false, true>(sf, shapes, ip, b, persistent, ctx, st)
             : launch32<false, false>(sf, shapes, ip, b, persistent, ctx, st);
}

}  // namespace qcams
