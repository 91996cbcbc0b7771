// The pair-force factor u = V'(r)/r of one pair at squared distance s, as
// the FP64 integrators form it (Sec. 3.2 potentials): the reciprocal square
// root and the exponential of elem64.cuh, 10 FP64 instructions for a Morse
// pair.  Shared by the one-thread-per-trajectory and the lane-group
// integrators.
#pragma once

#include <cuda_runtime.h>

#include "qcams_device.cuh"
#include "elem64.cuh"

namespace qcams {
namespace {

// u of a Lennard-Jones pair with any exponents.  The difference's fused
// product is written out: left to the compiler it is the other one in some
// kernels, and the one-thread and lane-group forms would differ in the last
// bit.
template <class OP>
__device__ __forceinline__ double lj_u(const DevPair& q, double ri, const OP& op) {
  return op.mul(fma(-q.c2, ipow(ri, q.m), op.mul(q.c3, ipow(ri, q.n))), op.mul(ri, ri));
}

// The exponents' arguments take alpha r as (alpha s) (1/sqrt(s)): alpha s
// is formed while the reciprocal square root is refined, so the argument
// is one FP64 instruction after it instead of two (the same instruction
// count as forming r = s / sqrt(s) first).
template <bool MORSE, class OP>
__device__ __forceinline__ double pair_u(const DevPair& q, double s, const double* __restrict__ T,
                                         const OP& op) {
  float rf;   // FP32 estimate of r, for the exponential's table index
  const double ri = rsqrt_seeded(s, rf, op);
  if (MORSE) {
    // u = x (1 - x) / r, x = e^{-alpha (r - re)}; the factor 2 alpha De is in kf_morse
    const double as = op.mul(q.c0, s);
    const double x = texp_hint(fma(-as, ri, q.c1), fmaf(-q.ef0, rf, q.ef1), T, op);
    return op.mul(fma(-x, x, x), ri);
  }
  // generic kernels (mixed systems): u = V'(r)/r with the table exponential
  if (q.kind == QCAMS_MORSE) {
    const double as = op.mul(q.c0, s), c2ri = op.mul(q.c2, ri);
    const double x = texp_hint(fma(-as, ri, q.c1), fmaf(-q.ef0, rf, q.ef1), T, op);
    return op.mul(fma(-x, x, x), c2ri);
  }
  if (q.kind == QCAMS_BUCK) {
    // u = 6 C6 / r^8 - A B e^{-B r} / r, the exponential taking A B as the
    // offset ln(A B) of its argument: 9 FP64 instructions
    const double ri2 = op.mul(ri, ri), ri4 = op.mul(ri2, ri2), bs = op.mul(q.c1, s);
    const double ex = texp_hint(fma(-bs, ri, q.lc2), fmaf(-q.ef0, rf, q.ef1), T, op);
    return fma(q.c3, op.mul(ri4, ri4), -op.mul(ex, ri));
  }
  if (q.kind == QCAMS_LJ && q.n == 6 && (q.m == 12 || q.m == 8)) {
    // pot_g's form for these exponents
    const double ri2 = op.mul(ri, ri), ri4 = op.mul(ri2, ri2), ri6 = op.mul(ri4, ri2);
    const double h = q.m == 12 ? ri6 : ri4;
    return op.mul(fma(q.c3, ri6, -op.mul(q.c2, op.mul(h, h))), ri2);
  }
  return lj_u(q, ri, op);
}

}  // namespace
}  // namespace qcams
