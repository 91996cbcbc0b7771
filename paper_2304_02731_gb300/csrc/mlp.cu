// Learned importance-sampling proposal: a small MLP trained on the method's
// own (initial condition -> outcome) data, turned into a defensive-mixture
// proposal over (b^2, cos theta, phi, eta, chi) whose likelihood-ratio
// weights keep the cross-section estimator unbiased (every sampled
// trajectory is still integrated exactly).
//
// Tensor-core design (sm_103a, warp-level mma.sync m16n8k16, BF16 inputs,
// FP32 accumulation): each warp carries 16 samples through the network.  The
// accumulator fragment of two adjacent 16x8 output tiles has exactly the
// register layout of the A operand of a 16x16 slice, so a layer's SiLU output
// is fed to the next layer's products without touching shared memory.  The
// backward pass reuses the same fragments: dA = dZ W reads the weight tiles
// of the forward pass transposed (ldmatrix.trans).  Training leaves each block
// round's transposed activations and errors in shared tiles; the weight
// gradients dW = dZ^T A are then block GEMMs over the round's samples (K = 64
// or 128), accumulated in registers and added to the global gradient once per
// round.
//
// The network is ~9k multiply-adds per sample: negligible next to the
// trajectory integration, so a warp-level mma kernel is enough here.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "qcams.h"
#include "qcams_device.cuh"

namespace qcams {
namespace {

constexpr int IN = 8, H = 64, OUT = 4, NP = QCAMS_MLP_NPARAMS;
constexpr int OW1 = 0, OB1 = OW1 + H * IN, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H,
              OB3 = OW3 + H * H, OW4 = OB3 + H, OB4 = OW4 + OUT * H;
static_assert(OB4 + OUT == NP, "parameter layout");
static_assert(OW1 % 4 == 0 && OW2 % 4 == 0 && OW3 % 4 == 0 && OW4 % 4 == 0 && IN % 4 == 0,
              "weight-gradient quads are 16-byte aligned");
constexpr int WARPS = 4, THREADS = WARPS * 32;
constexpr double kPi = 3.14159265358979323846;

struct Std {
  float mean[8], inv_std[8];
};

// Shared-memory weight tiles (BF16), W as [N][K]: the forward pass takes its
// B operands from rows of W (ldmatrix), the backward pass dA = dZ W the same
// tiles transposed (ldmatrix.trans).  Padding: W1 K 8 -> 16, W4 N 4 -> 8.
// Every row is padded by 8 elements (16 B): the 8 row segments of 16 bytes
// that a matrix load touches lie on 32 distinct banks.
constexpr int PK = 8;   // row padding (BF16 elements)
struct alignas(16) WeightsSmem {   // 16-byte row-segment stores
  __nv_bfloat16 w1[H][16 + PK];
  __nv_bfloat16 w2[H][H + PK];
  __nv_bfloat16 w3[H][H + PK];
  __nv_bfloat16 w4[8][H + PK];
  float b1[H], b2[H], b3[H], b4[8];
};
// Training works in block rounds of RS = 64 CPW samples (4 warps x CPW
// chunks of 16).  Each chunk's forward and backward pass leave, in
// block-wide shared tiles, the transposed inputs, activations and
// back-propagated errors of its 16 samples (BF16, [unit][sample]); after the
// round each warp forms 16 rows of every weight gradient dW = dZ^T A as an
// MMA product over the round's samples, accumulated in registers and added
// to the global gradient once.  Rows are padded by 8 elements for the
// matrix loads and stores, as the weights' are.
template <int CPW>
struct alignas(16) BlockTiles {
  static constexpr int RS = 16 * WARPS * CPW;   // samples per block round
  static constexpr int LDT = RS + PK;           // row stride (BF16 elements)
  __nv_bfloat16 xt[16][LDT];         // X^T  [feature (padded to 16)][sample]
  __nv_bfloat16 at[3][H][LDT];       // A1^T, A2^T, A3^T [unit][sample]
  __nv_bfloat16 dzt[3][H][LDT];      // dZ1^T, dZ2^T, dZ3^T [unit][sample]
  __nv_bfloat16 dz4t[16][LDT];       // dZ4^T [output (padded to 16)][sample]
};
// Bias gradients of the block (b1, b2, b3, b4), FP32 sums of the FP32 dZ
// fragments.
constexpr int GB1 = 0, NGB = 3 * H + OUT;
template <int CPW>
struct TrainSmem {
  WeightsSmem w;
  float gb[NGB];
  BlockTiles<CPW> t;
};

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
// D += A B for one m16n8k16 tile (BF16 in, FP32 accumulate).
__device__ __forceinline__ void mma(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four 8 x 8 BF16 matrices from shared memory, lane l giving the address of
// row l mod 8 of matrix l / 8 (16 bytes, 16-byte aligned); TRANS: each one
// transposed.  Lane (g, q) receives elements (g, 2q), (g, 2q + 1).
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t* r, const __nv_bfloat16* row) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(row);
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
// The reverse, transposed: four (two) fragments to rows of their columns.
__device__ __forceinline__ void stsm4t(__nv_bfloat16* row, const uint32_t* r) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(row)),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void stsm2t(__nv_bfloat16* row, uint32_t r0, uint32_t r1) {
  asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(row)),
               "r"(r0), "r"(r1) : "memory");
}
// A 16-sample, 64-unit tile in A-fragment order (a[s]: units 16 s ..) to the
// rows of dst ([unit][sample]) at sample columns col .. col + 15.
template <int LDT>
__device__ __forceinline__ void store_units(__nv_bfloat16 (*dst)[LDT], int col,
                                            const uint32_t (*a)[4]) {
  const int l = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < 4; ++s)
    stsm4t(&dst[16 * s + 8 * (l >> 4) + (l & 7)][col + 8 * ((l >> 3) & 1)], a[s]);
}
// An 8-unit tile (fragments of samples 0-7 and 8-15) likewise.
template <int LDT>
__device__ __forceinline__ void store_tile8(__nv_bfloat16 (*dst)[LDT], int col, uint32_t r0,
                                            uint32_t r1) {
  const int l = threadIdx.x & 15;
  stsm2t(&dst[l & 7][col + 8 * (l >> 3)], r0, r1);
}

// Logistic function: __expf and the fast divide (a few ulp; the products it
// feeds are rounded to BF16).  For z below about -87 the quotient is 0.
__device__ __forceinline__ float sigm(float z) { return __fdividef(1.0f, 1.0f + __expf(-z)); }

// Weights to shared memory (blockDim.x == THREADS).  With p 16-byte aligned
// every matrix starts on a 16-byte boundary: each thread issues all of its
// 16-byte loads of 8-element row segments first, then stores each segment
// to its row.  Otherwise, element loads.
__device__ void load_weights(WeightsSmem& W, const __nv_bfloat16* p, const float* pf) {
  const __nv_bfloat16 zero = __float2bfloat16(0.0f);
  if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
    constexpr int N1 = H * IN / 8, N2 = H * H / 8, N4 = OUT * H / 8;
    constexpr int NSEG = N1 + 2 * N2 + N4, PER = (NSEG + THREADS - 1) / THREADS;
    static_assert(IN == 8 && (OW2 % 8) == 0 && (OW3 % 8) == 0 && (OW4 % 8) == 0,
                  "16-byte row segments");
    uint4 v[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int i = threadIdx.x + k * THREADS;
      int off = 0;
      if (i < N1) off = OW1 + 8 * i;
      else if (i < N1 + N2) off = OW2 + 8 * (i - N1);
      else if (i < N1 + 2 * N2) off = OW3 + 8 * (i - N1 - N2);
      else if (i < NSEG) off = OW4 + 8 * (i - N1 - 2 * N2);
      if (i < NSEG) v[k] = *reinterpret_cast<const uint4*>(p + off);
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int i = threadIdx.x + k * THREADS;
      if (i >= NSEG) continue;
      if (i < N1) {
        *reinterpret_cast<uint4*>(&W.w1[i][0]) = v[k];
        *reinterpret_cast<uint4*>(&W.w1[i][8]) = make_uint4(0u, 0u, 0u, 0u);
        continue;
      }
      const bool is4 = i >= N1 + 2 * N2;
      const int j = i < N1 + N2 ? i - N1 : i < N1 + 2 * N2 ? i - N1 - N2 : i - N1 - 2 * N2;
      const int r = j / (H / 8), c = 8 * (j % (H / 8));
      __nv_bfloat16* row = is4 ? &W.w4[r][c] : i < N1 + N2 ? &W.w2[r][c] : &W.w3[r][c];
      *reinterpret_cast<uint4*>(row) = v[k];
    }
    for (int i = threadIdx.x; i < (8 - OUT) * H; i += blockDim.x) W.w4[OUT + i / H][i % H] = zero;
  } else {
    for (int i = threadIdx.x; i < H * 16; i += blockDim.x) {
      const int r = i / 16, c = i % 16;
      W.w1[r][c] = c < IN ? p[OW1 + r * IN + c] : zero;
    }
    for (int i = threadIdx.x; i < H * H; i += blockDim.x) {
      const int r = i / H, c = i % H;
      W.w2[r][c] = p[OW2 + i];
      W.w3[r][c] = p[OW3 + i];
    }
    for (int i = threadIdx.x; i < 8 * H; i += blockDim.x) {
      const int r = i / H, c = i % H;
      W.w4[r][c] = r < OUT ? p[OW4 + r * H + c] : zero;
    }
  }
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    W.b1[i] = pf[OB1 + i];
    W.b2[i] = pf[OB2 + i];
    W.b3[i] = pf[OB3 + i];
  }
  if (threadIdx.x < 8) W.b4[threadIdx.x] = threadIdx.x < OUT ? pf[OB4 + threadIdx.x] : 0.0f;
}

// Features of the 16 rows handled by this lane's fragment rows: either from
// x[n][8] or (proposal mode) from the centre of grid cell `row`.
struct CellGrid {
  int n_b2, n_cth, n_phi, n_eta, n_chi;
  float E, v, j, b2_max;
};
// Minibatch rows: row i is a uniform one of `n` samples, from Philox4x32-10
// with key = seed and counter (i, step_lo, step_hi, 4); the 64-bit word w1:w0
// is mapped by the high half of w * n (bias <= n / 2^64).
struct RowSrc {
  int64_t n;
  uint64_t seed, step;
  __device__ __forceinline__ int64_t at(int64_t i) const {
    const uint4 w = philox4x32_10(
        make_uint4((uint32_t)i, (uint32_t)step, (uint32_t)(step >> 32), 4u),
        make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    const unsigned long long u = ((unsigned long long)w.y << 32) | w.x;
    return (int64_t)__umul64hi(u, (unsigned long long)n);
  }
};
__device__ __forceinline__ void features(const float* x, int64_t src, int64_t n,
                                         int64_t row, const CellGrid* grid, float* f) {
  if (row >= n) {
#pragma unroll
    for (int k = 0; k < IN; ++k) f[k] = 0.0f;
    return;
  }
  if (!grid) {
#pragma unroll
    for (int k = 0; k < IN; ++k) f[k] = x[src * IN + k];
    return;
  }
  int64_t c = row;
  const int i_chi = (int)(c % grid->n_chi); c /= grid->n_chi;
  const int i_eta = (int)(c % grid->n_eta); c /= grid->n_eta;
  const int i_phi = (int)(c % grid->n_phi); c /= grid->n_phi;
  const int i_cth = (int)(c % grid->n_cth); c /= grid->n_cth;
  const int i_b2 = (int)c;
  f[0] = grid->E;
  f[1] = sqrtf(grid->b2_max * (i_b2 + 0.5f) / grid->n_b2);
  f[2] = grid->v;
  f[3] = grid->j;
  f[4] = acosf(2.0f * (i_cth + 0.5f) / grid->n_cth - 1.0f);
  f[5] = 2.0f * (float)kPi * (i_phi + 0.5f) / grid->n_phi;
  f[6] = (i_chi + 0.5f) / grid->n_chi;
  f[7] = 2.0f * (float)kPi * (i_eta + 0.5f) / grid->n_eta;
}

// Forward pass of 16 samples (rows base .. base+15) by one warp; this lane's
// rows base + g and base + g + 8 are samples src0 and src1.  Returns the
// logits fragment (rows g and g+8, columns 2q, 2q+1 of the padded 16x8 tile).
// With TRAIN, ds receives SiLU'(Z) of layers 1-3 (accumulator order) and the
// transposed inputs and activations go to the block tiles T, at sample
// columns col .. col + 15, for the backward pass.
template <bool TRAIN, int CPW>
__device__ __forceinline__ void forward16(const WeightsSmem& W, float (*ds)[32], BlockTiles<CPW>* T,
                                          int col, const float* x, int64_t src0, int64_t src1,
                                          int64_t n, int64_t base, const CellGrid* grid,
                                          const Std& sd, float* logit) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  // this lane's row of two adjacent 8-unit tiles in a matrix load
  const int wrow = 8 * (lane >> 4) + (lane & 7), wcol = 8 * ((lane >> 3) & 1);
  float f0[IN], f1[IN];
  features(x, src0, n, base + g, grid, f0);
  features(x, src1, n, base + g + 8, grid, f1);
#pragma unroll
  for (int k = 0; k < IN; ++k) {
    f0[k] = (f0[k] - sd.mean[k]) * sd.inv_std[k];
    f1[k] = (f1[k] - sd.mean[k]) * sd.inv_std[k];
    if (base + g >= n) f0[k] = 0.0f;
    if (base + g + 8 >= n) f1[k] = 0.0f;
  }
  // features 2q, 2q + 1 by selects (no dynamic register indexing)
  auto pick = [&](const float* f, int e) {
    return q == 0 ? f[e] : q == 1 ? f[2 + e] : q == 2 ? f[4 + e] : f[6 + e];
  };
  uint32_t a[4][4];  // A fragments of the current layer input (up to 4 k-slices)
  a[0][0] = pack2(pick(f0, 0), pick(f0, 1));
  a[0][1] = pack2(pick(f1, 0), pick(f1, 1));
  a[0][2] = 0u;
  a[0][3] = 0u;
  if (TRAIN) store_tile8(T->xt, col, a[0][0], a[0][1]);
#pragma unroll
  for (int layer = 0; layer < 3; ++layer) {
    const float* bias = layer == 0 ? W.b1 : layer == 1 ? W.b2 : W.b3;
    float c[8][4];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const float2 b = *reinterpret_cast<const float2*>(&bias[8 * t + 2 * q]);
      c[t][0] = c[t][2] = b.x;
      c[t][1] = c[t][3] = b.y;
    }
    // k-slices outside: eight independent accumulators in flight
#pragma unroll
    for (int s = 0; s < (layer == 0 ? 1 : 4); ++s) {
#pragma unroll
      for (int t = 0; t < 8; t += 2) {
        uint32_t b[4];
        ldsm4<false>(b, layer == 0   ? &W.w1[8 * t + wrow][wcol]
                        : layer == 1 ? &W.w2[8 * t + wrow][16 * s + wcol]
                                     : &W.w3[8 * t + wrow][16 * s + wcol]);
        mma(c[t], a[s], b[0], b[1]);
        mma(c[t + 1], a[s], b[2], b[3]);
      }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      // SiLU of tiles 2s (units 16s + 2q, +1) and 2s + 1 (units 16s + 8 + 2q,
      // +1), rows g and g + 8; with TRAIN also SiLU'(z) = sg (1 + z (1 - sg))
      float v[8];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float z = c[2 * s + h][e], sg = sigm(z);
          v[4 * h + e] = z * sg;
          if (TRAIN) ds[layer][4 * (2 * s + h) + e] = sg * (1.0f + z * (1.0f - sg));
        }
      a[s][0] = pack2(v[0], v[1]);
      a[s][1] = pack2(v[2], v[3]);
      a[s][2] = pack2(v[4], v[5]);
      a[s][3] = pack2(v[6], v[7]);
    }
    if (TRAIN) store_units(T->at[layer], col, a);
  }
  logit[0] = logit[2] = W.b4[2 * q];
  logit[1] = logit[3] = W.b4[2 * q + 1];
#pragma unroll
  for (int s = 0; s < 4; s += 2) {
    uint32_t b[4];   // W4's one tile: k-slices s and s + 1
    ldsm4<false>(b, &W.w4[lane & 7][16 * s + 8 * (lane >> 3)]);
    mma(logit, a[s], b[0], b[1]);
    mma(logit, a[s + 1], b[2], b[3]);
  }
}

// Softmax over the 4 logits of one row held by lanes q = 0 (columns 0, 1)
// and q = 1 (columns 2, 3); returns this lane's two probabilities.
__device__ __forceinline__ void softmax_pair(float z0, float z1, float* p0, float* p1) {
  const float o0 = __shfl_xor_sync(0xffffffffu, z0, 1);
  const float o1 = __shfl_xor_sync(0xffffffffu, z1, 1);
  const float m = fmaxf(fmaxf(z0, z1), fmaxf(o0, o1));
  const float e0 = __expf(z0 - m), e1 = __expf(z1 - m);
  const float s = e0 + e1 + __expf(o0 - m) + __expf(o1 - m);
  *p0 = e0 / s;
  *p1 = e1 / s;
}

// One warp's 16 rows m0 .. m0+15 of dW = dZ^T A over the round's RS samples,
// for the NT 8-column tiles from column n0: A operand from dZ^T (rows
// = output units, samples contiguous), B operand from A^T (rows = input
// units, samples contiguous: the col layout of B), FP32 accumulation in
// registers; added once to the global gradient gW (row-major, n_in columns)
// for rows < n_out and columns < n_in.
template <int NT, int LDT>
__device__ __forceinline__ void block_dw(const __nv_bfloat16 (*dzt)[LDT],
                                         const __nv_bfloat16 (*at)[LDT], int m0, int n0, int n_out,
                                         int n_in, float* gW) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const bool vec4 = (reinterpret_cast<uintptr_t>(gW) & 15u) == 0;
  float d[NT][4];
#pragma unroll
  for (int t = 0; t < NT; ++t) d[t][0] = d[t][1] = d[t][2] = d[t][3] = 0.0f;
#pragma unroll
  for (int ks = 0; ks < (LDT - PK) / 16; ++ks) {
    uint32_t a[4];
    ldsm4<false>(a, &dzt[m0 + 8 * ((lane >> 3) & 1) + (lane & 7)][16 * ks + 8 * (lane >> 4)]);
#pragma unroll
    for (int t = 0; t < NT; t += 2) {   // (one tile: the second is the tile's zero padding)
      uint32_t b[4];
      ldsm4<false>(b, &at[n0 + 8 * t + 8 * (lane >> 4) + (lane & 7)]
                         [16 * ks + 8 * ((lane >> 3) & 1)]);
      mma(d[t], a, b[0], b[1]);
      if (t + 1 < NT) mma(d[t + 1], a, b[2], b[3]);
    }
  }
  // Lanes q and q ^ 1 hold columns 2q, 2q + 1 of rows g and g + 8: the even
  // one takes both lanes' share of row g, the odd one of row g + 8, four
  // consecutive columns each (vector atomics, sm_90 and later; n_in is a
  // multiple of 4 and the parameter offsets are too).
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    const bool odd = q & 1;
    const float s0 = odd ? d[t][0] : d[t][2], s1 = odd ? d[t][1] : d[t][3];
    const float o0 = __shfl_xor_sync(0xffffffffu, s0, 1), o1 = __shfl_xor_sync(0xffffffffu, s1, 1);
    const float4 v = odd ? make_float4(o0, o1, d[t][2], d[t][3])
                         : make_float4(d[t][0], d[t][1], o0, o1);
    const int r = m0 + g + (odd ? 8 : 0), c = n0 + 8 * t + 2 * (q & 2);
    if (c < n_in && r < n_out) {
      float* at = &gW[r * n_in + c];
      if (vec4) {
        atomicAdd(reinterpret_cast<float4*>(at), v);
      } else {   // a gradient buffer that is not 16-byte aligned
        atomicAdd(at, v.x);
        atomicAdd(at + 1, v.y);
        atomicAdd(at + 2, v.z);
        atomicAdd(at + 3, v.w);
      }
    }
  }
}

// Bias gradients of a 64-unit layer: the sums over the 16 samples of dZ's
// columns, added to gb.  A column's order of sums is that of a butterfly over
// the eight row lanes: rows g and g + 8, then lanes g ^ 1, g ^ 2 and g ^ 4.
// The 16 columns of a lane quad take those three steps by halving (14
// shuffles where butterflies take 48), which leaves lane (g, q) with columns
// 8 r + 2 q and + 1, r being g with its three bits reversed.
__device__ __forceinline__ void accumulate_db(const float (*dz)[4], float* gb) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  float s[8][2];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    s[t][0] = dz[t][0] + dz[t][2];
    s[t][1] = dz[t][1] + dz[t][3];
  }
#pragma unroll
  for (int bit = 1, half = 4; half > 0; bit <<= 1, half >>= 1) {
    const bool up = g & bit;
#pragma unroll
    for (int t = 0; t < half; ++t)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float send = up ? s[t][e] : s[t + half][e], keep = up ? s[t + half][e] : s[t][e];
        s[t][e] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * bit);
      }
  }
  const int r = (g & 1) << 2 | (g & 2) | g >> 2;
  atomicAdd(&gb[8 * r + 2 * q], s[0][0]);
  atomicAdd(&gb[8 * r + 2 * q + 1], s[0][1]);
}
// The same for the 4 outputs (columns 0-3 of one tile).
__device__ __forceinline__ void accumulate_db4(const float* dz, float* gb) {
  const int lane = threadIdx.x & 31;
  float s0 = dz[0] + dz[2], s1 = dz[1] + dz[3];
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
  }
  if (lane < 2) {
    atomicAdd(&gb[2 * lane], s0);
    atomicAdd(&gb[2 * lane + 1], s1);
  }
}

// Gradient of the mean cross-entropy over n rows: samples 0 .. n - 1 or, with
// DRAW, the minibatch rows.at(0 .. n - 1).  Block rounds of RS samples: each
// warp carries its chunks of 16 through the forward and backward passes
// (activations and errors to the block tiles, bias gradients to shared FP32
// sums), then the four weight gradients of the round are formed as block
// GEMMs (warp w: rows 16w .. 16w+15 of dW1..dW3, columns 16w .. 16w+15 of
// dW4) and added to the global gradient.
template <int CPW, bool DRAW>
__global__ void __launch_bounds__(THREADS) k_mlp_grad(const __nv_bfloat16* pb, const float* pf,
                                                      Std sd, const float* x,
                                                      const uint8_t* label, RowSrc rows,
                                                      int64_t n, float* grad, float* loss) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem<CPW>& S = *reinterpret_cast<TrainSmem<CPW>*>(smem_raw);
  constexpr int RS = BlockTiles<CPW>::RS, LDT = BlockTiles<CPW>::LDT;
  load_weights(S.w, pb, pf);
  for (int i = threadIdx.x; i < NGB; i += blockDim.x) S.gb[i] = 0.0f;
  // padding rows of the X^T and dZ4^T tiles (never written by the passes)
  const __nv_bfloat16 zero = __float2bfloat16(0.0f);
  for (int i = threadIdx.x; i < (16 - IN) * LDT; i += blockDim.x) S.t.xt[IN + i / LDT][i % LDT] = zero;
  for (int i = threadIdx.x; i < (16 - 8) * LDT; i += blockDim.x) S.t.dz4t[8 + i / LDT][i % LDT] = zero;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const float inv_n = 1.0f / (float)n;
  float loss_acc = 0.0f;
  const int64_t rounds = (n + RS - 1) / RS;
  for (int64_t rnd = blockIdx.x; rnd < rounds; rnd += gridDim.x) {
    for (int c = 0; c < CPW; ++c) {
      const int col = 16 * (WARPS * c + warp);
      const int64_t base = rnd * RS + col;
      float lg[4], ds[3][32];
      const int64_t r0 = base + g, r1 = base + g + 8;
      const int64_t s0 = DRAW ? rows.at(r0) : r0, s1 = DRAW ? rows.at(r1) : r1;
      forward16<true, CPW>(S.w, ds, &S.t, col, x, s0, s1, n, base, nullptr, sd, lg);
      // softmax cross-entropy and dZ4 = (p - onehot) / n; rows past n and
      // rows without a target have dZ4 = 0 and so add nothing below
      float dz4[1][4] = {{0.f, 0.f, 0.f, 0.f}};
      float p[4];
      softmax_pair(lg[0], lg[1], &p[0], &p[1]);
      softmax_pair(lg[2], lg[3], &p[2], &p[3]);
      if (q < 2) {
        int l0 = r0 < n ? (int)label[s0] : -1;
        int l1 = r1 < n ? (int)label[s1] : -1;
        if (l0 >= OUT) l0 = -1;   // AMBIG / FAIL lanes carry no target
        if (l1 >= OUT) l1 = -1;
        for (int e = 0; e < 2; ++e) {
          const int k = 2 * q + e;
          if (l0 >= 0) {
            dz4[0][e] = (p[e] - (k == l0 ? 1.0f : 0.0f)) * inv_n;
            if (k == l0) loss_acc -= __logf(fmaxf(p[e], 1e-30f)) * inv_n;
          }
          if (l1 >= 0) {
            dz4[0][2 + e] = (p[2 + e] - (k == l1 ? 1.0f : 0.0f)) * inv_n;
            if (k == l1) loss_acc -= __logf(fmaxf(p[2 + e], 1e-30f)) * inv_n;
          }
        }
      }
      accumulate_db4(dz4[0], &S.gb[3 * H]);
      // dA3 = dZ4 W4: A operand from the dZ4 fragment (K padded 8 -> 16)
      uint32_t a[4][4];
      a[0][0] = pack2(dz4[0][0], dz4[0][1]);
      a[0][1] = pack2(dz4[0][2], dz4[0][3]);
      a[0][2] = 0u;
      a[0][3] = 0u;
      store_tile8(S.t.dz4t, col, a[0][0], a[0][1]);
#pragma unroll
      for (int layer = 2; layer >= 0; --layer) {
        float dz[8][4];
#pragma unroll
        for (int t = 0; t < 8; ++t) dz[t][0] = dz[t][1] = dz[t][2] = dz[t][3] = 0.0f;
        if (layer == 2) {
#pragma unroll
          for (int t = 0; t < 8; t += 4) {
            uint32_t b[4];   // rows = outputs: tiles t .. t + 3, upper half of K zero
            ldsm4<true>(b, &S.w.w4[lane & 7][8 * (t + (lane >> 3))]);
#pragma unroll
            for (int k = 0; k < 4; ++k) mma(dz[t + k], a[0], b[k], 0u);
          }
        } else {
          const __nv_bfloat16 (*w)[H + PK] = layer == 1 ? S.w.w3 : S.w.w2;
#pragma unroll
          for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int t = 0; t < 8; t += 2) {
              uint32_t b[4];
              ldsm4<true>(b, &w[16 * s + 8 * ((lane >> 3) & 1) + (lane & 7)][8 * t + 8 * (lane >> 4)]);
              mma(dz[t], a[s], b[0], b[1]);
              mma(dz[t + 1], a[s], b[2], b[3]);
            }
        }
        // dZ = dA * SiLU'(Z)
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) dz[t][e] *= ds[layer][4 * t + e];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          a[s][0] = pack2(dz[2 * s][0], dz[2 * s][1]);
          a[s][1] = pack2(dz[2 * s][2], dz[2 * s][3]);
          a[s][2] = pack2(dz[2 * s + 1][0], dz[2 * s + 1][1]);
          a[s][3] = pack2(dz[2 * s + 1][2], dz[2 * s + 1][3]);
        }
        store_units(S.t.dzt[layer], col, a);
        accumulate_db(dz, &S.gb[GB1 + H * layer]);
      }
    }
    __syncthreads();   // the round's tiles are complete
    const int m0 = 16 * warp;
    block_dw<1>(S.t.dzt[0], S.t.xt, m0, 0, H, IN, grad + OW1);
    block_dw<8>(S.t.dzt[1], S.t.at[0], m0, 0, H, H, grad + OW2);
    block_dw<8>(S.t.dzt[2], S.t.at[1], m0, 0, H, H, grad + OW3);
    block_dw<2>(S.t.dz4t, S.t.at[2], 0, m0, OUT, H, grad + OW4);
    __syncthreads();   // tiles are rewritten by the next round
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
  if (lane == 0 && loss) atomicAdd(loss, loss_acc);
  for (int i = threadIdx.x; i < NGB; i += blockDim.x) {
    const int k = i < 3 * H ? (i / H == 0 ? OB1 : i / H == 1 ? OB2 : OB3) + i % H : OB4 + (i - 3 * H);
    if (S.gb[i] != 0.0f) atomicAdd(&grad[k], S.gb[i]);
  }
}

__global__ void __launch_bounds__(THREADS) k_mlp_infer(const __nv_bfloat16* pb, const float* pf,
                                                       Std sd, const float* x, int64_t n,
                                                       CellGrid grid, int use_grid,
                                                       float* probs, double* g_out,
                                                       double eps) {
  __shared__ WeightsSmem W;
  load_weights(W, pb, pf);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const int64_t chunks = (n + 15) / 16;
  for (int64_t ch = (int64_t)blockIdx.x * WARPS + warp; ch < chunks;
       ch += (int64_t)gridDim.x * WARPS) {
    const int64_t base = ch * 16;
    float lg[4], p[4];
    forward16<false, 1>(W, nullptr, nullptr, 0, x, base + g, base + g + 8, n, base,
                        use_grid ? &grid : nullptr, sd, lg);
    softmax_pair(lg[0], lg[1], &p[0], &p[1]);
    softmax_pair(lg[2], lg[3], &p[2], &p[3]);
    const int64_t r0 = base + g, r1 = base + g + 8;
    if (probs && q < 2) {
      if (r0 < n) { probs[r0 * 4 + 2 * q] = p[0]; probs[r0 * 4 + 2 * q + 1] = p[1]; }
      if (r1 < n) { probs[r1 * 4 + 2 * q] = p[2]; probs[r1 * 4 + 2 * q + 1] = p[3]; }
    }
    if (g_out) {
      // p_R = P(R_AC) + P(R_BC): columns 1 (lane q = 0) and 2 (lane q = 1)
      const float mine0 = q == 0 ? p[1] : p[0], mine1 = q == 0 ? p[3] : p[2];
      const float other0 = __shfl_xor_sync(0xffffffffu, mine0, 1);
      const float other1 = __shfl_xor_sync(0xffffffffu, mine1, 1);
      if (q == 0) {
        if (r0 < n) g_out[r0] = sqrt(eps + (double)mine0 + (double)other0);
        if (r1 < n) g_out[r1] = sqrt(eps + (double)mine1 + (double)other1);
      }
    }
  }
}

// Adam step (beta1 0.9, beta2 0.999, eps 1e-8; c1, c2 the bias corrections).
// With clear, the gradient is zeroed for the next training step.
__global__ void k_adam(float* p, float* m, float* v, float* grad, __nv_bfloat16* pb, float lr,
                       float c1, float c2, bool clear) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NP; i += gridDim.x * blockDim.x) {
    const float gr = grad[i];
    const float mi = 0.9f * m[i] + 0.1f * gr;
    const float vi = 0.999f * v[i] + 0.001f * gr * gr;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    p[i] = pi;
    pb[i] = __float2bfloat16(pi);
    if (clear) grad[i] = 0.0f;
  }
}

// The rows of training step `step` (RowSrc).
__global__ void k_draw_idx(int64_t* idx, int batch, RowSrc rows) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < batch) idx[i] = rows.at(i);
}

__global__ void k_mlp_init(float* p, float* m, float* v, __nv_bfloat16* pb, uint64_t seed) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NP; i += gridDim.x * blockDim.x) {
    float fan_in = 0.0f;
    if (i < OB1) fan_in = IN;
    else if (i >= OW2 && i < OB2) fan_in = H;
    else if (i >= OW3 && i < OB3) fan_in = H;
    else if (i >= OW4 && i < OB4) fan_in = H;
    float val = 0.0f;
    if (fan_in > 0.0f) {
      const uint4 w = philox4x32_10(make_uint4((uint32_t)i, 0u, 3u, 0u),
                                    make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
      const float u = (float)u01(w.x);
      val = (2.0f * u - 1.0f) * rsqrtf(fan_in);
    }
    p[i] = val;
    m[i] = 0.0f;
    v[i] = 0.0f;
    pb[i] = __float2bfloat16(val);
  }
}

__global__ void k_mlp_sync(const float* p, __nv_bfloat16* pb) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NP; i += gridDim.x * blockDim.x)
    pb[i] = __float2bfloat16(p[i]);
}

__global__ void k_features(int64_t n, const double* E, const double* b, const int32_t* v,
                           const int32_t* j, const double* u0, const double* u1,
                           const double* u2, const double* u3, float* x) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  x[i * 8 + 0] = (float)E[i];
  x[i * 8 + 1] = (float)b[i];
  x[i * 8 + 2] = (float)v[i];
  x[i * 8 + 3] = (float)j[i];
  x[i * 8 + 4] = (float)acos(fmin(1.0, fmax(-1.0, 2.0 * u0[i] - 1.0)));
  x[i * 8 + 5] = (float)(2.0 * kPi * u1[i]);
  x[i * 8 + 6] = (float)u3[i];
  x[i * 8 + 7] = (float)(2.0 * kPi * u2[i]);
}

// Sums and sums of squares of the 8 columns of x, in FP64: thread t takes
// the elements t, t + (grid size), .. of the flat array, all of column t mod
// 8, so loads are coalesced and a thread has two sums.  Bound by the FP64
// pipe, two instructions an element (the conversion runs on the integer
// pipe).  1 M rows: 157 us with 16 sums and shared atomics per thread, now
// 51 us.
constexpr int kMomentsBlock = 512;
__global__ void __launch_bounds__(kMomentsBlock) k_moments(const float* x, int64_t n, double* acc) {
  __shared__ double s[kMomentsBlock / 32][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double a = 0.0, b = 0.0;
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)kMomentsBlock + threadIdx.x; i < 8 * n;
       i += (int64_t)gridDim.x * kMomentsBlock) {
    const float f = x[i];
    const unsigned u = __float_as_uint(f), e = u & 0x7f800000u;
    // normal f on the integer pipe, the rest by a conversion
    const double v = e == 0u || e == 0x7f800000u
                         ? (double)f
                         : __hiloint2double((int)((u & 0x80000000u) |
                                                  (((u & 0x7fffffffu) >> 3) + (896u << 20))),
                                            (int)(u << 29));
    a += v;
    b = fma(v, v, b);
  }
#pragma unroll
  for (int o = 8; o < 32; o <<= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane < 8) {
    s[warp][lane] = a;
    s[warp][8 + lane] = b;
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    double t = 0.0;
    for (int w = 0; w < kMomentsBlock / 32; ++w) t += s[w][threadIdx.x];
    atomicAdd(&acc[threadIdx.x], t);
  }
}

// Normalisation of the proposal and its integer CDF, in a fixed summation
// order (deterministic bits): 1,024 runs of consecutive cells are summed cell
// by cell, the run sums by a halving tree.  q needs a correctly rounded FP64
// division per cell, about 20 instructions of the scarce FP64 pipe, so the
// work is spread over all SMs in four small kernels (one block of one SM took
// 180 us for 32,768 cells, 160 of them at the FP64 pipe's rate; now 20 us):
//   k_run_sums   run sums, staged through shared memory (coalesced)
//   k_normalise  total, q, qfix and each scan block's sum of qfix
//   k_scan_sums  exclusive prefixes of the block sums
//   k_cdf        inclusive scan within each block
// The intermediate values live in cdf until k_cdf overwrites it: the run
// sums (as doubles) in its first 1,024 entries, each scan block's sum and
// then prefix in the block's last entry.
constexpr int kRuns = 1024;
constexpr int kScanCells = 2048;   // cells per scan block
static_assert(kScanCells > kRuns, "a scan block's last entry lies beyond the run sums");
constexpr int kRunTile = 32;

__global__ void __launch_bounds__(32) k_run_sums(const double* g, int64_t n_cells, int64_t* cdf,
                                                 int scan_blocks) {
  __shared__ double tile[kRunTile][kRunTile + 1];
  const int lane = threadIdx.x;
  const int64_t per = (n_cells + kRuns - 1) / kRuns;
  const int64_t run0 = (int64_t)blockIdx.x * kRunTile;
  const int64_t lo = (run0 + lane) * per, hi = min(n_cells, lo + per);
  double sum = 0.0;
  for (int64_t c0 = 0; c0 < per; c0 += kRunTile) {
#pragma unroll 8
    for (int r = 0; r < kRunTile; ++r) {   // row r: cells c0 .. c0 + 31 of run run0 + r
      const int64_t c = (run0 + r) * per + c0 + lane;
      tile[r][lane] = c0 + lane < per && c < n_cells ? g[c] : 0.0;
    }
    __syncwarp();
    const int64_t last = min(per - c0, (int64_t)kRunTile);
    for (int k = 0; k < last; ++k)
      if (lo + c0 + k < hi) sum += tile[lane][k];
    __syncwarp();
  }
  // runs past the last cell are empty; only runs that exist have an entry
  if (lo < n_cells) cdf[run0 + lane] = __double_as_longlong(sum);
  if (scan_blocks > 1)   // clear the scan blocks' sums
    for (int64_t b = run0 + lane; b < scan_blocks; b += kRuns)
      cdf[min(n_cells, (b + 1) * kScanCells) - 1] = 0;
}

constexpr int kNormBlock = 256;   // small blocks: the divisions spread over the SMs
static_assert(kScanCells % kNormBlock == 0, "a block lies in one scan block");
__global__ void __launch_bounds__(kNormBlock) k_normalise(double* g, int64_t n_cells, double alpha,
                                                          int64_t* qfix, int64_t* cdf, bool sums) {
  __shared__ double ds[kRuns];
  const int t = threadIdx.x;
  const int64_t per = (n_cells + kRuns - 1) / kRuns;
  for (int r = t; r < kRuns; r += kNormBlock)
    ds[r] = r * per < n_cells ? __longlong_as_double(cdf[r]) : 0.0;
  __syncthreads();
  for (int o = kRuns / 2; o > 0; o >>= 1) {
    for (int r = t; r < o; r += kNormBlock) ds[r] += ds[r + o];
    __syncthreads();
  }
  const double total = ds[0];
  const int64_t c = (int64_t)blockIdx.x * kNormBlock + t;
  long long qi = 0;
  if (c < n_cells) {
    const double qc = alpha / (double)n_cells + (1.0 - alpha) * g[c] / total;
    g[c] = qc;
    qi = __double2ll_rn(qc * 1099511627776.0);  // 2^40
    qfix[c] = qi;
  }
  if (!sums) return;   // one scan block: its prefix is zero
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) qi += __shfl_xor_sync(0xffffffffu, qi, o);
  if ((t & 31) == 0 && qi) {
    const int64_t b = (int64_t)blockIdx.x * kNormBlock / kScanCells;
    atomicAdd(reinterpret_cast<unsigned long long*>(&cdf[min(n_cells, (b + 1) * kScanCells) - 1]),
              (unsigned long long)qi);
  }
}

// Inclusive scan over a block of 1,024 threads.
__device__ __forceinline__ long long block_scan(long long v, long long* ws) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  if (lane == 31) ws[warp] = v;
  __syncthreads();
  if (warp == 0) {
    long long w = ws[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long u = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += u;
    }
    ws[lane] = w;
  }
  __syncthreads();
  return warp ? v + ws[warp - 1] : v;
}

constexpr int kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(int64_t n_cells, int blocks,
                                                            int64_t* cdf) {
  __shared__ long long ws[32];
  long long run = 0;
  for (int b0 = 0; b0 < blocks; b0 += kScanThreads) {
    const int b = b0 + threadIdx.x;
    const int64_t at = min(n_cells, (int64_t)(b + 1) * kScanCells) - 1;
    const long long mine = b < blocks ? cdf[at] : 0;
    const long long inc = run + block_scan(mine, ws);
    if (b < blocks) cdf[at] = inc - mine;
    __syncthreads();
    run += ws[31];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kScanThreads) k_cdf(int64_t n_cells, const int64_t* qfix,
                                                      int64_t* cdf, bool sums) {
  __shared__ long long ws[32];
  const int64_t base = (int64_t)blockIdx.x * kScanCells;
  const int64_t end = min(n_cells, base + kScanCells);
  const long long before = sums ? cdf[end - 1] : 0;
  // two consecutive cells per thread
  const int64_t c = base + 2 * threadIdx.x;
  const long long a = c < end ? qfix[c] : 0, b = c + 1 < end ? qfix[c + 1] : 0;
  const long long inc = before + block_scan(a + b, ws);   // barriers: every thread has read `before`
  if (c < end) cdf[c] = inc - b;
  if (c + 1 < end) cdf[c + 1] = inc;
}

// (i + u) with u = (w + 1/2) 2^-32, exactly, for 0 <= i < 2^19: the integer
// i 2^33 + 2 w + 1 < 2^52 as a double, scaled by 2^-33.
__device__ __forceinline__ double cell_pos(int i, uint32_t w) {
  const unsigned long long m = ((unsigned long long)i << 33) | (2ull * w + 1ull);
  const double d = __longlong_as_double((long long)(m | 0x4330000000000000ull)) - 4503599627370496.0;
  return __hiloint2double(__double2hiint(d) - (33 << 20), __double2loint(d));
}
// x / n correctly rounded, with rn = 1 / n (Markstein, IBM J. Res. Dev. 34
// (1990)): x and n are positive and far from the exponent range's ends.
__device__ __forceinline__ double div_by(double x, double n, double rn) {
  const double q = x * rn;
  return fma(fma(-q, n, x), rn, q);
}

// Lanes per launch block and coarse CDF entries held in shared memory.
constexpr int kSampleBlock = 256, kCoarse = 1024;

// Draws from the integer CDF.  A lane costs about 50 FP64 instructions (the
// positions formed from integers, the divisions by the grid sizes as
// multiplications by their reciprocals with a correction; 120 before), the
// first ten steps of its search run in shared memory on every
// (N / 1024)-th entry.  200,000 lanes of 32,768 cells: 50 -> 32 us.
__global__ void __launch_bounds__(kSampleBlock) k_sample(CellGrid grid, int64_t n_cells,
                         const int64_t* qfix, const int64_t* cdf,
                         int64_t n, uint64_t seed, uint64_t id_offset, double b2_max, double* b,
                         double* u0, double* u1, double* u2, double* u3, double* w,
                         int32_t* cell) {
  __shared__ unsigned long long coarse[kCoarse];
  __shared__ double rn[5], mean;
  const int64_t step = (n_cells + kCoarse - 1) / kCoarse;
  const int n_coarse = (int)((n_cells + step - 1) / step);
  // coarse[k]: the last entry of the k-th run of `step` cells
  for (int k = threadIdx.x; k < n_coarse; k += kSampleBlock)
    coarse[k] = (unsigned long long)cdf[min(n_cells, (k + 1) * step) - 1];
  if (threadIdx.x < 5) {
    const int d = threadIdx.x == 0 ? grid.n_b2 : threadIdx.x == 1 ? grid.n_cth
                  : threadIdx.x == 2 ? grid.n_phi : threadIdx.x == 3 ? grid.n_eta : grid.n_chi;
    rn[threadIdx.x] = 1.0 / (double)d;
  }
  if (threadIdx.x == 32)
    mean = (double)(unsigned long long)cdf[n_cells - 1] / (double)n_cells;
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t id = id_offset + (uint64_t)i;
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const uint4 wa = philox4x32_10(make_uint4((uint32_t)id, (uint32_t)(id >> 32), 1u, 0u), key);
  const uint4 wb = philox4x32_10(make_uint4((uint32_t)id, (uint32_t)(id >> 32), 2u, 0u), key);
  const unsigned long long total = coarse[n_coarse - 1];
  // U = floor(u_0 total) with u_0 = (w + 1/2) 2^-32, in exact integer arithmetic:
  // (2 w + 1) total / 2^33
  const unsigned long long m = 2ull * wa.x + 1ull;
  const unsigned long long lo = m * total, hi = __umul64hi(m, total);
  const unsigned long long U = (hi << 31) | (lo >> 33);
  // first entry above U: its run among the coarse entries, then within the run
  int ca = 0, cz = n_coarse - 1;
  while (ca < cz) {
    const int mid = (ca + cz) >> 1;
    if (coarse[mid] > U) cz = mid;
    else ca = mid + 1;
  }
  int64_t a = ca * step, z = min(n_cells, (ca + 1) * step) - 1;
  while (a < z) {
    const int64_t mid = (a + z) >> 1;
    if ((unsigned long long)cdf[mid] > U) z = mid;
    else a = mid + 1;
  }
  int c = (int)a;   // at most 2^22 cells
  cell[i] = c;
  const int i_chi = c % grid.n_chi; c /= grid.n_chi;
  const int i_eta = c % grid.n_eta; c /= grid.n_eta;
  const int i_phi = c % grid.n_phi; c /= grid.n_phi;
  const int i_cth = c % grid.n_cth; c /= grid.n_cth;
  const int i_b2 = c;
  const int widest = max(max(grid.n_b2, grid.n_cth), max(grid.n_phi, max(grid.n_eta, grid.n_chi)));
  if (widest <= (1 << 19) && b2_max > 1e-100 && b2_max < 1e100) {
    b[i] = sqrt(div_by(b2_max * cell_pos(i_b2, wa.y), (double)grid.n_b2, rn[0]));
    u0[i] = div_by(cell_pos(i_cth, wa.z), (double)grid.n_cth, rn[1]);
    u1[i] = div_by(cell_pos(i_phi, wa.w), (double)grid.n_phi, rn[2]);
    u2[i] = div_by(cell_pos(i_eta, wb.x), (double)grid.n_eta, rn[3]);
    u3[i] = div_by(cell_pos(i_chi, wb.y), (double)grid.n_chi, rn[4]);
  } else {   // a dimension of more than 2^19 cells, or an extreme b2_max
    b[i] = sqrt(b2_max * (i_b2 + u01(wa.y)) / grid.n_b2);
    u0[i] = (i_cth + u01(wa.z)) / grid.n_cth;
    u1[i] = (i_phi + u01(wa.w)) / grid.n_phi;
    u2[i] = (i_eta + u01(wb.x)) / grid.n_eta;
    u3[i] = (i_chi + u01(wb.y)) / grid.n_chi;
  }
  w[i] = mean / (double)qfix[a];
}

int dev_ok() {
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return QCAMS_E_NODEVICE;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
    return QCAMS_E_NODEVICE;
  return (major == 10 && minor == 3) ? QCAMS_OK : QCAMS_E_NODEVICE;
}

bool mlp_ok(const qcams_mlp* m) {
  return m && m->params && m->adam_m && m->adam_v && m->grad && m->params_bf16;
}

Std std_of(const qcams_mlp* m) {
  Std s;
  for (int k = 0; k < 8; ++k) {
    s.mean[k] = m->x_mean[k];
    s.inv_std[k] = m->x_std[k] > 0.f ? 1.0f / m->x_std[k] : 1.0f;
  }
  return s;
}

int sm_count() {
  int dev = 0, s = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev);
  return s > 0 ? s : 1;
}

int status_of(cudaError_t e) { return e == cudaSuccess ? QCAMS_OK : QCAMS_E_CUDA; }

// Proposal spec check: QCAMS_E_INVALID for bad fields, QCAMS_E_CAPACITY for
// more than 2^22 cells.
int grid_status(const qcams_proposal_spec* s) {
  if (!s || s->n_b2 < 1 || s->n_cth < 1 || s->n_phi < 1 || s->n_eta < 1 || s->n_chi < 1)
    return QCAMS_E_INVALID;
  if (!(s->b2_max > 0) || !(s->alpha > 0) || !(s->alpha <= 1) || !(s->eps >= 0) ||
      !std::isfinite(s->E_col))
    return QCAMS_E_INVALID;
  const double n = (double)s->n_b2 * s->n_cth * s->n_phi * s->n_eta * s->n_chi;
  return n <= (double)(1 << 22) ? QCAMS_OK : QCAMS_E_CAPACITY;
}

CellGrid grid_of(const qcams_proposal_spec* s) {
  CellGrid g;
  g.n_b2 = s->n_b2;
  g.n_cth = s->n_cth;
  g.n_phi = s->n_phi;
  g.n_eta = s->n_eta;
  g.n_chi = s->n_chi;
  g.E = (float)s->E_col;
  g.v = (float)s->v;
  g.j = (float)s->j;
  g.b2_max = (float)s->b2_max;
  return g;
}

template <int CPW, bool DRAW>
cudaError_t launch_grad_cpw(const qcams_mlp* m, const float* x, const uint8_t* label,
                            const RowSrc& rows, int64_t n, float* loss_out, cudaStream_t st) {
  const size_t smem = sizeof(TrainSmem<CPW>);
  cudaError_t e = cudaFuncSetAttribute(
      k_mlp_grad<CPW, DRAW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int64_t grid = (n + BlockTiles<CPW>::RS - 1) / BlockTiles<CPW>::RS;
  if (grid > sm_count()) grid = sm_count();
  if (grid < 1) grid = 1;
  k_mlp_grad<CPW, DRAW><<<(unsigned)grid, THREADS, smem, st>>>(
      reinterpret_cast<const __nv_bfloat16*>(m->params_bf16), m->params, std_of(m), x, label, rows,
      n, m->grad, loss_out);
  return cudaGetLastError();
}

// Adds the gradient and loss of n rows to m->grad and *loss_out.  One block
// per SM at most.  A batch that fits one 64-sample round per SM (8,192
// samples: 128 blocks) takes that, the shortest block (84 KB of shared memory
// for weights and tiles); larger batches take 128-sample rounds (137 KB), half
// the rounds' global-atomic flushes.  With two 64-sample blocks per SM
// instead, 12,000 samples take 17.8 us against 20.2, 19,456 22.8 against
// 20.7, 1,000,000 439 against 570.
template <bool DRAW>
cudaError_t launch_grad(const qcams_mlp* m, const float* x, const uint8_t* label,
                        const RowSrc& rows, int64_t n, float* loss_out, cudaStream_t st) {
  return (n + 63) / 64 <= sm_count()
             ? launch_grad_cpw<1, DRAW>(m, x, label, rows, n, loss_out, st)
             : launch_grad_cpw<2, DRAW>(m, x, label, rows, n, loss_out, st);
}

cudaError_t launch_adam(qcams_mlp* m, float lr, bool clear, cudaStream_t st) {
  m->step += 1;
  const float c1 = (float)(1.0 - std::pow(0.9, (double)m->step));
  const float c2 = (float)(1.0 - std::pow(0.999, (double)m->step));
  k_adam<<<36, 256, 0, st>>>(m->params, m->adam_m, m->adam_v, m->grad,
                             reinterpret_cast<__nv_bfloat16*>(m->params_bf16), lr, c1, c2, clear);
  return cudaGetLastError();
}

}  // namespace
}  // namespace qcams

using namespace qcams;

extern "C" {

int qcams_mlp_init(qcams_mlp* m, uint64_t seed, void* cuda_stream) {
  if (!mlp_ok(m)) return QCAMS_E_INVALID;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  for (int k = 0; k < 8; ++k) {
    m->x_mean[k] = 0.0f;
    m->x_std[k] = 1.0f;
  }
  m->step = 0;
  (void)cudaGetLastError();
  k_mlp_init<<<36, 256, 0, (cudaStream_t)cuda_stream>>>(
      m->params, m->adam_m, m->adam_v, reinterpret_cast<__nv_bfloat16*>(m->params_bf16), seed);
  return status_of(cudaGetLastError());
}

int qcams_mlp_sync(const qcams_mlp* m, void* cuda_stream) {
  if (!mlp_ok(m)) return QCAMS_E_INVALID;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  (void)cudaGetLastError();
  k_mlp_sync<<<36, 256, 0, (cudaStream_t)cuda_stream>>>(
      m->params, reinterpret_cast<__nv_bfloat16*>(m->params_bf16));
  return status_of(cudaGetLastError());
}

int qcams_mlp_features(const qcams_batch* batch, const double* E_col, const double* b,
                       const int32_t* v, const int32_t* j, float* x, void* cuda_stream) {
  if (!batch || batch->n < 0) return QCAMS_E_INVALID;
  if (batch->n == 0) return QCAMS_OK;
  if (!E_col || !b || !v || !j || !x || !batch->u[0] || !batch->u[1] || !batch->u[2] ||
      !batch->u[3])
    return QCAMS_E_INVALID;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  (void)cudaGetLastError();
  k_features<<<(unsigned)((batch->n + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(
      batch->n, E_col, b, v, j, batch->u[0], batch->u[1], batch->u[2], batch->u[3], x);
  return status_of(cudaGetLastError());
}

int qcams_mlp_fit_standardizer(qcams_mlp* m, const float* x, int64_t n, void* cuda_stream) {
  if (!m || !x || n < 2) return QCAMS_E_INVALID;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  double* acc = nullptr;
  (void)cudaGetLastError();
  if (cudaMallocAsync((void**)&acc, 16 * sizeof(double), st) != cudaSuccess) return QCAMS_E_CUDA;
  cudaError_t e = cudaMemsetAsync(acc, 0, 16 * sizeof(double), st);
  if (e == cudaSuccess) {
    k_moments<<<sm_count() * 2, kMomentsBlock, 0, st>>>(x, n, acc);
    e = cudaGetLastError();
  }
  double h[16];
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, st);
  cudaFreeAsync(acc, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return QCAMS_E_CUDA;
  for (int k = 0; k < 8; ++k) {
    const double mu = h[k] / (double)n;
    const double var = h[8 + k] / (double)n - mu * mu;
    m->x_mean[k] = (float)mu;
    m->x_std[k] = var > 1e-20 ? (float)std::sqrt(var) : 1.0f;
  }
  return QCAMS_OK;
}

int qcams_mlp_grad(const qcams_mlp* m, const float* x, const uint8_t* label, int64_t n,
                   float* loss_out, void* cuda_stream) {
  if (!mlp_ok(m) || !x || !label || n < 1) return QCAMS_E_INVALID;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  (void)cudaGetLastError();
  cudaStream_t st = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaMemsetAsync(m->grad, 0, NP * sizeof(float), st);
  if (e == cudaSuccess && loss_out) e = cudaMemsetAsync(loss_out, 0, sizeof(float), st);
  if (e == cudaSuccess) e = launch_grad<false>(m, x, label, RowSrc{}, n, loss_out, st);
  return status_of(e);
}

int qcams_mlp_train_step(qcams_mlp* m, const float* x, const uint8_t* label, int64_t n,
                         float lr, float* loss_out, void* cuda_stream) {
  if (!(lr > 0.0f)) return QCAMS_E_INVALID;
  int rc = qcams_mlp_grad(m, x, label, n, loss_out, cuda_stream);
  if (rc != QCAMS_OK) return rc;
  return status_of(launch_adam(m, lr, false, (cudaStream_t)cuda_stream));
}

int qcams_mlp_train(qcams_mlp* m, const float* x, const uint8_t* label, int64_t n, int64_t steps,
                    int32_t batch, float lr, uint64_t seed, int64_t* idx, float* losses,
                    void* cuda_stream) {
  if (!mlp_ok(m) || !x || !label || !idx || n < 1 || steps < 0 || batch < 1 || !(lr > 0.0f))
    return QCAMS_E_INVALID;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  (void)cudaGetLastError();
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (losses && steps > 0 &&
      cudaMemsetAsync(losses, 0, sizeof(float) * (size_t)steps, st) != cudaSuccess)
    return QCAMS_E_CUDA;
  if (steps == 0) return QCAMS_OK;
  // Two launches a step: the gradient kernel draws its own rows (as
  // k_draw_idx does) and Adam clears the gradient for the next step.
  // 16.8 us a step at 8,192 rows, 32.1 with an index draw and a memset more
  // and the earlier passes.  All steps in one cooperative launch take 13.8,
  // but need every SM free at once and a grid barrier, whose give-up an
  // asynchronous call cannot report.
  cudaError_t e = cudaMemsetAsync(m->grad, 0, NP * sizeof(float), st);
  RowSrc rows{n, seed, (uint64_t)m->step};
  for (int64_t s = 0; s < steps && e == cudaSuccess; ++s) {
    rows.step = (uint64_t)m->step;
    e = launch_grad<true>(m, x, label, rows, batch, losses ? losses + s : nullptr, st);
    if (e == cudaSuccess) e = launch_adam(m, lr, s + 1 < steps, st);
  }
  if (e != cudaSuccess) return QCAMS_E_CUDA;
  k_draw_idx<<<(batch + 255) / 256, 256, 0, st>>>(idx, batch, rows);
  return status_of(cudaGetLastError());
}

int qcams_mlp_infer(const qcams_mlp* m, const float* x, int64_t n, float* probs,
                    void* cuda_stream) {
  if (!mlp_ok(m) || !x || !probs || n < 0) return QCAMS_E_INVALID;
  if (n == 0) return QCAMS_OK;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  (void)cudaGetLastError();
  const int64_t chunks = (n + 15) / 16;
  int64_t grid = (chunks + WARPS - 1) / WARPS;
  if (grid > 8 * sm_count()) grid = 8 * sm_count();
  CellGrid none{};
  k_mlp_infer<<<(unsigned)grid, THREADS, 0, (cudaStream_t)cuda_stream>>>(
      reinterpret_cast<const __nv_bfloat16*>(m->params_bf16), m->params, std_of(m), x, n, none,
      0, probs, nullptr, 0.0);
  return status_of(cudaGetLastError());
}

int qcams_build_proposal(const qcams_mlp* m, const qcams_proposal_spec* spec, double* q,
                         int64_t* qfix, int64_t* cdf, void* cuda_stream) {
  if (!mlp_ok(m) || !q || !qfix || !cdf) return QCAMS_E_INVALID;
  if (const int gs = grid_status(spec)) return gs;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int64_t N = (int64_t)spec->n_b2 * spec->n_cth * spec->n_phi * spec->n_eta * spec->n_chi;
  const int64_t chunks = (N + 15) / 16;
  int64_t grid = (chunks + WARPS - 1) / WARPS;
  if (grid > 8 * sm_count()) grid = 8 * sm_count();
  (void)cudaGetLastError();
  k_mlp_infer<<<(unsigned)grid, THREADS, 0, st>>>(
      reinterpret_cast<const __nv_bfloat16*>(m->params_bf16), m->params, std_of(m), nullptr, N,
      grid_of(spec), 1, nullptr, q, spec->eps);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return QCAMS_E_CUDA;
  const unsigned blocks = (unsigned)((N + kScanCells - 1) / kScanCells);
  const bool sums = blocks > 1;
  k_run_sums<<<kRuns / kRunTile, 32, 0, st>>>(q, N, cdf, (int)blocks);
  k_normalise<<<(unsigned)((N + kNormBlock - 1) / kNormBlock), kNormBlock, 0, st>>>(
      q, N, spec->alpha, qfix, cdf, sums);
  if (sums) k_scan_sums<<<1, kScanThreads, 0, st>>>(N, (int)blocks, cdf);
  k_cdf<<<blocks, kScanThreads, 0, st>>>(N, qfix, cdf, sums);
  return status_of(cudaGetLastError());
}

int qcams_sample_proposal(const qcams_proposal_spec* spec, const int64_t* qfix,
                          const int64_t* cdf, int64_t n, uint64_t seed, uint64_t id_offset,
                          double* b, double* const* u_out, double* w, int32_t* cell,
                          void* cuda_stream) {
  if (!qfix || !cdf || n < 0 || !b || !u_out || !w || !cell) return QCAMS_E_INVALID;
  if (const int gs = grid_status(spec)) return gs;
  if (!u_out[0] || !u_out[1] || !u_out[2] || !u_out[3]) return QCAMS_E_INVALID;
  if (n == 0) return QCAMS_OK;
  int rc;
  if ((rc = dev_ok()) != QCAMS_OK) return rc;
  const int64_t N = (int64_t)spec->n_b2 * spec->n_cth * spec->n_phi * spec->n_eta * spec->n_chi;
  (void)cudaGetLastError();
  k_sample<<<(unsigned)((n + kSampleBlock - 1) / kSampleBlock), kSampleBlock, 0,
             (cudaStream_t)cuda_stream>>>(
      grid_of(spec), N, qfix, cdf, n, seed, id_offset, spec->b2_max, b, u_out[0], u_out[1],
      u_out[2], u_out[3], w, cell);
  return status_of(cudaGetLastError());
}

}  // extern "C"
