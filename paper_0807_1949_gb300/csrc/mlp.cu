// Learned line impedance: a 3-layer perceptron 8 -> 64 -> 64 -> 1 (ReLU) that maps 8 local
// features of a line end to log Z (impedance matching, §7.1, governs convergence; the network
// replaces the input-impedance rule with impedances found by search).  Weights are held in BF16
// for the forward and backward passes (FP32 accumulation); Adam keeps an FP32 master copy.
//
// Parameter layout (P = 4801 floats): W1[64][8], b1[64], W2[64][64], b2[64], W3[64], b3.
// Forward and gradient run on the tensor cores with FP32 activations split into exact bf16 terms.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "internal.h"

namespace vtm {

constexpr int kIn = VTM_MLP_IN;
constexpr int kH = VTM_MLP_HIDDEN;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH, kParams = kOffB3 + 1;

static_assert(kParams == VTM_MLP_PARAMS, "parameter count");

// D += A B on the tensor cores, bf16 operands, FP32 accumulation: 16 x 8 += 16 x 16 times 16 x 8,
// and 16 x 8 times 8 x 8.  Lane 4 g + t holds of A the pairs at rows g, g + 8 and columns 2 t (+ 8),
// of B the pairs at rows 2 t (+ 8) of column g, of D rows g, g + 8 and columns 2 t, 2 t + 1.
__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(b));
}

// A pair of floats as three bf16 pairs, p[0] + p[1] + p[2] = the floats exactly (8 + 8 + 8 bits); an
// infinity or NaN is the first term alone.  POS: both are >= 0 (or NaN).
template <bool POS>
__device__ __forceinline__ void split3(float x, float y, uint32_t (&p)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    p[i] = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
    x -= __uint_as_float(__float_as_uint(x) & 0xFFFF0000u);
    y -= __uint_as_float(__float_as_uint(y) & 0xFFFF0000u);
    if (i == 0) {  // inf - inf
      x = POS ? fmaxf(x, 0.f) : x == x ? x : 0.f;
      y = POS ? fmaxf(y, 0.f) : y == y ? y : 0.f;
    }
  }
}

// The same with the first two terms rounded to nearest: their remainders are at most 2^-8 and 2^-17 of the
// power of two below |x|, of either sign, and the third term is exact.  For products of two split
// operands, where the terms' own products that are left out count: with cut-off terms the remainders all
// have x's sign and are up to twice as large, and leaving out mid lo + lo mid (and lo lo) lost up to 2^-21
// of a product, always towards zero; rounded ones lose 2^-24 at most and nothing on average.
__device__ __forceinline__ void split3_nearest(float x, float y, uint32_t (&p)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p[i]) : "f"(y), "f"(x));
    x -= __uint_as_float(p[i] << 16);
    y -= __uint_as_float(p[i] & 0xFFFF0000u);
    if (i == 0) {  // an infinity (or a value that rounds to one) or NaN is the first term alone
      x = fabsf(x) < INFINITY ? x : 0.f;
      y = fabsf(y) < INFINITY ? y : 0.f;
    }
  }
}

// Entries 2 t, 2 t + 1 of sample i; VEC: X is 8-byte aligned.
template <bool VEC>
__device__ __forceinline__ float2 load_pair(const float* __restrict__ X, int64_t i, int64_t n, int t) {
  if (i >= n) return make_float2(0.f, 0.f);
  const float* p = X + i * kIn + 2 * t;
  if constexpr (VEC) return *reinterpret_cast<const float2*>(p);
  else return make_float2(p[0], p[1]);
}

// Forward pass, one warp per 16 samples at a time.  The activations stay FP32: as operands they are
// three exact bf16 terms, the weights are bf16 to begin with, so every product is exact.  The sums of
// the two lower terms (2^-8 of the first) accumulate by themselves and those of the first term K step
// by K step, all added in FP32: the tensor core's own accumulation cuts off instead of rounding, and
// short chains keep that below the rounding of an FP32 loop.  The hidden layer goes from the first
// product's accumulators straight into the second one's operand registers; the second layer's weights
// stay in registers.
//
// What bounds it: the tensor pipe (120 products of 2 cycles each per 16 samples: 39 us for 760,000)
// and, close to it, the instructions that split the activations.  760,000 samples: 369 us with one
// thread per sample and the weights from shared memory, 72 us so (error against FP64 8.7e-8 and
// 4.5e-8).
constexpr int kFwdThreads = 128;

template <bool VEC>
__global__ void __launch_bounds__(kFwdThreads, 3) k_mlp_forward(const __nv_bfloat16* __restrict__ wb,
                                                               const float* __restrict__ X, float* __restrict__ y,
                                                               int64_t n) {
  __shared__ float2 sb1[kH / 2], sb2[kH / 2], sw3[kH / 2];
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  if (threadIdx.x < kH / 2) {
    const int j = 2 * threadIdx.x;
    sb1[threadIdx.x] = make_float2(__bfloat162float(wb[kOffB1 + j]), __bfloat162float(wb[kOffB1 + j + 1]));
    sb2[threadIdx.x] = make_float2(__bfloat162float(wb[kOffB2 + j]), __bfloat162float(wb[kOffB2 + j + 1]));
    sw3[threadIdx.x] = make_float2(__bfloat162float(wb[kOffW3 + j]), __bfloat162float(wb[kOffW3 + j + 1]));
  }
  const float b3 = __bfloat162float(wb[kOffB3]);
  // weight operands: column (output) 8 nb + g, rows (inputs) 16 ks + 2 t, + 8; all even offsets
  const uint32_t* w32 = reinterpret_cast<const uint32_t*>(wb);
  uint32_t w1[8], w2[8][4][2];
#pragma unroll
  for (int nb = 0; nb < 8; ++nb) {
    w1[nb] = w32[(kOffW1 + (8 * nb + g) * kIn + 2 * t) / 2];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int h = 0; h < 2; ++h) w2[nb][ks][h] = w32[(kOffW2 + (8 * nb + g) * kH + 16 * ks + 8 * h + 2 * t) / 2];
  }
  __syncthreads();
  const int64_t warps = (int64_t)gridDim.x * (kFwdThreads / 32);
  for (int64_t tile = blockIdx.x * (int64_t)(kFwdThreads / 32) + (threadIdx.x >> 5); tile * 16 < n; tile += warps) {
    const int64_t i0 = tile * 16 + g, i1 = i0 + 8;
    const float2 x0 = load_pair<VEC>(X, i0, n, t), x1 = load_pair<VEC>(X, i1, n, t);
    uint32_t xa[3], xb[3];
    split3<false>(x0.x, x0.y, xa);
    split3<false>(x1.x, x1.y, xb);
    // layer 1, and its output as the three terms of the next operand (16 inputs per K step)
    uint32_t h1[3][4][4];
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) {
      float lo[4] = {0.f, 0.f, 0.f, 0.f}, hi[4] = {0.f, 0.f, 0.f, 0.f};
      mma_k8(lo, xa[2], xb[2], w1[nb]);
      mma_k8(lo, xa[1], xb[1], w1[nb]);
      mma_k8(hi, xa[0], xb[0], w1[nb]);
      const float2 b = sb1[4 * nb + t];
      uint32_t p[3], q[3];
      split3<true>(fmaxf((hi[0] + b.x) + lo[0], 0.f), fmaxf((hi[1] + b.y) + lo[1], 0.f), p);
      split3<true>(fmaxf((hi[2] + b.x) + lo[2], 0.f), fmaxf((hi[3] + b.y) + lo[3], 0.f), q);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        h1[k][nb >> 1][2 * (nb & 1)] = p[k];
        h1[k][nb >> 1][2 * (nb & 1) + 1] = q[k];
      }
    }
    // layer 2 and the output's weighted sum, eight units at a time
    float o0 = 0.f, o1 = 0.f;
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) {
      float lo[4] = {0.f, 0.f, 0.f, 0.f}, hi[4][4];
#pragma unroll
      for (int k = 2; k >= 1; --k)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) mma_k16(lo, h1[k][ks], w2[nb][ks][0], w2[nb][ks][1]);
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
#pragma unroll
        for (int e = 0; e < 4; ++e) hi[ks][e] = 0.f;
        mma_k16(hi[ks], h1[0][ks], w2[nb][ks][0], w2[nb][ks][1]);
      }
      const float2 b = sb2[4 * nb + t], w3 = sw3[4 * nb + t];
      float a[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float v = ((hi[0][e] + hi[1][e]) + (hi[2][e] + hi[3][e])) + lo[e] + ((e & 1) ? b.y : b.x);
        a[e] = fmaxf(v, 0.f);
      }
      o0 = fmaf(w3.x, a[0], fmaf(w3.y, a[1], o0));
      o1 = fmaf(w3.x, a[2], fmaf(w3.y, a[3], o1));
    }
    o0 += __shfl_xor_sync(0xffffffffu, o0, 1);
    o1 += __shfl_xor_sync(0xffffffffu, o1, 1);
    o0 += __shfl_xor_sync(0xffffffffu, o0, 2);
    o1 += __shfl_xor_sync(0xffffffffu, o1, 2);
    if (t == 0 && i0 < n) y[i0] = o0 + b3;
    if (t == 1 && i1 < n) y[i1] = o1 + b3;
  }
}

// Mean-squared-error loss over n samples and its gradient w.r.t. the (BF16) weights.  A CTA takes
// tiles of 64 samples, 16 per warp.  Forward as in k_mlp_forward; the layers' deltas and activations
// (FP32 values as three exact bf16 terms) go to shared memory, where ldmatrix.trans turns them into
// the operands of the sums over samples: warp m computes rows 16 m .. 16 m + 15 of dW2 = D2^T H1 and
// of dW1 = D1^T X, and db2, db1 as products with columns of ones.  Of the nine products of terms
// (split3_nearest) six count, the other three are at most 2^-24 of the whole; those of the two first terms
// accumulate apart from the rest, and every tile's sums are added in FP32, the bias sums' after every 16
// samples (through one accumulator for all terms of a tile the tensor core cut off twelve times: 64 equal
// samples gave biases up to 6e-7 away from one sample's, now the same bits).  Each CTA writes its partial
// gradient and loss; k_mlp_reduce adds the CTAs' partials in their order, so the gradient is the same bit for
// bit from run to run.
//
// What bounds it: latency at the training loop's 16,384 samples (one or two tiles per CTA).  There
// 115 us for the call with one thread per sample, serial sums over the tile and an atomic per
// parameter and tile, 55 us so (loss and gradients read back by the caller included; error against
// FP64 2.0e-7 and 0.8e-7).
constexpr int kGradWarps = 4;
constexpr int kGradThreads = 32 * kGradWarps;
constexpr int kTile = 16 * kGradWarps;      // samples per tile
constexpr int kPart = kParams + 1;          // a CTA's partial: gradient, loss
constexpr int kRow = kH + 8;                // bf16 entries of a row in shared memory (conflict-free ldmatrix)

struct GradSmem {
  __nv_bfloat16 w2[kH][kRow];               // W2[j2][j]
  __nv_bfloat16 w2t[kH][kRow];              // W2[j2][j] at [j][j2]
  __nv_bfloat16 h1[3][kTile][kRow];
  __nv_bfloat16 d2[3][kTile][kRow];
  __nv_bfloat16 d1[3][kTile][kRow];
  __nv_bfloat16 xs[3][kTile][kIn];
  float2 b1[kH / 2], b2[kH / 2], w3[kH / 2];
  float dw3[kGradWarps][kH];
  float sums[kGradWarps][2];                // db3, loss
};

__device__ __forceinline__ void ldmatrix_t(const __nv_bfloat16* p, uint32_t (&v)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}

template <bool VEC>
__global__ void __launch_bounds__(kGradThreads, 2) k_mlp_grad(const __nv_bfloat16* __restrict__ wb,
                                                             const float* __restrict__ X, const float* __restrict__ tg,
                                                             int64_t n, float inv_n, float* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GradSmem& sm = *reinterpret_cast<GradSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  for (int i = tid; i < kH * kH; i += kGradThreads) {
    const __nv_bfloat16 v = wb[kOffW2 + i];
    sm.w2[i / kH][i % kH] = v;
    sm.w2t[i % kH][i / kH] = v;
  }
  if (tid < kH / 2) {
    const int j = 2 * tid;
    sm.b1[tid] = make_float2(__bfloat162float(wb[kOffB1 + j]), __bfloat162float(wb[kOffB1 + j + 1]));
    sm.b2[tid] = make_float2(__bfloat162float(wb[kOffB2 + j]), __bfloat162float(wb[kOffB2 + j + 1]));
    sm.w3[tid] = make_float2(__bfloat162float(wb[kOffW3 + j]), __bfloat162float(wb[kOffW3 + j + 1]));
  }
  const float b3 = __bfloat162float(wb[kOffB3]);
  const uint32_t* w32 = reinterpret_cast<const uint32_t*>(wb);
  uint32_t w1[8];
#pragma unroll
  for (int nb = 0; nb < 8; ++nb) w1[nb] = w32[(kOffW1 + (8 * nb + g) * kIn + 2 * t) / 2];
  // sums over this CTA's tiles
  float aw2[8][4], aw1[4], ab2[2], ab1[2], aw3[8][2], ab3 = 0.f, aloss = 0.f;
#pragma unroll
  for (int nb = 0; nb < 8; ++nb) {
#pragma unroll
    for (int e = 0; e < 4; ++e) aw2[nb][e] = 0.f;
    aw3[nb][0] = aw3[nb][1] = 0.f;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) aw1[e] = 0.f;
  ab2[0] = ab2[1] = ab1[0] = ab1[1] = 0.f;
  __syncthreads();

  // 16 x 64 outputs of a layer's product from its operand terms a and weights w ([output][input])
  auto layer = [&](const uint32_t (&a)[3][4][4], const __nv_bfloat16 (&w)[kH][kRow], int nb, float (&v)[4]) {
    float lo[4] = {0.f, 0.f, 0.f, 0.f}, hi[4][4];
    uint32_t wr[4][2];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        wr[ks][h] = *reinterpret_cast<const uint32_t*>(&w[8 * nb + g][16 * ks + 8 * h + 2 * t]);
#pragma unroll
    for (int k = 2; k >= 1; --k)
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) mma_k16(lo, a[k][ks], wr[ks][0], wr[ks][1]);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
#pragma unroll
      for (int e = 0; e < 4; ++e) hi[ks][e] = 0.f;
      mma_k16(hi[ks], a[0][ks], wr[ks][0], wr[ks][1]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = ((hi[0][e] + hi[1][e]) + (hi[2][e] + hi[3][e])) + lo[e];
  };
  // a pair of rows' values of columns 8 nb + 2 t, + 1 as terms: into operand registers and shared memory
  auto keep = [&](float v0, float v1, float v2, float v3, int nb, uint32_t (*a)[4][4],
                  __nv_bfloat16 (&dst)[3][kTile][kRow]) {
    uint32_t p[3], q[3];
    split3_nearest(v0, v1, p);
    split3_nearest(v2, v3, q);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (a) {
        a[k][nb >> 1][2 * (nb & 1)] = p[k];
        a[k][nb >> 1][2 * (nb & 1) + 1] = q[k];
      }
      *reinterpret_cast<uint32_t*>(&dst[k][16 * warp + g][8 * nb + 2 * t]) = p[k];
      *reinterpret_cast<uint32_t*>(&dst[k][16 * warp + g + 8][8 * nb + 2 * t]) = q[k];
    }
  };

  for (int64_t tile = blockIdx.x; tile * kTile < n; tile += gridDim.x) {
    const int64_t i0 = tile * kTile + 16 * warp + g, i1 = i0 + 8;
    const float2 x0 = load_pair<VEC>(X, i0, n, t), x1 = load_pair<VEC>(X, i1, n, t);
    const float t0 = i0 < n ? tg[i0] : 0.f, t1 = i1 < n ? tg[i1] : 0.f;
    uint32_t xa[3], xb[3];
    split3_nearest(x0.x, x0.y, xa);
    split3_nearest(x1.x, x1.y, xb);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      *reinterpret_cast<uint32_t*>(&sm.xs[k][16 * warp + g][2 * t]) = xa[k];
      *reinterpret_cast<uint32_t*>(&sm.xs[k][16 * warp + g + 8][2 * t]) = xb[k];
    }
    uint32_t op[3][4][4];  // h1, then d2
    uint32_t live1 = 0;    // h1 > 0, bit 4 nb + e
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) {
      float lo[4] = {0.f, 0.f, 0.f, 0.f}, hi[4] = {0.f, 0.f, 0.f, 0.f};
      mma_k8(lo, xa[2], xb[2], w1[nb]);
      mma_k8(lo, xa[1], xb[1], w1[nb]);
      mma_k8(hi, xa[0], xb[0], w1[nb]);
      const float2 b = sm.b1[4 * nb + t];
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        v[e] = fmaxf((hi[e] + ((e & 1) ? b.y : b.x)) + lo[e], 0.f);
        live1 |= (v[e] > 0.f ? 1u : 0u) << (4 * nb + e);
      }
      keep(v[0], v[1], v[2], v[3], nb, op, sm.h1);
    }
    float h2[8][4], o0 = 0.f, o1 = 0.f;
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) {
      layer(op, sm.w2, nb, h2[nb]);
      const float2 b = sm.b2[4 * nb + t], w3 = sm.w3[4 * nb + t];
#pragma unroll
      for (int e = 0; e < 4; ++e) h2[nb][e] = fmaxf(h2[nb][e] + ((e & 1) ? b.y : b.x), 0.f);
      o0 = fmaf(w3.x, h2[nb][0], fmaf(w3.y, h2[nb][1], o0));
      o1 = fmaf(w3.x, h2[nb][2], fmaf(w3.y, h2[nb][3], o1));
    }
    o0 += __shfl_xor_sync(0xffffffffu, o0, 1);
    o1 += __shfl_xor_sync(0xffffffffu, o1, 1);
    o0 += __shfl_xor_sync(0xffffffffu, o0, 2);
    o1 += __shfl_xor_sync(0xffffffffu, o1, 2);
    const float e0 = i0 < n ? (o0 + b3) - t0 : 0.f, e1 = i1 < n ? (o1 + b3) - t1 : 0.f;
    const float dy0 = 2.f * e0 * inv_n, dy1 = 2.f * e1 * inv_n;
    if (t == 0) {
      ab3 += dy0 + dy1;
      aloss += (e0 * e0 + e1 * e1) * inv_n;
    }
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) {
      const float2 w3 = sm.w3[4 * nb + t];
      aw3[nb][0] += dy0 * h2[nb][0] + dy1 * h2[nb][2];
      aw3[nb][1] += dy0 * h2[nb][1] + dy1 * h2[nb][3];
      keep(h2[nb][0] > 0.f ? dy0 * w3.x : 0.f, h2[nb][1] > 0.f ? dy0 * w3.y : 0.f,
           h2[nb][2] > 0.f ? dy1 * w3.x : 0.f, h2[nb][3] > 0.f ? dy1 * w3.y : 0.f, nb, op, sm.d2);
    }
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) {
      float v[4];
      layer(op, sm.w2t, nb, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = (live1 >> (4 * nb + e)) & 1u ? v[e] : 0.f;
      keep(v[0], v[1], v[2], v[3], nb, nullptr, sm.d1);
    }
    __syncthreads();
    // ---- sums over the tile's samples: rows 16 warp .. + 15
    const int ms = (lane >> 4) * 8 + (lane & 7), mc = ((lane >> 3) & 1) * 8;  // A: matrices (0, 0) (0, 8) (8, 0) (8, 8)
    const int bs = ((lane >> 3) & 1) * 8 + (lane & 7), bc = (lane >> 4) * 8;  // B: (0, 0) (8, 0) (0, 8) (8, 8)
    // sums of 16 samples' deltas (rows g, g + 8) added to a layer's bias sums: first terms in the even
    // columns, the others in the odd ones
    const uint32_t even = (g & 1) ? 0u : 0x3F803F80u, odd = (g & 1) ? 0x3F803F80u : 0u;
    auto bias = [&](const uint32_t (&A)[3][4], float (&sum)[2]) {
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      mma_k16(d, A[2], odd, odd);
      mma_k16(d, A[1], odd, odd);
      mma_k16(d, A[0], even, even);
      sum[0] += d[0] + d[1];
      sum[1] += d[2] + d[3];
    };
    {
      float hi[8][4], lo[8][4];
#pragma unroll
      for (int nb = 0; nb < 8; ++nb)
#pragma unroll
        for (int e = 0; e < 4; ++e) hi[nb][e] = lo[nb][e] = 0.f;
#pragma unroll
      for (int ks = 0; ks < kTile / 16; ++ks) {
        uint32_t A[3][4];
#pragma unroll
        for (int k = 0; k < 3; ++k) ldmatrix_t(&sm.d2[k][16 * ks + ms][16 * warp + mc], A[k]);
        bias(A, ab2);
#pragma unroll
        for (int np = 0; np < 4; ++np) {
          uint32_t B[3][4];
#pragma unroll
          for (int k = 0; k < 3; ++k) ldmatrix_t(&sm.h1[k][16 * ks + bs][16 * np + bc], B[k]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int nb = 2 * np + h;
            mma_k16(lo[nb], A[2], B[0][2 * h], B[0][2 * h + 1]);
            mma_k16(lo[nb], A[0], B[2][2 * h], B[2][2 * h + 1]);
            mma_k16(lo[nb], A[1], B[1][2 * h], B[1][2 * h + 1]);
            mma_k16(lo[nb], A[1], B[0][2 * h], B[0][2 * h + 1]);
            mma_k16(lo[nb], A[0], B[1][2 * h], B[1][2 * h + 1]);
            mma_k16(hi[nb], A[0], B[0][2 * h], B[0][2 * h + 1]);
          }
        }
      }
#pragma unroll
      for (int nb = 0; nb < 8; ++nb)
#pragma unroll
        for (int e = 0; e < 4; ++e) aw2[nb][e] += hi[nb][e] + lo[nb][e];
    }
    {
      float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kp = 0; kp < kTile / 32; ++kp) {
        uint32_t B[3][4];  // samples 32 kp + 0, 8, 16, 24 of the features
#pragma unroll
        for (int k = 0; k < 3; ++k) ldmatrix_t(&sm.xs[k][32 * kp + lane][0], B[k]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t A[3][4];
#pragma unroll
          for (int k = 0; k < 3; ++k) ldmatrix_t(&sm.d1[k][32 * kp + 16 * h + ms][16 * warp + mc], A[k]);
          bias(A, ab1);
          mma_k16(lo, A[2], B[0][2 * h], B[0][2 * h + 1]);
          mma_k16(lo, A[0], B[2][2 * h], B[2][2 * h + 1]);
          mma_k16(lo, A[1], B[1][2 * h], B[1][2 * h + 1]);
          mma_k16(lo, A[1], B[0][2 * h], B[0][2 * h + 1]);
          mma_k16(lo, A[0], B[1][2 * h], B[1][2 * h + 1]);
          mma_k16(hi, A[0], B[0][2 * h], B[0][2 * h + 1]);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) aw1[e] += hi[e] + lo[e];
    }
    __syncthreads();
  }
  // ---- this CTA's partial
  float* P = part + (size_t)blockIdx.x * kPart;
  const int r0 = 16 * warp + g;
#pragma unroll
  for (int nb = 0; nb < 8; ++nb)
#pragma unroll
    for (int e = 0; e < 4; ++e) P[kOffW2 + (r0 + 8 * (e >> 1)) * kH + 8 * nb + 2 * t + (e & 1)] = aw2[nb][e];
#pragma unroll
  for (int e = 0; e < 4; ++e) P[kOffW1 + (r0 + 8 * (e >> 1)) * kIn + 2 * t + (e & 1)] = aw1[e];
  if (t == 0) {
    P[kOffB2 + r0] = ab2[0];
    P[kOffB2 + r0 + 8] = ab2[1];
    P[kOffB1 + r0] = ab1[0];
    P[kOffB1 + r0 + 8] = ab1[1];
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
#pragma unroll
    for (int nb = 0; nb < 8; ++nb)
#pragma unroll
      for (int e = 0; e < 2; ++e) aw3[nb][e] += __shfl_xor_sync(0xffffffffu, aw3[nb][e], o);
    ab3 += __shfl_xor_sync(0xffffffffu, ab3, o);
    aloss += __shfl_xor_sync(0xffffffffu, aloss, o);
  }
  if (g == 0)
#pragma unroll
    for (int nb = 0; nb < 8; ++nb)
#pragma unroll
      for (int e = 0; e < 2; ++e) sm.dw3[warp][8 * nb + 2 * t + e] = aw3[nb][e];
  if (lane == 0) {
    sm.sums[warp][0] = ab3;
    sm.sums[warp][1] = aloss;
  }
  __syncthreads();
  if (tid < kH + 2) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kGradWarps; ++w) v += tid < kH ? sm.dw3[w][tid] : sm.sums[w][tid - kH];
    P[tid < kH ? kOffW3 + tid : tid == kH ? kOffB3 : kParams] = v;
  }
}

// Gradient and loss from the CTAs' partials, in their order: 8 runs of them per output, then those.
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ part, int nparts, float* __restrict__ grad,
                                                   float* __restrict__ loss) {
  __shared__ float red[8][32];
  const int o = threadIdx.x & 31, run = threadIdx.x >> 5, i = blockIdx.x * 32 + o;
  float v = 0.f;
  if (i < kPart) {
    const int c0 = nparts * run / 8, c1 = nparts * (run + 1) / 8;
#pragma unroll 8
    for (int c = c0; c < c1; ++c) v += part[(size_t)c * kPart + i];
  }
  red[run][o] = v;
  __syncthreads();
  if (run == 0 && i < kPart) {
    v = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) v += red[k][o];
    if (i < kParams) grad[i] = v;
    else *loss = v;
  }
}

__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v, const float* __restrict__ g,
                       __nv_bfloat16* __restrict__ wb, int np, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  p[i] = pi;
  wb[i] = __float2bfloat16_rn(pi);
}

__global__ void k_to_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ wb, int np) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < np) wb[i] = __float2bfloat16_rn(p[i]);
}

}  // namespace vtm

struct vtm_mlp {
  float* p = nullptr;       // FP32 master parameters (device)
  float* m = nullptr;       // Adam first moment
  float* v = nullptr;       // Adam second moment
  float* g = nullptr;       // gradient
  float* loss = nullptr;    // device scalar
  float* part = nullptr;    // the gradient kernel's partials
  int part_ctas = 0;
  float* h_loss = nullptr;  // pinned
  __nv_bfloat16* wb = nullptr;  // BF16 weights used by the kernels
  int64_t step = 0;
  ~vtm_mlp() {
    cudaFree(p);
    cudaFree(m);
    cudaFree(v);
    cudaFree(g);
    cudaFree(loss);
    cudaFree(part);
    cudaFreeHost(h_loss);
    cudaFree(wb);
  }
};

namespace vtm {

#define MLP_CUDA(call)                                                                           \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess) fail(VTM_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// SplitMix64 (Steele, Lea, Flood 2014), used as a counter-based generator for the initial weights.
static uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

static double uniform01(uint64_t seed, uint64_t k) { return (double)(splitmix64(seed * 0x100000001B3ull + k) >> 11) * 0x1.0p-53; }

vtm_mlp* mlp_create(uint64_t seed) {
  std::unique_ptr<vtm_mlp> m(new vtm_mlp());
  const size_t pb = kParams * sizeof(float);
  MLP_CUDA(cudaMalloc(&m->p, pb));
  MLP_CUDA(cudaMalloc(&m->m, pb));
  MLP_CUDA(cudaMalloc(&m->v, pb));
  MLP_CUDA(cudaMalloc(&m->g, pb));
  MLP_CUDA(cudaMalloc(&m->loss, sizeof(float)));
  MLP_CUDA(cudaMalloc(&m->wb, kParams * sizeof(__nv_bfloat16)));
  // the gradient's workspace (5.8 MB), here so that the first gradient costs what the others do
  int dev = 0, nsm = 1;
  MLP_CUDA(cudaGetDevice(&dev));
  MLP_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  m->part_ctas = 2 * nsm;  // as many CTAs as run at a time
  MLP_CUDA(cudaMalloc(&m->part, (size_t)m->part_ctas * kPart * sizeof(float)));
  MLP_CUDA(cudaMallocHost(&m->h_loss, sizeof(float)));
  for (const void* k : {(const void*)k_mlp_grad<true>, (const void*)k_mlp_grad<false>})
    MLP_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)));
  // He-uniform weights, zero biases
  std::vector<float> h(kParams, 0.f);
  auto fill = [&](int off, int rows, int cols) {
    const double a = std::sqrt(6.0 / cols);
    for (int r = 0; r < rows * cols; ++r) h[off + r] = (float)((2.0 * uniform01(seed, off + r) - 1.0) * a);
  };
  fill(kOffW1, kH, kIn);
  fill(kOffW2, kH, kH);
  fill(kOffW3, 1, kH);
  MLP_CUDA(cudaMemcpy(m->p, h.data(), pb, cudaMemcpyHostToDevice));
  MLP_CUDA(cudaMemset(m->m, 0, pb));
  MLP_CUDA(cudaMemset(m->v, 0, pb));
  MLP_CUDA(cudaMemset(m->g, 0, pb));
  k_to_bf16<<<(kParams + 255) / 256, 256>>>(m->p, m->wb, kParams);
  MLP_CUDA(cudaGetLastError());
  MLP_CUDA(cudaDeviceSynchronize());
  return m.release();
}

void mlp_set_params(vtm_mlp* m, const float* host) {
  MLP_CUDA(cudaMemcpy(m->p, host, kParams * sizeof(float), cudaMemcpyHostToDevice));
  MLP_CUDA(cudaMemset(m->m, 0, kParams * sizeof(float)));
  MLP_CUDA(cudaMemset(m->v, 0, kParams * sizeof(float)));
  m->step = 0;
  k_to_bf16<<<(kParams + 255) / 256, 256>>>(m->p, m->wb, kParams);
  MLP_CUDA(cudaGetLastError());
  MLP_CUDA(cudaDeviceSynchronize());
}

void mlp_get_params(const vtm_mlp* m, float* host) {
  MLP_CUDA(cudaMemcpy(host, m->p, kParams * sizeof(float), cudaMemcpyDeviceToHost));
}

void mlp_get_grads(const vtm_mlp* m, float* host) {
  MLP_CUDA(cudaMemcpy(host, m->g, kParams * sizeof(float), cudaMemcpyDeviceToHost));
}

void mlp_forward(const vtm_mlp* m, const float* X, float* y, int64_t n, cudaStream_t st) {
  if (n <= 0) return;
  // three CTAs per SM, fewer where the samples do not fill them
  const int64_t ctas = (n + 16 * (kFwdThreads / 32) - 1) / (16 * (kFwdThreads / 32));
  int dev = 0, nsm = 1;
  MLP_CUDA(cudaGetDevice(&dev));
  MLP_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const unsigned grid = (unsigned)std::min<int64_t>(ctas, 3 * nsm);
  if (reinterpret_cast<uintptr_t>(X) % 8 == 0) k_mlp_forward<true><<<grid, kFwdThreads, 0, st>>>(m->wb, X, y, n);
  else k_mlp_forward<false><<<grid, kFwdThreads, 0, st>>>(m->wb, X, y, n);
  MLP_CUDA(cudaGetLastError());
}

float mlp_loss_grad(vtm_mlp* m, const float* X, const float* t, int64_t n, cudaStream_t st) {
  if (n <= 0) fail(VTM_ERR_INVALID, "empty batch");
  const int grid = (int)std::min<int64_t>((n + kTile - 1) / kTile, m->part_ctas);
  const float inv_n = 1.f / (float)n;
  if (reinterpret_cast<uintptr_t>(X) % 8 == 0)
    k_mlp_grad<true><<<grid, kGradThreads, sizeof(GradSmem), st>>>(m->wb, X, t, n, inv_n, m->part);
  else
    k_mlp_grad<false><<<grid, kGradThreads, sizeof(GradSmem), st>>>(m->wb, X, t, n, inv_n, m->part);
  MLP_CUDA(cudaGetLastError());
  k_mlp_reduce<<<(kPart + 31) / 32, 256, 0, st>>>(m->part, grid, m->g, m->loss);
  MLP_CUDA(cudaGetLastError());
  MLP_CUDA(cudaMemcpyAsync(m->h_loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost, st));
  MLP_CUDA(cudaStreamSynchronize(st));
  return *m->h_loss;
}

void mlp_destroy(vtm_mlp* m) { delete m; }

void mlp_adam(vtm_mlp* m, float lr, float b1, float b2, float eps, cudaStream_t st) {
  m->step++;
  const float c1 = 1.f - (float)std::pow((double)b1, (double)m->step);
  const float c2 = 1.f - (float)std::pow((double)b2, (double)m->step);
  k_adam<<<(kParams + 255) / 256, 256, 0, st>>>(m->p, m->m, m->v, m->g, m->wb, kParams, lr, b1, b2, eps, c1, c2);
  MLP_CUDA(cudaGetLastError());
}

}  // namespace vtm
