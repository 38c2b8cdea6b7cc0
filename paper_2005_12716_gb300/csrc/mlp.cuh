// The learned-correction network shared by the training kernels and the fused gather: sizes,
// parameter offsets, the BF16 packed weight layout, GELU, and the per-warp layers of training and
// plain inference on m16n8k16 fragments (see mlp.cu for the network's definition).
#pragma once

#include <cuda_bf16.h>

#include <cstddef>

#include "internal.cuh"
#include "mma.cuh"

namespace swense {

// The error flag of the learned gather's bounded waits (as grid_async_flag).
int learned_async_flag(bool reset, int* was_set);

namespace mlpnet {

constexpr int NIN = 67, KIN = 80, NH = 64, NOUT = 4, NO = 8, XLD = 68;
constexpr int OFF_W1 = 0, OFF_B1 = NH * NIN, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NOUT * NH, NPARAM = OFF_B3 + NOUT;
static_assert(NPARAM == SWENSE_MLP_NPARAM, "parameter count");

// BF16 copies of the weights in the layouts the MMAs read, plus FP32 biases. The forward part
// comes first (PackedFwd is a prefix of Packed), so inference kernels copy only that.
struct Packed {
  __nv_bfloat16 w1[NH][KIN];    // B of layer 1: [n = hidden][k = input], inputs 67..79 zero
  __nv_bfloat16 w2[NH][NH];     // B of layer 2: [n][k]
  __nv_bfloat16 w3[NO][NH];     // B of layer 3: rows 4..7 zero
  float b1[NH], b2[NH], b3[NO];
  float out_scale;              // inference output multiplier (training targets were divided by it)
  float pad_[3];
  __nv_bfloat16 w2t[NH][NH];    // W2 transposed (backward)
  __nv_bfloat16 w3t[NH][16];    // W3 transposed, k padded to 16 (backward)
};
struct PackedFwd {
  __nv_bfloat16 w1[NH][KIN];
  __nv_bfloat16 w2[NH][NH];
  __nv_bfloat16 w3[NO][NH];
  float b1[NH], b2[NH], b3[NO];
  float out_scale;
  float pad_[3];
};
static_assert(offsetof(Packed, w2t) == sizeof(PackedFwd) && offsetof(Packed, out_scale) == offsetof(PackedFwd, out_scale) &&
              offsetof(Packed, b1) == offsetof(PackedFwd, b1), "PackedFwd is a prefix of Packed");
static_assert(sizeof(PackedFwd) % 16 == 0, "forward part is copied in 16-byte words");
static_assert(sizeof(Packed) <= SWENSE_MLP_PACKED_BYTES, "packed weight size");
static_assert(sizeof(Packed) % 16 == 0, "packed weight size must be a multiple of 16 bytes");

__device__ __forceinline__ unsigned ld_u32(const __nv_bfloat16* p) {
  return *reinterpret_cast<const unsigned*>(p);
}

// GELU, tanh form: 0.5 x (1 + tanh(u)), u = sqrt(2/pi) (x + 0.044715 x^3). Training's form, with
// tanh(u) = 1 - 2 / (1 + e^{2u}) (saturates correctly at both ends; absolute error ~1e-7 near
// u = 0, far below the BF16 operands it feeds): its activations are rounded to BF16, where another
// form's last bit can flip a rounding, and a run goes on from an older checkpoint bit for bit.
__device__ __forceinline__ float gelu_tanh_u(float x) {
  const float c = 0.7978845608028654f;
  const float u = c * fmaf(0.044715f * x, x * x, x);
  return 1.f - __fdividef(2.f, 1.f + __expf(2.f * u));
}
__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + gelu_tanh_u(x)); }
__device__ __forceinline__ float gelu_grad(float x) {
  const float c = 0.7978845608028654f;
  const float t = gelu_tanh_u(x);
  return 0.5f * (1.f + t) + 0.5f * x * (1.f - t * t) * c * fmaf(3.f * 0.044715f, x * x, 1.f);
}
// Inference's form, x / (1 + e^{-2u}): the same function without the cancellation, of two values side by
// side in nine instructions; the exponential is one of two (2 log2(e) sqrt(2/pi) folded into the
// polynomial), and an overflowing one gives 0, as it should.
__device__ __forceinline__ float2 gelu_fast2(float2 x) {
  const float k1 = -2.f * 1.4426950408889634f * 0.7978845608028654f, k3 = k1 * 0.044715f;
  const float2 w = pmul(x, pfma(make_float2(k3, k3), pmul(x, x), make_float2(k1, k1)));
  float2 e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(w.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(w.y));
  const float2 d = cadd(e, make_float2(1.f, 1.f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
  return pmul(x, r);
}

// ------------------------------------------------------------------------------ forward
// B fragments of 8 outputs (rows n of W) and 32 (or 16) inputs from k on: the 8 x 8 blocks that the lanes
// of each quarter (half) warp point at, row by row.
__device__ __forceinline__ void ldmatrix4(const __nv_bfloat16* p, unsigned (&b)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(unsigned(__cvta_generic_to_shared(p))));
}
__device__ __forceinline__ void load_b32(const __nv_bfloat16* W, int ldw, int lane, unsigned (&b)[4]) {
  ldmatrix4(W + (lane & 7) * ldw + 8 * (lane >> 3), b);
}
__device__ __forceinline__ void load_b16(const __nv_bfloat16* W, int ldw, int lane, unsigned (&b)[2]) {
  const unsigned a = unsigned(__cvta_generic_to_shared(W + (lane & 7) * ldw + 8 * ((lane >> 3) & 1)));
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(b[0]), "=r"(b[1]) : "r"(a));
}
// Fragments of two blocks of 8 outputs and 8 inputs.
__device__ __forceinline__ void load_b8x2(const __nv_bfloat16* W, int ldw, int lane, unsigned (&b)[2]) {
  const unsigned a = unsigned(__cvta_generic_to_shared(W + (lane & 15) * ldw));
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(b[0]), "=r"(b[1]) : "r"(a));
}

// Layer with K = 16 * KS inputs held as A fragments, N = 8 * NT outputs; W in shared memory, rows 16-byte
// aligned.
template <int KS, int NT>
__device__ __forceinline__ void layer(float (&z)[NT][4], const unsigned (&a)[KS][4], const __nv_bfloat16* W, int ldw,
                                      const float* bias, int lane) {
  const int t = lane & 3;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const float2 bb = *reinterpret_cast<const float2*>(&bias[8 * nt + 2 * t]);
    z[nt][0] = bb.x;
    z[nt][1] = bb.y;
    z[nt][2] = bb.x;
    z[nt][3] = bb.y;
    const __nv_bfloat16* wr = W + 8 * nt * ldw;
#pragma unroll
    for (int kk = 0; kk + 1 < KS; kk += 2) {
      unsigned b[4];
      load_b32(wr + 16 * kk, ldw, lane, b);
      mma16816(z[nt], a[kk], b[0], b[1]);
      mma16816(z[nt], a[kk + 1], b[2], b[3]);
    }
    if constexpr (KS & 1) {
      unsigned b[2];
      load_b16(wr + 16 * (KS - 1), ldw, lane, b);
      mma16816(z[nt], a[KS - 1], b[0], b[1]);
    }
  }
}

// Accumulator fragments (16 x 8*NT, FP32) -> A fragments (16 x 16*NT/2) after GELU, in BF16.
template <int NT>
__device__ __forceinline__ void to_a(const float (&z)[NT][4], unsigned (&a)[NT / 2][4]) {
#pragma unroll
  for (int kk = 0; kk < NT / 2; ++kk) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float* c = z[2 * kk + h];
      a[kk][2 * h] = bf2(gelu(c[0]), gelu(c[1]));
      a[kk][2 * h + 1] = bf2(gelu(c[2]), gelu(c[3]));
    }
  }
}

// ------------------------------------------------------------------------------ inference
// Inputs and activations in two BF16 halves (hi + lo). The three offsets that follow the 64 stencil values
// fill one step of eight inputs with both their halves (dx, dy, dz, then the low halves, then zeros)
// against a copy of W1 whose inputs 64..66 stand again at 67..69 (repeat_offsets): half a step where hi and
// lo of a padded one would be two.
__device__ __forceinline__ unsigned offsets_a(float dx, float dy, float dz, int q) {
  unsigned h, l, hz, lz;
  bf2_split(dx, dy, h, l);
  bf2_split(dz, 0.f, hz, lz);
  return q == 0 ? h : q == 1 ? (hz & 0xffffu) | (l << 16) : q == 2 ? (l >> 16) | (lz << 16) : 0u;
}
__device__ __forceinline__ uint4 repeat_offsets(uint4 w) {   // w: a row's inputs 64..71 in BF16
  return make_uint4(w.x, (w.y & 0xffffu) | (w.x << 16), (w.x >> 16) | (w.y << 16), w.w);
}

// Two blocks of 8 outputs at a time, n0 on, of a layer: the two blocks are the next layer's k-step.
template <int KS>
__device__ __forceinline__ void outputs16(float (&z)[2][4], const unsigned (&ahi)[KS][4], const unsigned (&alo)[KS][4],
                                          const __nv_bfloat16* W, int ldw, const float* bias, int n0, int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float2 bb = *reinterpret_cast<const float2*>(&bias[n0 + 8 * i + 2 * (lane & 3)]);
    z[i][0] = bb.x;
    z[i][1] = bb.y;
    z[i][2] = bb.x;
    z[i][3] = bb.y;
  }
  // lanes 0..15 point at the rows of the first block (their two halves of 8 inputs), 16..31 at the second's
  const __nv_bfloat16* wr = W + (n0 + (lane & 7) + 8 * (lane >> 4)) * ldw + 8 * ((lane >> 3) & 1);
#pragma unroll
  for (int kk = 0; kk < KS; ++kk) {
    unsigned b[4];
    ldmatrix4(wr + 16 * kk, b);
    mma16816(z[0], ahi[kk], b[0], b[1]);
    mma16816(z[1], ahi[kk], b[2], b[3]);
    mma16816(z[0], alo[kk], b[0], b[1]);
    mma16816(z[1], alo[kk], b[2], b[3]);
  }
}

__device__ __forceinline__ void activate(const float (&z)[2][4], unsigned (&hi)[4], unsigned (&lo)[4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    bf2_split(gelu_fast2(make_float2(z[h][0], z[h][1])), hi[2 * h], lo[2 * h]);
    bf2_split(gelu_fast2(make_float2(z[h][2], z[h][3])), hi[2 * h + 1], lo[2 * h + 1]);
  }
}

// The three layers of 16 rows (xo: offsets_a of rows g and g + 8). The MMAs of the next 16 outputs stand
// between a block's own and its activation, which hides part of either.
template <class Weights>
__device__ __forceinline__ void infer(float (&o)[4], const unsigned (&xh)[4][4], const unsigned (&xl)[4][4],
                                      const unsigned (&xo)[2], const Weights& W, int ld1, int ld2, int lane) {
  unsigned h1h[4][4], h1l[4][4];
  float z[2][2][4];
  auto layer1 = [&](int g) {
    outputs16<4>(z[g & 1], xh, xl, &W.w1[0][0], ld1, W.b1, 16 * g, lane);
    unsigned b[2];
    load_b8x2(&W.w1[16 * g][64], ld1, lane, b);
    mma1688(z[g & 1][0], xo, b[0]);
    mma1688(z[g & 1][1], xo, b[1]);
  };
  auto layer2 = [&](int g) { outputs16<4>(z[g & 1], h1h, h1l, &W.w2[0][0], ld2, W.b2, 16 * g, lane); };
  layer1(0);
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if (g < 3) layer1(g + 1);
    activate(z[g & 1], h1h[g], h1l[g]);
  }
  const float2 bb = *reinterpret_cast<const float2*>(&W.b3[2 * (lane & 3)]);
  o[0] = o[2] = bb.x;
  o[1] = o[3] = bb.y;
  layer2(0);
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if (g < 3) layer2(g + 1);
    unsigned hi[4], lo[4], b[2];
    activate(z[g & 1], hi, lo);
    load_b16(&W.w3[0][16 * g], ld2, lane, b);
    mma16816(o, hi, b[0], b[1]);
    mma16816(o, lo, b[0], b[1]);
  }
}

}  // namespace mlpnet
}  // namespace swense
