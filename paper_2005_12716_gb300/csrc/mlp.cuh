// The learned-correction network shared by the training kernels and the fused gather: sizes,
// parameter offsets, the BF16 packed weight layout, GELU, and the per-warp layer step on
// m16n8k16 fragments (see mlp.cu for the network's definition).
#pragma once

#include <cuda_bf16.h>

#include <cstddef>

#include "internal.cuh"
#include "mma.cuh"

namespace swense {
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
// Inference's form, x / (1 + e^{-2u}): the same function in seven instructions instead of twelve and
// without the cancellation; the exponential is one of two (2 log2(e) sqrt(2/pi) folded into the
// polynomial), and an overflowing one gives 0, as it should.
__device__ __forceinline__ float gelu_fast(float x) {
  const float k1 = -2.f * 1.4426950408889634f * 0.7978845608028654f, k3 = k1 * 0.044715f;
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * fmaf(k3, x * x, k1)));
  return __fdividef(x, 1.f + e);
}

// ------------------------------------------------------------------------------ forward
// B fragments of 8 outputs (rows n of W) and 32 (or 16) inputs from k on: the 8 x 8 blocks that the lanes
// of each quarter (half) warp point at, row by row.
__device__ __forceinline__ void load_b32(const __nv_bfloat16* W, int ldw, int lane, unsigned (&b)[4]) {
  const unsigned a = unsigned(__cvta_generic_to_shared(W + (lane & 7) * ldw + 8 * (lane >> 3)));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(a));
}
__device__ __forceinline__ void load_b16(const __nv_bfloat16* W, int ldw, int lane, unsigned (&b)[2]) {
  const unsigned a = unsigned(__cvta_generic_to_shared(W + (lane & 7) * ldw + 8 * ((lane >> 3) & 1)));
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(b[0]), "=r"(b[1]) : "r"(a));
}

// Layer with K = 16 * KS inputs held as A fragments (hi and optional lo), N = 8 * NT outputs; W in
// shared memory, rows 16-byte aligned.
template <int KS, int NT, bool SPLIT>
__device__ __forceinline__ void layer(float (&z)[NT][4], const unsigned (&ahi)[KS][4],
                                      const unsigned (&alo)[KS][4], const __nv_bfloat16* W, int ldw,
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
      mma16816(z[nt], ahi[kk], b[0], b[1]);
      if (SPLIT) mma16816(z[nt], alo[kk], b[0], b[1]);
      mma16816(z[nt], ahi[kk + 1], b[2], b[3]);
      if (SPLIT) mma16816(z[nt], alo[kk + 1], b[2], b[3]);
    }
    if constexpr (KS & 1) {
      unsigned b[2];
      load_b16(wr + 16 * (KS - 1), ldw, lane, b);
      mma16816(z[nt], ahi[KS - 1], b[0], b[1]);
      if (SPLIT) mma16816(z[nt], alo[KS - 1], b[0], b[1]);
    }
  }
}

// Accumulator fragments (16 x 8*NT, FP32) -> A fragments (16 x 16*NT/2) after GELU: hi and lo halves for
// inference, BF16 for training.
template <int NT, bool SPLIT>
__device__ __forceinline__ void to_a(const float (&z)[NT][4], unsigned (&ahi)[NT / 2][4],
                                     unsigned (&alo)[NT / 2][4]) {
#pragma unroll
  for (int kk = 0; kk < NT / 2; ++kk) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float* c = z[2 * kk + h];
      auto act = [](float x) { return SPLIT ? gelu_fast(x) : gelu(x); };
      const float g0 = act(c[0]), g1 = act(c[1]), g2 = act(c[2]), g3 = act(c[3]);
      if (SPLIT) {
        bf2_split(g0, g1, ahi[kk][2 * h], alo[kk][2 * h]);
        bf2_split(g2, g3, ahi[kk][2 * h + 1], alo[kk][2 * h + 1]);
      } else {
        ahi[kk][2 * h] = bf2(g0, g1);
        ahi[kk][2 * h + 1] = bf2(g2, g3);
      }
    }
  }
}


}  // namespace mlpnet
}  // namespace swense
