// Incident VOF fraction and relaxation-zone blending on CFD cells.
//
// Paper: subsection on the prevention of wave reflections with the relaxation zone technique.
// A cell's relaxation weight is w = -2x^3 + 3x^2 (Eq. weightFunction) of its non-dimensional
// distance x into a zone; the complementary velocity is blended to zero (Eq. swUcRelax) and the
// VOF fraction to the incident one (Eq. swVOFRelax), both instances of Eq. relaxationZone. The
// incident fraction alpha_I comes from the incident elevation eta_I (reconstruction section,
// interpolation step): the surface is taken as horizontal across the cell at eta_I of its centre,
// and alpha_I is the part of the cell's vertical extent below it.
//
// Cells over threads, four neighbours per thread; the zones are a kernel parameter. Cells
// outside every zone (w = 0) keep alpha and u_C as they are and are not rewritten, so the kernel
// writes little beyond alpha_I in the body of the domain.
#include <algorithm>
#include <cmath>

#include "internal.cuh"

namespace swense {
namespace {

struct Zones {
  int n;
  int kind[SWENSE_MAX_ZONES];
  float inner[SWENSE_MAX_ZONES], inv_len[SWENSE_MAX_ZONES], cx[SWENSE_MAX_ZONES], cy[SWENSE_MAX_ZONES];
};

// clamp to [0, 1] that keeps NaN
__device__ __forceinline__ float unit_clamp(float x) { return x < 0.f ? 0.f : (x > 1.f ? 1.f : x); }

// Weights of N cells side by side: a zone's parameters and kind are looked up once for all of them, and
// their square roots do not wait on one another.
template <int N>
__device__ __forceinline__ void zone_weights(const Zones& Z, const float (&x)[N], const float (&y)[N], float (&w)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) w[i] = 0.f;
  for (int k = 0; k < Z.n; ++k) {
    const int kind = Z.kind[k];
    const float cx = Z.cx[k], cy = Z.cy[k], inner = Z.inner[k], inv_len = Z.inv_len[k];
    float s[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (kind == SWENSE_ZONE_X) s[i] = x[i];
      else if (kind == SWENSE_ZONE_Y) s[i] = y[i];
      else s[i] = sqrtf((x[i] - cx) * (x[i] - cx) + (y[i] - cy) * (y[i] - cy));
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float xn = unit_clamp((s[i] - inner) * inv_len);
      w[i] = fmaxf(w[i], xn * xn * (3.f - 2.f * xn));
    }
  }
}

// One cell of weight w: alpha_I, and in a zone the blends in place.
__device__ __forceinline__ float cell_fraction(float2 ze, float e) { return unit_clamp((e - ze.x) / (ze.y - ze.x)); }
__device__ __forceinline__ float blend(float w, float ai, float alpha) { return fmaf(w, ai, (1.f - w) * alpha); }
__device__ __forceinline__ float relax_cell(int64_t c, float w, float2 ze, float e, float* __restrict__ alpha,
                                            float* __restrict__ uc) {
  const float ai = cell_fraction(ze, e);
  if (w > 0.f) {
    const float keep = 1.f - w;
    if (alpha) alpha[c] = blend(w, ai, alpha[c]);
    if (uc) {
      uc[3 * c] *= keep;
      uc[3 * c + 1] *= keep;
      uc[3 * c + 2] *= keep;
    }
  }
  return ai;
}

// The blends of four neighbouring cells (16-byte aligned arrays), read as whole words, all of them before any
// is used; written as words where all four lie in a zone, else one by one, since cells outside are not written.
__device__ __forceinline__ void blend_cells(int64_t c, const float (&w)[4], float4 ai, float* __restrict__ alpha,
                                            float* __restrict__ uc) {
  float al[4], u[12];
  float4* pa = reinterpret_cast<float4*>(alpha + c);
  float4* pu = reinterpret_cast<float4*>(uc + 3 * c);
  if (alpha) *reinterpret_cast<float4*>(al) = *pa;
  if (uc) {
#pragma unroll
    for (int i = 0; i < 3; ++i) *reinterpret_cast<float4*>(u + 4 * i) = pu[i];
  }
  const float a4[4] = {ai.x, ai.y, ai.z, ai.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    al[i] = blend(w[i], a4[i], al[i]);
#pragma unroll
    for (int d = 0; d < 3; ++d) u[3 * i + d] *= 1.f - w[i];
  }
  if (w[0] > 0.f && w[1] > 0.f && w[2] > 0.f && w[3] > 0.f) {
    if (alpha) *pa = *reinterpret_cast<float4*>(al);
    if (uc) {
#pragma unroll
      for (int i = 0; i < 3; ++i) pu[i] = *reinterpret_cast<float4*>(u + 4 * i);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (!(w[i] > 0.f)) continue;
    if (alpha) alpha[c + i] = al[i];
    if (uc) {
#pragma unroll
      for (int d = 0; d < 3; ++d) uc[3 * (c + i) + d] = u[3 * i + d];
    }
  }
}

// Four cells a thread, 1024 a block. VEC (16-byte aligned arrays): neighbours, as whole 16-byte words, six loads
// and two stores for 128 bytes, where a cell at a time read x and y as scalars 12 bytes apart; in a zone the
// blends are four more of each. Else cells a block's width apart, all their loads before any is used.
// 2,048,000 cells, four zones: 16 us in mesh order with 44 % of the cells in a zone (23.5 a cell at a time),
// 22.7 in no order with 60 % (21.4; 32.2 with the blends a cell after the other, 48 bytes apart).
template <bool VEC>
__global__ void __launch_bounds__(256) k_relax_cells(const float* __restrict__ xyz,
                                                     const float2* __restrict__ zext,
                                                     const float* __restrict__ eta, int64_t nc,
                                                     Zones Z, float* __restrict__ alpha_i,
                                                     float* __restrict__ alpha,
                                                     float* __restrict__ uc,
                                                     float* __restrict__ weight) {
  const int64_t stride = 4 * int64_t(gridDim.x) * blockDim.x;
  for (int64_t c0 = 4 * int64_t(blockIdx.x) * blockDim.x; c0 < nc; c0 += stride) {
    const int64_t c = c0 + 4 * threadIdx.x;
    if (VEC && c + 4 <= nc) {
      const float4* p = reinterpret_cast<const float4*>(xyz + 3 * c);
      const float4* q = reinterpret_cast<const float4*>(zext + c);
      const float4 p0 = __ldg(&p[0]), p1 = __ldg(&p[1]), p2 = __ldg(&p[2]), q0 = __ldg(&q[0]), q1 = __ldg(&q[1]);
      const float4 e = __ldg(reinterpret_cast<const float4*>(eta + c));
      const float x[4] = {p0.x, p0.w, p1.z, p2.y}, y[4] = {p0.y, p1.x, p1.w, p2.z};
      float w[4];
      zone_weights<4>(Z, x, y, w);
      float4 ai;
      ai.x = cell_fraction(make_float2(q0.x, q0.y), e.x);
      ai.y = cell_fraction(make_float2(q0.z, q0.w), e.y);
      ai.z = cell_fraction(make_float2(q1.x, q1.y), e.z);
      ai.w = cell_fraction(make_float2(q1.z, q1.w), e.w);
      if ((w[0] > 0.f || w[1] > 0.f || w[2] > 0.f || w[3] > 0.f) && (alpha || uc)) blend_cells(c, w, ai, alpha, uc);
      if (alpha_i) *reinterpret_cast<float4*>(alpha_i + c) = ai;
      if (weight) *reinterpret_cast<float4*>(weight + c) = make_float4(w[0], w[1], w[2], w[3]);
      continue;
    }
    // VEC: the last cells, fewer than four; else the thread's four of the block's 1024
    const int64_t k0 = VEC ? c : c0 + threadIdx.x, step = VEC ? 1 : blockDim.x;
    float x[4], y[4], e[4], w[4];
    float2 ze[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t k = k0 + i * step < nc ? k0 + i * step : nc - 1;   // in-bounds repeat past the end, unused
      x[i] = __ldg(&xyz[3 * k]);
      y[i] = __ldg(&xyz[3 * k + 1]);
      ze[i] = __ldg(&zext[k]);
      e[i] = __ldg(&eta[k]);
    }
    zone_weights<4>(Z, x, y, w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t k = k0 + i * step;
      if (k >= nc) break;
      const float ai = relax_cell(k, w[i], ze[i], e[i], alpha, uc);
      if (alpha_i) alpha_i[k] = ai;
      if (weight) weight[k] = w[i];
    }
  }
}

}  // namespace
}  // namespace swense

using namespace swense;

extern "C" int swense_relax_cells(const float* cell_xyz, const float* cell_zext, const float* eta_c,
                                  int64_t nc, const swense_relax_zone* zones, int32_t n_zones,
                                  float* alpha_i, float* alpha, float* u_c, float* weight,
                                  void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (nc < 0) return fail(SWENSE_ERR_ARG, "negative cell count");
  if (n_zones < 0 || n_zones > SWENSE_MAX_ZONES)
    return fail(SWENSE_ERR_ARG, "n_zones must lie in 0..SWENSE_MAX_ZONES");
  if (n_zones > 0 && !zones) return fail(SWENSE_ERR_ARG, "NULL zones");
  Zones Z{};
  Z.n = n_zones;
  for (int k = 0; k < n_zones; ++k) {
    const swense_relax_zone& z = zones[k];
    if (z.kind != SWENSE_ZONE_X && z.kind != SWENSE_ZONE_Y && z.kind != SWENSE_ZONE_RADIAL)
      return fail(SWENSE_ERR_ARG, "unknown zone kind");
    if (!(std::isfinite(z.inner) && std::isfinite(z.outer)) || z.inner == z.outer)
      return fail(SWENSE_ERR_ARG, "zone boundaries must be finite and distinct");
    Z.kind[k] = z.kind;
    Z.inner[k] = z.inner;
    Z.inv_len[k] = float(1.0 / (double(z.outer) - double(z.inner)));
    Z.cx[k] = z.cx;
    Z.cy[k] = z.cy;
  }
  if (nc == 0) return SWENSE_OK;
  if (!cell_xyz || !cell_zext || !eta_c) return fail(SWENSE_ERR_ARG, "NULL input");
  if (reinterpret_cast<uintptr_t>(cell_zext) & 7) return fail(SWENSE_ERR_ARG, "cell_zext must be 8-byte aligned");
  const uintptr_t all = reinterpret_cast<uintptr_t>(cell_xyz) | reinterpret_cast<uintptr_t>(cell_zext) |
                        reinterpret_cast<uintptr_t>(eta_c) | reinterpret_cast<uintptr_t>(alpha_i) |
                        reinterpret_cast<uintptr_t>(weight) | reinterpret_cast<uintptr_t>(alpha) |
                        reinterpret_cast<uintptr_t>(u_c);
  const bool vec = (all & 15) == 0;
  const int threads = 256;
  const int64_t blocks = std::min<int64_t>((nc + 4 * threads - 1) / (4 * threads), int64_t(1) << 30);
  const float2* ze = reinterpret_cast<const float2*>(cell_zext);
  if (vec) k_relax_cells<true><<<unsigned(blocks), threads, 0, stream>>>(cell_xyz, ze, eta_c, nc, Z, alpha_i, alpha, u_c, weight);
  else k_relax_cells<false><<<unsigned(blocks), threads, 0, stream>>>(cell_xyz, ze, eta_c, nc, Z, alpha_i, alpha, u_c, weight);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}
