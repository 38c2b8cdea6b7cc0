// Shared-memory inverse DFT (sign +, unnormalised) used by the grid reconstruction kernels.
//
// Iterative Cooley-Tukey decimation in time, in place: the caller scatters each length-n input
// into bit-reversed positions; the stages then combine sub-transforms of length h into 4h
// (two radix-2 stages fused in registers, three twiddle products), preceded by one radix-2 stage
// when log2(n) is odd. Output is in natural order. `batch` arrays of length n lie back to back.
#pragma once

#include "internal.cuh"

namespace swense {

// tw[j] = e^{+2 pi i j / SWENSE_MAX_FFT}
__device__ __forceinline__ void fft_inv_inplace(float2* data, int n, int log2n, int batch,
                                                const float2* __restrict__ tw) {
  const int nthr = blockDim.x;
  int h = 1;
  if (log2n & 1) {
    const int half = n >> 1;
    for (int t = threadIdx.x; t < batch * half; t += nthr) {
      const int b = t / half, j = t - b * half;
      float2* a = data + size_t(b) * n + 2 * j;
      const float2 x0 = a[0], x1 = a[1];
      a[0] = cadd(x0, x1);
      a[1] = csub(x0, x1);
    }
    h = 2;
    __syncthreads();
  }
  const int quarter = n >> 2;
  for (; h < n; h <<= 2) {
    const int s1 = SWENSE_MAX_FFT / (2 * h);  // twiddle stride of the length-2h stage
    const int s2 = s1 >> 1;                   // ... of the length-4h stage
    for (int t = threadIdx.x; t < batch * quarter; t += nthr) {
      const int b = t / quarter, r = t - b * quarter;
      const int g = r / h, j = r - g * h;
      float2* a = data + size_t(b) * n + g * 4 * h + j;
      const float2 w1 = __ldg(&tw[j * s1]);
      const float2 w2 = __ldg(&tw[j * s2]);
      const float2 x0 = a[0], x1 = a[h], x2 = a[2 * h], x3 = a[3 * h];
      const float2 t1 = cmul(w1, x1);
      const float2 a0 = cadd(x0, t1), a1 = csub(x0, t1);
      const float2 t3 = cmul(w1, x3);
      const float2 a2 = cadd(x2, t3), a3 = csub(x2, t3);
      const float2 t2 = cmul(w2, a2);
      const float2 u = cmul_i(cmul(w2, a3));
      a[0] = cadd(a0, t2);
      a[2 * h] = csub(a0, t2);
      a[h] = cadd(a1, u);
      a[3 * h] = csub(a1, u);
    }
    __syncthreads();
  }
}

// Depth factors of the spectral decomposition at vertical position z for |k| = k:
//   finite depth h > 0: F = cosh(k(z+h))/cosh(kh), S = sinh(k(z+h))/cosh(kh), written as
//     (e^{kz} +- e^{-k(z+2h)}) / (1 + e^{-2kh}) so that no term overflows;
//   deep water (h <= 0): F = S = e^{kz}.
// k*z is formed as an unevaluated sum hi + lo (fma residual) so the factor keeps FP32 accuracy
// for the large |k z| of the levels above z = 0.
__device__ __forceinline__ void depth_factors(float k, float z, float h, float& F, float& S) {
  const float kz = k * z;
  const float kz_lo = fmaf(k, z, -kz);
  float e1 = expf(kz);
  e1 = fmaf(e1, kz_lo, e1);
  if (h <= 0.f) {
    F = e1;
    S = e1;
    return;
  }
  const float e2 = expf(-k * (z + 2.f * h));
  const float d = 1.f + expf(-2.f * k * h);
  F = (e1 + e2) / d;
  S = (e1 - e2) / d;
}

// Prefilter of the periodic cubic-spline scheme. The spline interpolating grid values f_i is
// sum_j c_j B3(x/h - j) with (c_{i-1} + 4 c_i + c_{i+1}) / 6 = f_i; for one Fourier mode this
// divides its amplitude by the symbol (2 + cos(2 pi j / N)) / 3 of that averaging, per axis. So
// B-spline coefficients on the grid are the inverse transform of the modes divided by the
// symbols: 1 / prod over the horizontal axes, for signed mode j on an axis of N refined nodes.
__device__ __forceinline__ float spline_prefilter(int m, int Nx, int n, int Ny) {
  float f = 3.f / (2.f + cospif(2.f * float(m) / float(Nx)));
  if (Ny > 1) f *= 3.f / (2.f + cospif(2.f * float(n) / float(Ny)));
  return f;
}

}  // namespace swense

namespace swense {

// ------------------------------------------------------------------------------------------------
// Per-warp Stockham inverse DFT of length N = 32 E (8 <= E <= 64), radix-8 passes followed by one
// radix-4 or radix-2 pass when log2 N is not a multiple of 3 (Stockham autosort: natural order in
// and out). Butterfly j of a pass with radix R after NS points have been combined reads
// x[j + r N/R], multiplies by e^{2 pi i (j mod NS) r / (NS R)}, takes the length-R DFT and writes
// y[(j / NS) NS R + (j mod NS) + r NS]. Lane l owns butterflies j = l + 32 b. Between passes the
// data go through a warp-private shared buffer with one pad element per 16 (index i + i/16),
// which keeps every exchange at the 2-wavefront minimum; the first pass reads registers filled
// by the caller (element b*8 + r holds position l + 32 b + r N/8) and the last pass leaves
// element b*R + r holding output position l + 32 b + r N/R (coalesced stores).

constexpr int stk_l2(int n) { return n <= 1 ? 0 : 1 + stk_l2(n >> 1); }
constexpr int stk_npass(int n) { return stk_l2(n) / 3 + (stk_l2(n) % 3 != 0 ? 1 : 0); }
constexpr int stk_radix(int n, int p) {
  return p < stk_l2(n) / 3 ? 8 : (stk_l2(n) % 3 == 1 ? 2 : 4);
}
constexpr int stk_ns(int n, int p) { return p == 0 ? 1 : stk_ns(n, p - 1) * stk_radix(n, p - 1); }
// distinct values of (j mod NS) among one lane's butterflies of pass p
constexpr int stk_dist(int n, int p) {
  return stk_ns(n, p) <= 32 ? 1
                            : (stk_ns(n, p) / 32 < n / 32 / stk_radix(n, p) ? stk_ns(n, p) / 32
                                                                            : n / 32 / stk_radix(n, p));
}
constexpr int stk_twoff(int n, int p) {
  return p <= 1 ? 0 : stk_twoff(n, p - 1) + stk_dist(n, p - 1) * (stk_radix(n, p - 1) - 1);
}
// passes 1 .. stk_regpass - 1 keep their twiddles in registers; later passes read the pass-major
// tables below (L1)
constexpr int stk_regpass(int n) { return n <= 256 ? stk_npass(n) : 2; }
constexpr int stk_twn(int n) { return stk_twoff(n, stk_regpass(n)) > 0 ? stk_twoff(n, stk_regpass(n)) : 1; }
constexpr int stk_buf(int n) { return n + n / 16; }   // padded buffer length (float2)

// Pass-major twiddles. Pass p >= 1 of an N-point transform (stride NS, radix R) multiplies by
// e^{+2 pi i jm r / (NS R)}, jm < NS, 0 < r < R. In the plain table that factor sits at
// jm r SWENSE_MAX_FFT / (NS R), so the lanes of a warp (consecutive jm) read entries r
// SWENSE_MAX_FFT / (NS R) apart: up to one L1 wavefront per lane. The twiddle array therefore also
// holds each factor at stk_twp(N, p) + (r - 1) NS + jm, where consecutive lanes read consecutive
// entries (2 wavefronts a warp). The tables of an N-point transform fill [SWENSE_MAX_FFT + N,
// SWENSE_MAX_FFT + 2 N): pass q holds NS_q (R_q - 1) = NS_{q+1} - NS_q entries, so pass p starts
// NS_p - NS_1 entries in.
constexpr int stk_twp(int n, int p) { return SWENSE_MAX_FFT + n + stk_ns(n, p) - stk_ns(n, 1); }
constexpr int kTwiddleLen = 3 * SWENSE_MAX_FFT;       // plain table + pass-major tables

// Exponent e of entry j of the twiddle array (the entry is e^{+2 pi i e / SWENSE_MAX_FFT}): j in
// the plain table; in the pass-major tables, jm r SWENSE_MAX_FFT / (NS R) of the transform size,
// pass, r and jm that slot j stands for; 0 in the slots no pass uses.
__host__ __device__ constexpr int twiddle_exponent(int j) {
  if (j < SWENSE_MAX_FFT) return j;
  const int i = j - SWENSE_MAX_FFT;
  int n = 1;
  while (2 * n <= i) n *= 2;                       // slot i lies in [n, 2n): the tables of size n
  int ns = stk_radix(n, 0);                        // stride NS_1 of pass 1
  const int o = i - n + ns;                        // pass p holds NS_p <= o < NS_{p+1}
  for (int p = 1; p < stk_npass(n); ++p) {
    const int R = stk_radix(n, p);
    if (o < ns * R) {
      const int q = o - ns;                        // (r - 1) NS + jm
      return (q % ns) * (q / ns + 1) * (SWENSE_MAX_FFT / (ns * R));
    }
    ns *= R;
  }
  return 0;
}

__device__ __forceinline__ int stk_pad(int i) { return i + (i >> 4); }

// Per-lane twiddles of the register-held passes (kernel-lifetime registers).
// (one template instance per pass, so every register index is a compile-time constant)
template <int N, int P = 1>
__device__ __forceinline__ void stk_init(float2 (&T)[stk_twn(N)], const float2* __restrict__ tw, int lane) {
  if constexpr (P < stk_regpass(N)) {
    constexpr int R = stk_radix(N, P), NS = stk_ns(N, P), D = stk_dist(N, P), OFF = stk_twoff(N, P);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int jm = NS <= 32 ? lane % NS : lane + 32 * d;
#pragma unroll
      for (int r = 1; r < R; ++r) T[OFF + d * (R - 1) + r - 1] = __ldg(&tw[jm * r * (SWENSE_MAX_FFT / (NS * R))]);
    }
    stk_init<N, P + 1>(T, tw, lane);
  }
}

// Inverse DFTs of length 2, 4, 8 in registers (natural order), constants folded.
__device__ __forceinline__ void stk_dft2(float2* v) {
  const float2 a = v[0];
  v[0] = cadd(a, v[1]);
  v[1] = csub(a, v[1]);
}
__device__ __forceinline__ void stk_dft4(float2& a0, float2& a1, float2& a2, float2& a3) {
  const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3);
  const float2 t3 = cmul_i(csub(a1, a3));
  a0 = cadd(t0, t2);
  a2 = csub(t0, t2);
  a1 = cadd(t1, t3);
  a3 = csub(t1, t3);
}
__device__ __forceinline__ void stk_dft8(float2* v) {
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  stk_dft4(e0, e1, e2, e3);
  stk_dft4(o0, o1, o2, o3);
  const float c = 0.70710678118654752f;                         // e^{i pi/4} = c (1 + i)
  o1 = make_float2(c * (o1.x - o1.y), c * (o1.x + o1.y));
  o2 = cmul_i(o2);
  o3 = make_float2(-c * (o3.x + o3.y), c * (o3.x - o3.y));      // e^{3 i pi/4} = c (-1 + i)
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1);
  v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2);
  v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3);
  v[7] = csub(e3, o3);
}

template <int N, int P>
__device__ __forceinline__ void stk_pass(float2 (&v)[N / 32], const float2 (&T)[stk_twn(N)],
                                         const float2* __restrict__ tw, float2* buf, int lane) {
  constexpr int E = N / 32, R = stk_radix(N, P), NS = stk_ns(N, P), B = E / R;
  if constexpr (P > 0 && P < stk_regpass(N)) {
    constexpr int OFF = stk_twoff(N, P);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int d = NS <= 32 ? 0 : b % (NS / 32);
#pragma unroll
      for (int r = 1; r < R; ++r)
        v[b * R + r] = cmul(v[b * R + r], T[OFF + d * (R - 1) + r - 1]);
    }
  } else if constexpr (P > 0) {
    constexpr int TP = stk_twp(N, P);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int jm = NS <= 32 ? lane % NS : lane + 32 * (b % (NS / 32));
#pragma unroll
      for (int r = 1; r < R; ++r) v[b * R + r] = cmul(v[b * R + r], __ldg(&tw[TP + (r - 1) * NS + jm]));
    }
  }
#pragma unroll
  for (int b = 0; b < B; ++b) {
    if constexpr (R == 8) stk_dft8(&v[b * 8]);
    else if constexpr (R == 4) stk_dft4(v[b * 4], v[b * 4 + 1], v[b * 4 + 2], v[b * 4 + 3]);
    else stk_dft2(&v[b * 2]);
  }
  if constexpr (P + 1 < stk_npass(N)) {
    // Output index of (b, r) = lane part + constant part with disjoint bits, so the padded index
    // splits the same way and every access is a per-pass base plus an immediate offset.
    const int lst = NS <= 32 ? (lane / NS) * NS * R + lane % NS : lane;
    float2* bst = buf + stk_pad(lst);
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int c = NS <= 32 ? 32 * b * R + r * NS
                               : (b / (NS / 32)) * NS * R + 32 * (b % (NS / 32)) + r * NS;
        bst[c + (c >> 4)] = v[b * R + r];
      }
    __syncwarp();
    constexpr int R2 = stk_radix(N, P + 1), B2 = E / R2;
    const float2* bld = buf + stk_pad(lane);
#pragma unroll
    for (int b = 0; b < B2; ++b)
#pragma unroll
      for (int r = 0; r < R2; ++r) {
        const int c = 32 * b + r * (N / R2);
        v[b * R2 + r] = bld[c + (c >> 4)];
      }
    __syncwarp();
    stk_pass<N, P + 1>(v, T, tw, buf, lane);
  }
}

// Full transform; see the block comment above for the register layouts in and out.
template <int N>
__device__ __forceinline__ void stk_fft(float2 (&v)[N / 32], const float2 (&T)[stk_twn(N)],
                                        const float2* __restrict__ tw, float2* buf, int lane) {
  static_assert(N >= 256 && N <= 2048, "per-warp Stockham sizes");
  stk_pass<N, 0>(v, T, tw, buf, lane);
}

}  // namespace swense

namespace swense {

// ------------------------------------------------------------------------------------------------
// Block-wide Stockham inverse DFT of length N by TH threads (E = N / TH >= 8 elements each), the
// same radix-8 (then 4 or 2) passes as stk_fft with "lane" generalised to the thread index and
// the exchange through a padded block-shared buffer under __syncthreads. Twiddles come from the
// pass-major tables (L1). Layouts: on entry element b*8 + r of thread t holds position
// t + TH b + r N/8; on exit element b*R + r holds t + TH b + r N/R (R = radix of the last pass).
template <int N, int TH, int P>
__device__ __forceinline__ void stkb_pass(float2 (&v)[N / TH], const float2* __restrict__ tw,
                                          float2* buf, int t) {
  constexpr int E = N / TH, R = stk_radix(N, P), NS = stk_ns(N, P), B = E / R;
  static_assert(B >= 1, "each thread holds at least one butterfly per pass");
  if constexpr (P > 0) {
    constexpr int TP = stk_twp(N, P);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int jm = NS <= TH ? t % NS : t + TH * (b % (NS / TH));
#pragma unroll
      for (int r = 1; r < R; ++r) v[b * R + r] = cmul(v[b * R + r], __ldg(&tw[TP + (r - 1) * NS + jm]));
    }
  }
#pragma unroll
  for (int b = 0; b < B; ++b) {
    if constexpr (R == 8) stk_dft8(&v[b * 8]);
    else if constexpr (R == 4) stk_dft4(v[b * 4], v[b * 4 + 1], v[b * 4 + 2], v[b * 4 + 3]);
    else stk_dft2(&v[b * 2]);
  }
  if constexpr (P + 1 < stk_npass(N)) {
    // thread part and constant part of each index have disjoint bits (as in stk_pass)
    const int lst = NS <= TH ? (t / NS) * NS * R + t % NS : t;
    float2* bst = buf + stk_pad(lst);
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int c = NS <= TH ? TH * b * R + r * NS
                               : (b / (NS / TH)) * NS * R + TH * (b % (NS / TH)) + r * NS;
        bst[c + (c >> 4)] = v[b * R + r];
      }
    __syncthreads();
    constexpr int R2 = stk_radix(N, P + 1), B2 = E / R2;
    const float2* bld = buf + stk_pad(t);
#pragma unroll
    for (int b = 0; b < B2; ++b)
#pragma unroll
      for (int r = 0; r < R2; ++r) {
        const int c = TH * b + r * (N / R2);
        v[b * R2 + r] = bld[c + (c >> 4)];
      }
    __syncthreads();
    stkb_pass<N, TH, P + 1>(v, tw, buf, t);
  }
}

template <int N, int TH>
__device__ __forceinline__ void stkb_fft(float2 (&v)[N / TH], const float2* __restrict__ tw, float2* buf,
                                         int t) {
  static_assert(N / TH >= 8 && N <= SWENSE_MAX_FFT && (TH & 15) == 0, "block Stockham sizes");
  static_assert(N / 8 >= TH, "constant index parts are multiples of the thread count");
  stkb_pass<N, TH, 0>(v, tw, buf, t);
}

// Two block-wide transforms of the same length side by side (buffers buf1, buf2): each pass
// applies to both before the shared barriers, so the pair takes the barriers of one transform
// and twice the independent work between them.
template <int N, int TH, int P>
__device__ __forceinline__ void stkb_pass2(float2 (&v1)[N / TH], float2 (&v2)[N / TH],
                                           const float2* __restrict__ tw, float2* buf1, float2* buf2, int t) {
  constexpr int E = N / TH, R = stk_radix(N, P), NS = stk_ns(N, P), B = E / R;
  if constexpr (P > 0) {
    constexpr int TP = stk_twp(N, P);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int jm = NS <= TH ? t % NS : t + TH * (b % (NS / TH));
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const float2 w = __ldg(&tw[TP + (r - 1) * NS + jm]);
        v1[b * R + r] = cmul(v1[b * R + r], w);
        v2[b * R + r] = cmul(v2[b * R + r], w);
      }
    }
  }
#pragma unroll
  for (int b = 0; b < B; ++b) {
    if constexpr (R == 8) {
      stk_dft8(&v1[b * 8]);
      stk_dft8(&v2[b * 8]);
    } else if constexpr (R == 4) {
      stk_dft4(v1[b * 4], v1[b * 4 + 1], v1[b * 4 + 2], v1[b * 4 + 3]);
      stk_dft4(v2[b * 4], v2[b * 4 + 1], v2[b * 4 + 2], v2[b * 4 + 3]);
    } else {
      stk_dft2(&v1[b * 2]);
      stk_dft2(&v2[b * 2]);
    }
  }
  if constexpr (P + 1 < stk_npass(N)) {
    const int lst = NS <= TH ? (t / NS) * NS * R + t % NS : t;
    float2* bst1 = buf1 + stk_pad(lst);
    float2* bst2 = buf2 + stk_pad(lst);
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int c = NS <= TH ? TH * b * R + r * NS
                               : (b / (NS / TH)) * NS * R + TH * (b % (NS / TH)) + r * NS;
        bst1[c + (c >> 4)] = v1[b * R + r];
        bst2[c + (c >> 4)] = v2[b * R + r];
      }
    __syncthreads();
    constexpr int R2 = stk_radix(N, P + 1), B2 = E / R2;
    const float2* bld1 = buf1 + stk_pad(t);
    const float2* bld2 = buf2 + stk_pad(t);
#pragma unroll
    for (int b = 0; b < B2; ++b)
#pragma unroll
      for (int r = 0; r < R2; ++r) {
        const int c = TH * b + r * (N / R2);
        v1[b * R2 + r] = bld1[c + (c >> 4)];
        v2[b * R2 + r] = bld2[c + (c >> 4)];
      }
    __syncthreads();
    stkb_pass2<N, TH, P + 1>(v1, v2, tw, buf1, buf2, t);
  }
}

template <int N, int TH>
__device__ __forceinline__ void stkb_fft2(float2 (&v1)[N / TH], float2 (&v2)[N / TH],
                                          const float2* __restrict__ tw, float2* buf1, float2* buf2, int t) {
  static_assert(N / TH >= 8 && N <= SWENSE_MAX_FFT && (TH & 15) == 0, "block Stockham sizes");
  static_assert(N / 8 >= TH, "constant index parts are multiples of the thread count");
  stkb_pass2<N, TH, 0>(v1, v2, tw, buf1, buf2, t);
}

}  // namespace swense

namespace swense {

// ------------------------------------------------------------------------------------------------
// Wide-radix inverse DFTs in two or three Stockham passes: N = R0 R1 (R2), with R0 elements a thread.
// A 16- or 32-point DFT in registers replaces two or three radix-8/-4 passes and their exchanges, so a
// transform of up to 1024 points goes through shared memory once and one of 2048 points twice. (Columns
// of 512 and 1024 points as 16 x 16 x N/256, with 24 warps per SM instead of 16 but a second exchange,
// were slower: eight levels of 1024 x 1024 columns 155 against 145 us, 64 of 512 x 512 130 against 101.)
// Pass p with stride NS and radix R: butterfly j reads x[j + r N/R], multiplies by
// e^{2 pi i (j mod NS) r / (NS R)} and writes y[(j / NS) NS R + (j mod NS) + r NS].

// cos(2 pi j / 32)
__host__ __device__ constexpr double root32_cos(int j) {
  j &= 31;
  if (j > 16) j = 32 - j;
  const bool neg = j > 8;
  if (neg) j = 16 - j;
  const double c = j == 0   ? 1.0
                   : j == 1 ? 0.98078528040323044913
                   : j == 2 ? 0.92387953251128675613
                   : j == 3 ? 0.83146961230254523708
                   : j == 4 ? 0.70710678118654752440
                   : j == 5 ? 0.55557023301960222474
                   : j == 6 ? 0.38268343236508977173
                   : j == 7 ? 0.19509032201612826785
                            : 0.0;
  return neg ? -c : c;
}
// v e^{2 pi i j / 32}, j a constant after unrolling
__device__ __forceinline__ float2 rot32(float2 v, int j) {
  j &= 31;
  if (j == 0) return v;
  if (j == 8) return make_float2(-v.y, v.x);
  if (j == 16) return make_float2(-v.x, -v.y);
  if (j == 24) return make_float2(v.y, -v.x);
  const float c = float(root32_cos(j)), s = float(root32_cos(j - 8));
  if (j == 4) return make_float2(c * (v.x - v.y), c * (v.x + v.y));
  if (j == 12) return make_float2(c * (v.x + v.y), c * (v.y - v.x));
  return cmul(v, make_float2(c, s));
}

// In-register DFT of v[0 .. R-1]; X[k] is left in v[dft_slot<R>(k)].
template <int R>
__host__ __device__ constexpr int dft_slot(int k) {
  return R == 32 ? 4 * (k % 8) + k / 8 : R == 16 ? 4 * (k % 4) + k / 4 : k;
}
template <int R>
__device__ __forceinline__ void wide_dft(float2* v) {
  if constexpr (R == 2) {
    stk_dft2(v);
  } else if constexpr (R == 4) {
    stk_dft4(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    stk_dft8(v);
  } else {
    // R = 4 Q, n = n2 + 4 n1, k = k1 + Q k2: Q-point DFTs over n1, twiddles W_R^{n2 k1}, 4-point over n2
    static_assert(R == 16 || R == 32, "register DFT sizes");
    constexpr int Q = R / 4;
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
      if constexpr (Q == 4) {
        stk_dft4(v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]);
      } else {
        float2 t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = v[n2 + 4 * i];
        stk_dft8(t);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[n2 + 4 * i] = t[i];
      }
    }
#pragma unroll
    for (int k1 = 0; k1 < Q; ++k1) {
#pragma unroll
      for (int n2 = 1; n2 < 4; ++n2) v[n2 + 4 * k1] = rot32(v[n2 + 4 * k1], n2 * k1 * (32 / R));
      stk_dft4(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
    }
  }
}

// Factors of the first two passes' product of length N = R0 R1 (32 <= N <= 1024): entry
// kWideTw + N + r R0 + j holds e^{2 pi i j r / N} (j < R0). Third pass (stride 256, radix N / 256,
// N = 512 .. 2048): entry kWideTw3 + N + 256 r + j holds e^{2 pi i j r / N} (j < 256).
// R0 of a column transform; rows use 16 x 16 passes from 256 points on (wide_r0 for N <= 256).
constexpr int wide_r0(int n) { return n >= 512 ? 32 : (n >= 128 ? 16 : 8); }
constexpr int kWideTw = kTwiddleLen, kWideTw3 = kWideTw + 2048, kTwiddleAll = kWideTw3 + 4096;
__host__ __device__ constexpr int wide_exponent(int i) {          // of twiddle entry i >= kWideTw
  const bool third = i >= kWideTw3;
  const int o = i - (third ? kWideTw3 : kWideTw);
  int n = 1;
  while (2 * n <= o) n *= 2;                       // slot o lies in [n, 2n)
  if (n < 32 || n > (third ? 2048 : 1024) || (third && n < 512)) return 0;
  const int q = third ? 256 : wide_r0(n);
  return ((o - n) % q) * ((o - n) / q) * (SWENSE_MAX_FFT / n);
}

// Two row transforms side by side by T = N / R0 threads (t = 0 .. T-1): element e of thread t holds
// position t + T e on entry, and element elem(b, r) position pos(t, b, r) on exit. The buffer is padded
// by one element in R0, which makes every exchange conflict-free.
template <int N>
struct WideRow {
  static constexpr int R0 = N >= 128 ? 16 : 8, R1 = N >= 256 ? 16 : N / R0, R2 = N / (R0 * R1);
  static constexpr int E = R0, T = N / E, RL = R2 > 1 ? R2 : R1, BL = E / RL;
  static constexpr int kBuf = N + N / R0;
  static constexpr int kRows = T >= 128 ? 1 : 128 / T;            // rows per 128-thread block
  __device__ static __forceinline__ int elem(int b, int r) { return b * RL + dft_slot<RL>(r); }
  __device__ static __forceinline__ int pos(int t, int b, int r) { return t + T * b + (N / RL) * r; }
  __device__ static __forceinline__ void sync() {
    if constexpr (T <= 32) __syncwarp();
    else __syncthreads();
  }
  // TWO: a buffer for each transform (b1, b2) and their exchanges side by side; otherwise they take the
  // one buffer b1 in turn: half the shared memory, for two more barriers an exchange.
  template <bool TWO, class Put, class Get>
  __device__ static __forceinline__ void exchange(float2 (&z1)[E], float2 (&z2)[E], float2* b1, float2* b2, Put put,
                                                  Get get) {
    put(z1, b1);
    if constexpr (TWO) put(z2, b2);
    sync();
    get(z1, b1);
    if constexpr (TWO) get(z2, b2);
    sync();
    if constexpr (!TWO) {
      put(z2, b1);
      sync();
      get(z2, b1);
      sync();
    }
  }
  template <bool TWO>
  __device__ static __forceinline__ void fft2(float2 (&z1)[E], float2 (&z2)[E], const float2* __restrict__ tw,
                                              float2* b1, float2* b2, int t) {
    constexpr int B1 = E / R1, S1 = N / R1;        // S1 is a multiple of R0: the pad index splits
    auto put0 = [&](float2 (&z)[E], float2* buf) {
#pragma unroll
      for (int r = 0; r < R0; ++r) buf[t * (R0 + 1) + r] = z[dft_slot<R0>(r)];
    };
    auto get0 = [&](float2 (&z)[E], float2* buf) {
#pragma unroll
      for (int b = 0; b < B1; ++b) {
        const int jj = t + T * b, base = jj + jj / R0;
#pragma unroll
        for (int r = 0; r < R1; ++r) z[b * R1 + r] = buf[base + r * (S1 + S1 / R0)];
      }
    };
    wide_dft<R0>(z1);
    wide_dft<R0>(z2);
    exchange<TWO>(z1, z2, b1, b2, put0, get0);
#pragma unroll
    for (int b = 0; b < B1; ++b) {
      const int jm = (t + T * b) % R0;
#pragma unroll
      for (int r = 1; r < R1; ++r) {
        const float2 w = __ldg(&tw[kWideTw + R0 * R1 + r * R0 + jm]);
        z1[b * R1 + r] = cmul(z1[b * R1 + r], w);
        z2[b * R1 + r] = cmul(z2[b * R1 + r], w);
      }
      wide_dft<R1>(&z1[b * R1]);
      wide_dft<R1>(&z2[b * R1]);
    }
    if constexpr (R2 > 1) {
      static_assert(R2 == 1 || (R0 == 16 && R1 == 16), "three passes start with 16 x 16");
      const int wb = (t / 16) * 272 + t % 16;
      auto put1 = [&](float2 (&z)[E], float2* buf) {
#pragma unroll
        for (int r = 0; r < 16; ++r) buf[wb + 17 * r] = z[dft_slot<16>(r)];
      };
      auto get1 = [&](float2 (&z)[E], float2* buf) {
#pragma unroll
        for (int b = 0; b < BL; ++b) {
          const int jj = t + T * b, base = jj + jj / 16;
#pragma unroll
          for (int r = 0; r < R2; ++r) z[b * R2 + r] = buf[base + 272 * r];
        }
      };
      exchange<TWO>(z1, z2, b1, b2, put1, get1);
#pragma unroll
      for (int b = 0; b < BL; ++b) {
        const int jj = t + T * b;
#pragma unroll
        for (int r = 1; r < R2; ++r) {
          const float2 w = __ldg(&tw[kWideTw3 + N + 256 * r + jj]);
          z1[b * R2 + r] = cmul(z1[b * R2 + r], w);
          z2[b * R2 + r] = cmul(z2[b * R2 + r], w);
        }
        wide_dft<R2>(&z1[b * R2]);
        wide_dft<R2>(&z2[b * R2]);
      }
    }
  }
};

}  // namespace swense
