// Stage 1 of the reconstruction: modal amplitudes -> (zero-padded) grid at arbitrary levels.
//
// Paper: reconstruction section, step "IFFT" (one inverse transform per vertical level onto
// uniformly spaced nodes), the zero-padding refinement (spectrum extended n times with zero
// modes -> n times finer grid) and the extension of the solution above z = 0.
//
// Columns of 32 to 1024 nodes and rows of 32 and more (3-D): k_form_modes makes the modal fields at z = 0
//   U = i kx A^phi, V = i ky A^phi, W = |k| A^phi, T = A^phit and A^eta
// of every time level once; then two passes per chunk of slots (the levels of all time levels, and eta):
//   columns (k_col_w)  per (slot, block of kx columns): depth factors F and S at the level, zero-padding
//           along ky, inverse transforms along y; writes G[slot][field][y][m] (complex, one-sided in m) to
//           the scratch workspace;
//   rows    (k_row_w; k_row_tb from 4096 nodes on; k_row_tma, an autotuner candidate)  per (slot, block of y
//           rows): the two real-field pairs packed into one complex spectrum each, Z1 = U + iV and
//           Z2 = W + iT (Hermitian extension over m, zero-padded to nx_r), inverse transforms along x, one
//           float4 (u, v, w, dphi/dt) per node.
// Other sizes, and requests whose scratch cannot be had: the same two passes over one time level's levels,
// in shared memory, each making its fields itself (k_pass_a, k_pass_b, and k_propagate before them); eta
// is one extra transform per time level (two grid rows per complex transform).
// 2-D (ny == 1): one kernel (k_line).
#include <algorithm>
#include <array>
#include <cmath>
#include <map>
#include <mutex>
#include <string>

#include "fft.cuh"
#include "internal.cuh"
#include "tma.cuh"

namespace swense {
namespace {

struct Levels {
  float z[SWENSE_MAX_LEVELS];
};

struct PassAArgs {
  const float2* A_phi;   // [ny][nxh1] of this time level
  const float2* A_phit;
  const float2* A_eta;
  float2* G;             // [nlev][4][Nyr][Mh] (levels) or [Nyr][Mh] (eta)
  const float2* tw;
  int ny, nxh1, Mh, Nyr, log2Nyr;
  int cb, fp;            // kx columns per CTA, fields per shared-memory pass
  int lev0;              // first level of the chunk
  int eta_mode;
  float kxs, kys, depth;
  int Nxr, spline;       // spline: store cubic B-spline coefficients (modes prefiltered)
};

__global__ void __launch_bounds__(256) k_pass_a(PassAArgs a, Levels L) {
  extern __shared__ float2 sm[];
  const int c0 = blockIdx.x * a.cb;
  const int slot = blockIdx.y;
  const int ncol = min(a.cb, a.Mh - c0);
  const float z = a.eta_mode ? 0.f : L.z[a.lev0 + slot];
  const int nfield = a.eta_mode ? 1 : 4;
  const int nyh = a.ny >> 1;
  for (int f0 = 0; f0 < nfield; f0 += a.fp) {
    const int nf = min(a.fp, nfield - f0);
    const int narr = nf * a.cb;
    for (int i = threadIdx.x; i < narr * a.Nyr; i += blockDim.x) sm[i] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int i = threadIdx.x; i < a.ny * a.cb; i += blockDim.x) {
      const int c = i % a.cb, r = i / a.cb;
      if (c >= ncol || r == nyh) continue;               // Nyquist row ignored
      const int m = c0 + c;
      const int n = r < nyh ? r : r - a.ny;
      const int pos = n >= 0 ? n : a.Nyr + n;            // zero-padding between +n and -n
      const unsigned br = bitrev(unsigned(pos), a.log2Nyr);
      const size_t gi = size_t(r) * a.nxh1 + m;
      const float pf = a.spline ? spline_prefilter(m, a.Nxr, n, a.Nyr) : 1.f;
      if (a.eta_mode) {
        const float2 e = __ldg(&a.A_eta[gi]);
        sm[c * a.Nyr + br] = make_float2(pf * e.x, pf * e.y);
        continue;
      }
      float2 Ap = __ldg(&a.A_phi[gi]);
      float2 At = __ldg(&a.A_phit[gi]);
      Ap = make_float2(pf * Ap.x, pf * Ap.y);
      At = make_float2(pf * At.x, pf * At.y);
      const float kx = float(m) * a.kxs, ky = float(n) * a.kys;
      const float k = sqrtf(kx * kx + ky * ky);
      float F, S;
      depth_factors(k, z, a.depth, F, S);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q < f0 || q >= f0 + nf) continue;
        float2 v;
        if (q == 0) v = make_float2(-kx * F * Ap.y, kx * F * Ap.x);        // i kx F A^phi
        else if (q == 1) v = make_float2(-ky * F * Ap.y, ky * F * Ap.x);   // i ky F A^phi
        else if (q == 2) v = make_float2(k * S * Ap.x, k * S * Ap.y);      // |k| S A^phi
        else v = make_float2(F * At.x, F * At.y);                          // F A^phit
        sm[((q - f0) * a.cb + c) * a.Nyr + br] = v;
      }
    }
    __syncthreads();
    fft_inv_inplace(sm, a.Nyr, a.log2Nyr, narr, a.tw);
    for (int i = threadIdx.x; i < nf * a.Nyr * a.cb; i += blockDim.x) {
      const int c = i % a.cb;
      const int rest = i / a.cb;
      const int y = rest % a.Nyr, q = rest / a.Nyr;
      if (c >= ncol) continue;
      const size_t go = ((size_t(slot) * nfield + f0 + q) * a.Nyr + y) * a.Mh + c0 + c;
      a.G[go] = sm[(q * a.cb + c) * a.Nyr + y];
    }
    __syncthreads();
  }
}

enum { B_LEVEL_G = 0, B_ETA_G = 1 };

struct PassBArgs {
  const float2* G;        // pass-A output (levels or eta)
  float4* nodes;          // [nz][Nyr][Nxr] of this time level
  float* eta;             // [Nyr][Nxr] of this time level
  const float2* tw;
  int Mh, Nxr, log2Nxr, Nyr;
  int rb;                 // rows (level modes) or row pairs (eta modes) per CTA
  int lev0;
  int mode;
};

// Hermitian packing of two one-sided spectra P, Q (coefficients of real fields p, q) into one
// full complex spectrum Z = P + iQ whose inverse transform is p + i q.
__device__ __forceinline__ void pack_pair(float2* Z, int m, int Nxr, int log2Nxr, float2 P, float2 Q) {
  if (m == 0) {
    Z[0] = make_float2(P.x, Q.x);                        // bitrev(0) == 0; real parts only
  } else {
    Z[bitrev(unsigned(m), log2Nxr)] = make_float2(P.x - Q.y, P.y + Q.x);
    Z[bitrev(unsigned(Nxr - m), log2Nxr)] = make_float2(P.x + Q.y, Q.x - P.y);
  }
}

__global__ void __launch_bounds__(256) k_pass_b(PassBArgs a) {
  extern __shared__ float2 sm[];
  const int slot = blockIdx.y;
  const bool eta_mode = a.mode == B_ETA_G;
  const int rows_per_cta = eta_mode ? 2 * a.rb : a.rb;
  const int y0 = blockIdx.x * rows_per_cta;
  const int narr = eta_mode ? a.rb : 2 * a.rb;
  for (int i = threadIdx.x; i < narr * a.Nxr; i += blockDim.x) sm[i] = make_float2(0.f, 0.f);
  __syncthreads();
  if (!eta_mode) {
    for (int i = threadIdx.x; i < a.rb * a.Mh; i += blockDim.x) {
      const int m = i % a.Mh, rr = i / a.Mh;
      const int y = y0 + rr;
      if (y >= a.Nyr) continue;
      const size_t base = (size_t(slot) * 4 * a.Nyr + y) * a.Mh + m;
      const size_t fs = size_t(a.Nyr) * a.Mh;
      const float2 U = __ldcg(&a.G[base]), V = __ldcg(&a.G[base + fs]);
      const float2 W = __ldcg(&a.G[base + 2 * fs]), T = __ldcg(&a.G[base + 3 * fs]);
      pack_pair(sm + size_t(2 * rr) * a.Nxr, m, a.Nxr, a.log2Nxr, U, V);
      pack_pair(sm + size_t(2 * rr + 1) * a.Nxr, m, a.Nxr, a.log2Nxr, W, T);
    }
  } else {
    for (int i = threadIdx.x; i < a.rb * a.Mh; i += blockDim.x) {
      const int m = i % a.Mh, pp = i / a.Mh;
      const int ya = y0 + 2 * pp, yb = ya + 1;
      if (ya >= a.Nyr) continue;
      const float2 Ea = __ldcg(&a.G[size_t(ya) * a.Mh + m]);
      const float2 Eb = yb < a.Nyr ? __ldcg(&a.G[size_t(yb) * a.Mh + m]) : make_float2(0.f, 0.f);
      pack_pair(sm + size_t(pp) * a.Nxr, m, a.Nxr, a.log2Nxr, Ea, Eb);
    }
  }
  __syncthreads();
  fft_inv_inplace(sm, a.Nxr, a.log2Nxr, narr, a.tw);
  if (!eta_mode) {
    float4* out = a.nodes + size_t(a.lev0 + slot) * a.Nyr * a.Nxr;
    for (int i = threadIdx.x; i < a.rb * a.Nxr; i += blockDim.x) {
      const int x = i % a.Nxr, rr = i / a.Nxr;
      const int y = y0 + rr;
      if (y >= a.Nyr) continue;
      const float2 z1 = sm[size_t(2 * rr) * a.Nxr + x];
      const float2 z2 = sm[size_t(2 * rr + 1) * a.Nxr + x];
      __stcs(&out[size_t(y) * a.Nxr + x], make_float4(z1.x, z1.y, z2.x, z2.y));
    }
  } else {
    for (int i = threadIdx.x; i < a.rb * a.Nxr; i += blockDim.x) {
      const int x = i % a.Nxr, pp = i / a.Nxr;
      const int ya = y0 + 2 * pp, yb = ya + 1;
      if (ya >= a.Nyr) continue;
      const float2 zz = sm[size_t(pp) * a.Nxr + x];
      __stcs(&a.eta[size_t(ya) * a.Nxr + x], zz.x);
      if (yb < a.Nyr) __stcs(&a.eta[size_t(yb) * a.Nxr + x], zz.y);
    }
  }
}

// Linear propagation of stored modes: A(t) = A(t_ref) e^{-i omega (t - t_ref)}, every time level
// in one launch (blockIdx.y). The phase is reduced to turns in FP64 (exact enough for long
// simulated times); the rotation is FP32.
struct PropTimes {
  double dt[64];       // t_l - t_ref per time level (a grid request has at most 64)
};
__global__ void k_propagate(const float2* __restrict__ Ae, const float2* __restrict__ Ap,
                            const float2* __restrict__ At, const double* __restrict__ omega,
                            int nslot, PropTimes T, float2* __restrict__ out_all) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nslot) return;
  const double dt = T.dt[blockIdx.y];
  float2* out = out_all + size_t(blockIdx.y) * 3 * nslot;
  const double turns = omega[i] * dt * 0.15915494309189533577;  // theta / (2 pi)
  const double frac = turns - rint(turns);
  float s, c;
  sincospif(2.f * float(frac), &s, &c);
  const float2 src[3] = {Ae[i], Ap[i], At[i]};
#pragma unroll
  for (int q = 0; q < 3; ++q)
    out[size_t(q) * nslot + i] =
        make_float2(fmaf(src[q].x, c, src[q].y * s), fmaf(src[q].y, c, -src[q].x * s));
}

// A 2-D (x, z) request in one launch: block (l, tl) propagates the one row of modes to time level tl
// (as k_propagate), forms level l's spectra Z1 = U and Z2 = W + iT (v is identically zero), l = nz:
// eta's, and transforms them in shared memory. Rows are short (256 modes in the regular-wave runs), so
// launches bound the request: five serial ones took 27 us, this one takes 5 us.
struct LineArgs {
  const float2 *Ae, *Ap, *At;
  const double* omega;
  float4* nodes;          // [n_tl][nz][Nxr]
  float* eta;             // [n_tl][Nxr]
  const float2* tw;
  int nxh1, Mh, Nxr, log2Nxr, nz, spline;
  float kxs, depth;
};
__global__ void __launch_bounds__(256) k_line(LineArgs a, const __grid_constant__ Levels L,
                                              const __grid_constant__ PropTimes T) {
  extern __shared__ float2 sm[];                 // Z1, Z2 (bit-reversed, then transformed in place)
  const int l = blockIdx.x, tl = blockIdx.y;
  const bool is_eta = l == a.nz;
  const int narr = is_eta ? 1 : 2;
  float2 *Z1 = sm, *Z2 = sm + a.Nxr;
  for (int i = threadIdx.x; i < narr * a.Nxr; i += blockDim.x) sm[i] = make_float2(0.f, 0.f);
  __syncthreads();
  const float z = is_eta ? 0.f : L.z[l];
  const float2 zero = make_float2(0.f, 0.f);
  for (int m = threadIdx.x; m < a.Mh; m += blockDim.x) {
    const size_t src = a.omega ? m : size_t(tl) * a.nxh1 + m;
    float c = 1.f, s = 0.f;
    if (a.omega) {
      const double turns = a.omega[m] * T.dt[tl] * 0.15915494309189533577;  // theta / (2 pi)
      sincospif(2.f * float(turns - rint(turns)), &s, &c);
    }
    const float pf = a.spline ? spline_prefilter(m, a.Nxr, 0, 1) : 1.f;
    auto mode = [&](const float2* A) {
      float2 v = __ldg(&A[src]);
      if (a.omega) v = make_float2(fmaf(v.x, c, v.y * s), fmaf(v.y, c, -v.x * s));
      return make_float2(pf * v.x, pf * v.y);
    };
    if (is_eta) {
      pack_pair(Z1, m, a.Nxr, a.log2Nxr, mode(a.Ae), zero);
      continue;
    }
    const float2 Ap = mode(a.Ap), At = mode(a.At);
    const float kx = float(m) * a.kxs;
    float F, S;
    depth_factors(kx, z, a.depth, F, S);
    pack_pair(Z1, m, a.Nxr, a.log2Nxr, make_float2(-kx * F * Ap.y, kx * F * Ap.x), zero);
    pack_pair(Z2, m, a.Nxr, a.log2Nxr, make_float2(kx * S * Ap.x, kx * S * Ap.y), make_float2(F * At.x, F * At.y));
  }
  __syncthreads();
  fft_inv_inplace(sm, a.Nxr, a.log2Nxr, narr, a.tw);
  if (is_eta) {
    float* out = a.eta + size_t(tl) * a.Nxr;
    for (int x = threadIdx.x; x < a.Nxr; x += blockDim.x) __stcs(&out[x], Z1[x].x);
  } else {
    float4* out = a.nodes + (size_t(tl) * a.nz + l) * a.Nxr;
    for (int x = threadIdx.x; x < a.Nxr; x += blockDim.x)
      __stcs(&out[x], make_float4(Z1[x].x, 0.f, Z2[x].x, Z2[x].y));
  }
}

// Modal fields at z = 0 of every time level (blockIdx.y) for the transposed pair's column pass:
// U = i kx A^phi, V = i ky A^phi, W = |k| A^phi, T = A^phit, propagated to the level's time (omega given,
// as in k_propagate; otherwise snapshot blockIdx.y) and with the spline prefilter; made
// once, where the column pass would make each at every vertical level. eta's modes come fifth,
// [tl][5][ny][ld], or (eta non-NULL: its own transform follows, which prefilters itself) are only
// propagated, [tl][ny][nx/2+1].
struct FormArgs {
  const float2 *Ae, *Ap, *At;
  const double* omega;
  float2 *eta, *fields;
  int ny, nxh1, ld, Nxr, Nyr, spline;
  float kxs, kys;
};
__global__ void __launch_bounds__(256) k_form_modes(FormArgs a, PropTimes T) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, nslot = a.ny * a.nxh1;
  if (i >= nslot) return;
  const int r = i / a.nxh1, m = i - r * a.nxh1, tl = blockIdx.y;
  float2 e, p, t;
  if (a.omega) {
    const double turns = a.omega[i] * T.dt[tl] * 0.15915494309189533577;  // theta / (2 pi)
    const double frac = turns - rint(turns);
    float s, c;
    sincospif(2.f * float(frac), &s, &c);
    auto turn = [&](float2 v) { return make_float2(fmaf(v.x, c, v.y * s), fmaf(v.y, c, -v.x * s)); };
    e = turn(__ldg(&a.Ae[i]));
    p = turn(__ldg(&a.Ap[i]));
    t = turn(__ldg(&a.At[i]));
    if (a.eta) a.eta[size_t(tl) * nslot + i] = e;
  } else {
    e = __ldg(&a.Ae[size_t(tl) * nslot + i]);
    p = __ldg(&a.Ap[size_t(tl) * nslot + i]);
    t = __ldg(&a.At[size_t(tl) * nslot + i]);
  }
  if (m >= a.nxh1 - 1) return;                     // the Nyquist column carries no mode
  const int n = r < a.ny / 2 ? r : r - a.ny;
  if (a.spline) {
    const float pf = spline_prefilter(m, a.Nxr, n, a.Nyr);
    e = make_float2(pf * e.x, pf * e.y);
    p = make_float2(pf * p.x, pf * p.y);
    t = make_float2(pf * t.x, pf * t.y);
  }
  const float kx = float(m) * a.kxs, ky = float(n) * a.kys, k = sqrtf(kx * kx + ky * ky);
  const size_t fs = size_t(a.ny) * a.ld;
  float2* o = a.fields + size_t(tl) * 5 * fs + size_t(r) * a.ld + m;
  o[0] = make_float2(-kx * p.y, kx * p.x);
  o[fs] = make_float2(-ky * p.y, ky * p.x);
  o[2 * fs] = make_float2(k * p.x, k * p.y);
  o[3 * fs] = t;
  o[4 * fs] = e;
}

constexpr int kThreads = 256;
constexpr size_t kSmemBudget = 64 * 1024;
// Level chunks of at most 512 MB, as few as that allows: each pass pays its first and last wave of blocks
// (about 20 us) once a chunk, which outweighs an intermediate that stays in L2 (2048 x 1024 modes, 256 levels:
// 7.44 ms, 7.89 at 256 MB, 9.07 at 64 MB; 512 x 256 modes, 128 levels in one chunk instead of one and a
// rest of two slots: 13 us less).
constexpr size_t kChunkBytes = size_t(512) << 20;
constexpr int kColLevels = 1;   // levels per column-transform CTA

int set_smem(const void* fn, size_t bytes) {
  SWENSE_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)));
  return SWENSE_OK;
}


struct ColArgs {
  const float2* A;       // [n_tl][5][ny][ldG] modal fields at z = 0 and eta (k_form_modes)
  float2* G;             // [nslot][4][Nyr][ldG]
  const float2* tw;
  int ny, Mh, Nyr, nz;
  int lpc;               // slots per CTA
  int lev0, nlev;        // chunk: first slot and slots. Slot tl nz + l is level l of time level tl
  int n_lev;             // n_tl nz; slot n_lev + tl is eta of time level tl
  float kxs, kys, depth;
  int ldG;               // m stride of the modal fields and of the transposed intermediate
};

struct RowArgs {
  const float2* G;       // [nslot][4][Nyr][ldG]
  float4* nodes;         // [n_tl nz][Nyr][Nxr]
  float* eta;            // [n_tl][Nyr][Nxr] (k_row_w)
  const float2* tw;
  int Mh, Nxr, Nyr, lev0, n_lev;
  int ldG;               // m stride of the transposed intermediate
  int polls;             // staged rows: polls of a bounded wait before it gives up
  int selftest;          // staged rows: 1 = issue no copy, so every wait runs out (self-test)
};

// m stride of the transposed intermediate: a whole number of 128-byte lines per field row, so
// the row pass can drop the rows it has consumed from L2 without touching a neighbour's data.
__host__ __device__ __forceinline__ int trans_ld(int Mh) { return (Mh + 15) & ~15; }

// Invalidate, without write-back, the L2 lines of nf field rows (stride fs float2) of ld float2
// each starting at row (128-byte aligned): their values are dead once the row pass has read
// them, so the column pass's writes need not reach DRAM. Lines spread over nt threads from t.
__device__ __forceinline__ void discard_rows(const float2* row, size_t fs, int nf, int ld, int t, int nt) {
  const int lines = ld / 16;
  for (int i = t; i < nf * lines; i += nt) {
    const float2* a = row + size_t(i / lines) * fs + size_t(i % lines) * 16;
    asm volatile("discard.global.L2 [%0], 128;" ::"l"(a) : "memory");
  }
}

// Transposed pair for 32- to 1024-point columns (and rows of 32 to 8192 points). The column pass
// writes G[level][field][y][m] with the m stride padded to whole 128-byte lines (ldG), so that a grid
// row's inputs are contiguous for the row pass.
//
// Column pass: a block owns kCols neighbouring kx columns of one level at a time, its lanes laid out
// column-fastest: every global access (modes in, intermediate out) is a run of kCols neighbouring m,
// with no transposing tile, and the one exchange between the two wide passes has whole rows of
// columns in neighbouring banks. The depth factors of a level are made once, in shared memory, for
// the four modal fields, which the block transforms one after another. Before, each field's block
// made its own (a square root and an exponential per point: 118 instructions a point against 64 now)
// and went through shared memory four times. Eight levels of 1024 x 1024 columns: 198 -> 146 us at
// 37 % issue (latency of the loads and of the in-register DFTs at 16 warps per SM); eight levels of
// 256-point columns padded to 1024: 61 -> 24 us; 64 levels of 256 x 256: 64 -> 42 us.
template <int N>
struct ColCfg {
  static constexpr int R0 = wide_r0(N), R1 = N / R0, E = R0, T = N / E, B1 = E / R1;
  static constexpr int kCols = N >= 256 ? 8 : (N >= 64 ? 16 : 32);
  static constexpr int kThr = T * kCols;
  // 8 columns are half a row of banks: one row of padding in R0 keeps the writes of neighbouring j
  // (rows R0 apart) in different halves
  static constexpr int kPad = kCols == 8 ? 1 : 0;
  static constexpr int kXch = (N + kPad * T) * kCols;
  static constexpr int kMin = N >= 1024 ? 2 : (N >= 512 ? 4 : (N >= 128 ? 6 : 8));   // blocks per SM
};

template <int N, bool FINITE>
__global__ void __launch_bounds__(ColCfg<N>::kThr, ColCfg<N>::kMin) k_col_w(ColArgs a, const __grid_constant__ Levels L) {
  using C = ColCfg<N>;
  constexpr int E = C::E, T = C::T, R0 = C::R0, R1 = C::R1;
  // exchange [rows][kCols], twiddles [N], depth factors [E][kThr] (each thread its own: the data of 32
  // elements alone take 64 registers)
  extern __shared__ float2 sm[];
  float2* xch = sm;
  float2* stw = sm + C::kXch;
  float* sF = reinterpret_cast<float*>(stw + N) + threadIdx.x;
  const int c = threadIdx.x % C::kCols, j = threadIdx.x / C::kCols;
  const int m = blockIdx.x * C::kCols + c;
  const bool colok = m < a.Mh;
  const int nyh = a.ny >> 1;
  for (int i = threadIdx.x; i < N; i += C::kThr) stw[i] = __ldg(&a.tw[kWideTw + N + i]);
  const float kx = float(m) * a.kxs;
  __syncthreads();
  // position p = j + T e holds wavenumber index n = p (first half) or p - N, i.e. row p or ny + p - N
  // of the modes; zero in the padding and at the Nyquist row
  const float2* A0 = a.A + size_t(j) * a.ldG + m;
  const int up = (a.ny - N) * a.ldG;
  auto live = [&](int e) { return colok && (e < E / 2 ? j + T * e < nyh : N - T * e - j < nyh); };
  for (int li = 0; li < a.lpc; ++li) {
    const int level = blockIdx.y * a.lpc + li;
    if (level >= a.nlev) break;                  // uniform over the block
    const int slot = a.lev0 + level;
    const bool is_eta = slot >= a.n_lev;
    const int tl = is_eta ? slot - a.n_lev : slot / a.nz;
    const float z = is_eta ? 0.f : L.z[slot - tl * a.nz];
    const int nq = is_eta ? 1 : 4;
#pragma unroll 1
    for (int qi = 0; qi < nq; ++qi) {
      const int q = is_eta ? 4 : (qi < 2 ? qi : 5 - qi);   // U, V, dphi/dt (factor F), then W (factor S)
      if (qi == 0 || (FINITE && qi == 3)) {
#pragma unroll 2
        for (int e = 0; e < E; ++e) {
          float f = 0.f;
          if (live(e)) {
            const float ky = float(e < E / 2 ? j + T * e : j + T * e - N) * a.kys;
            float F, S;
            depth_factors(sqrtf(kx * kx + ky * ky), z, a.depth, F, S);
            f = is_eta ? 1.f : (FINITE && qi == 3 ? S : F);
          }
          sF[e * C::kThr] = f;
        }
      }
      const float2* __restrict__ A = A0 + (size_t(tl) * 5 + q) * a.ny * a.ldG;
      float2 v[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        v[e] = make_float2(0.f, 0.f);
        if (live(e)) v[e] = __ldg(&A[e * T * a.ldG + (e < E / 2 ? 0 : up)]);
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float f = sF[e * C::kThr];
        v[e] = make_float2(f * v[e].x, f * v[e].y);
      }
      wide_dft<R0>(v);
#pragma unroll
      for (int r = 0; r < R0; ++r) xch[(j * (R0 + C::kPad) + r) * C::kCols + c] = v[dft_slot<R0>(r)];
      __syncthreads();
#pragma unroll
      for (int b = 0; b < C::B1; ++b)
#pragma unroll
        for (int r = 0; r < R1; ++r) v[b * R1 + r] = xch[(j + T * b + (R0 + C::kPad) * r) * C::kCols + c];
      __syncthreads();                           // the buffer is free for the next field
      float2* out = a.G + (size_t(level) * 4 + (is_eta ? 0 : q)) * N * a.ldG + m;
#pragma unroll
      for (int b = 0; b < C::B1; ++b) {
        const int jj = j + T * b;
#pragma unroll
        for (int r = 1; r < R1; ++r) v[b * R1 + r] = cmul(v[b * R1 + r], stw[r * R0 + jj]);
        wide_dft<R1>(&v[b * R1]);
        if (colok) {
#pragma unroll
          for (int r = 0; r < R1; ++r) __stcg(&out[(jj + R0 * r) * a.ldG], v[b * R1 + dft_slot<R1>(r)]);
        }
      }
    }
  }
}

// Set when a bounded wait of a staged row pass gives up; the host reads and clears it with
// swense_async_status.
__device__ int g_async_timeout;

// Row pass over the transposed intermediate for rows of 32 to 2048 points: T = N / R0 threads per grid
// row; its four modal fields packed as Z1 = U + iV and Z2 = W + iT over the full x spectrum, both
// transformed (WideRow), stored as float4. Persistent blocks take kRows rows of a slot at a time, whose
// fields (contiguous in G) arrive in shared memory by bulk copies on the block's mbarrier, the next
// rows' while the current ones are transformed: at padding 1 a row is 32 KB read twice (as mode m and
// mirrored as N - m), which straight loads could only fetch a third at a time for want of registers.
// A wait that does not complete within its bound sets the error flag and ends the block, as one.
// Eight levels of 1024 x 2048 nodes: at padding 1 149 -> 97 us (5.5 TB/s with the
// intermediate from memory), at padding 4 (a quarter of the input) 76 us; radix-8 passes with
// straight loads took 124 and 108.
// TWO: an exchange buffer for each of the two transforms, where the staged rows leave the room. SELF: no copy is
// issued (self-test; its own instance, since the question alone cost 1615 -> 1618 us on the padded grid).
template <int N, bool TWO, bool SELF = false>
__global__ void __launch_bounds__(WideRow<N>::T * WideRow<N>::kRows, WideRow<N>::E == 16 ? 4 : 8) k_row_w(RowArgs a, int items) {
  using W = WideRow<N>;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int t = threadIdx.x % W::T, rr = threadIdx.x / W::T;
  const size_t fs = size_t(a.Nyr) * a.ldG;
  const unsigned span = unsigned(W::kRows * a.ldG) * unsigned(sizeof(float2));   // bytes per field
  float2* stg = reinterpret_cast<float2*>(smraw);
  float2* buf = reinterpret_cast<float2*>(smraw + 4 * size_t(span)) + rr * (TWO ? 2 : 1) * W::kBuf;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw + 4 * size_t(span) + size_t(W::kRows) * (TWO ? 2 : 1) * W::kBuf * sizeof(float2));
  const int yblocks = a.Nyr / W::kRows;            // the row count is a multiple of kRows
  auto issue = [&](int item) {                     // by one thread
    const int level = item / yblocks, y0 = (item - level * yblocks) * W::kRows;
    const int nf = a.lev0 + level >= a.n_lev ? 1 : 4;   // eta: one field
    const float2* src = a.G + size_t(level) * 4 * fs + size_t(y0) * a.ldG;
    fence_proxy_async();                           // earlier reads of the buffer come first
    mbar_arrive_expect_tx(bar, nf * span);
    for (int f = 0; f < (SELF ? 0 : nf); ++f) bulk_g2s(stg + size_t(f) * W::kRows * a.ldG, src + f * fs, span, bar);
  };
  int item = blockIdx.x;
  if (item >= items) return;
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    fence_proxy_async();
    issue(item);
  }
  __syncthreads();
  for (unsigned ph = 0; item < items; ph ^= 1u) {
    const bool done = mbar_wait(bar, ph, a.polls);
    if (__syncthreads_or(!done)) {                 // one thread gave up: the whole block leaves
      if (threadIdx.x == 0) atomicExch(&g_async_timeout, 1);
      mbar_wait(bar, ph, a.polls);                 // the copy waited on is the only one in flight
      __syncthreads();
      return;
    }
    const int level = item / yblocks, y = (item - level * yblocks) * W::kRows + rr;
    const bool is_eta = a.lev0 + level >= a.n_lev;   // one field: Z1 = eta, the others zero
    const float2* S = stg + size_t(rr) * a.ldG;
    const size_t ss = size_t(W::kRows) * a.ldG;
    float2 z1[W::E], z2[W::E];
#pragma unroll
    for (int e = 0; e < W::E; ++e) {
      // positions of the upper half hold the mirrored (conjugate) modes N - p
      const int p = t + W::T * e, mm = e < W::E / 2 ? p : N - p;
      float2 U = make_float2(0.f, 0.f), V = U, X = U, Y = U;
      if (mm < a.Mh) {
        U = S[mm];
        if (!is_eta) {
          V = S[ss + mm];
          X = S[2 * ss + mm];
          Y = S[3 * ss + mm];
        }
      }
      if (e >= W::E / 2) {
        z1[e] = make_float2(U.x + V.y, V.x - U.y);
        z2[e] = make_float2(X.x + Y.y, Y.x - X.y);
      } else if (e == 0 && t == 0) {               // m = 0: the real parts only
        z1[e] = make_float2(U.x, V.x);
        z2[e] = make_float2(X.x, Y.x);
      } else {
        z1[e] = make_float2(U.x - V.y, U.y + V.x);
        z2[e] = make_float2(X.x - Y.y, X.y + Y.x);
      }
    }
    __syncthreads();                               // the staged rows have been read
    const int next = item + int(gridDim.x);
    if (threadIdx.x == 0 && next < items) issue(next);
    W::template fft2<TWO>(z1, z2, a.tw, buf, TWO ? buf + W::kBuf : buf, t);
    if (is_eta) {
      float* out = a.eta + (size_t(a.lev0 + level - a.n_lev) * a.Nyr + y) * N;
#pragma unroll
      for (int b = 0; b < W::BL; ++b)
#pragma unroll
        for (int r = 0; r < W::RL; ++r) __stcs(&out[W::pos(t, b, r)], z1[W::elem(b, r)].x);
    } else {
      float4* out = a.nodes + (size_t(a.lev0 + level) * a.Nyr + y) * N;
#pragma unroll
      for (int b = 0; b < W::BL; ++b)
#pragma unroll
        for (int r = 0; r < W::RL; ++r) {
          const int e = W::elem(b, r);
          __stcs(&out[W::pos(t, b, r)], make_float4(z1[e].x, z1[e].y, z2[e].x, z2[e].y));
        }
    }
    discard_rows(a.G + size_t(level) * 4 * fs + size_t(y) * a.ldG, fs, is_eta ? 1 : 4, a.ldG, t, W::T);
    item = next;
  }
}

// Row pass for 4096- and 8192-point rows: one block of kThreads per grid row of one level, inputs
// from the transposed intermediate (coalesced), block-wide Stockham transforms of Z1 = U + iV and
// Z2 = W + iT.
template <int N>
__global__ void __launch_bounds__(256, N >= 8192 ? 1 : 2) k_row_tb(RowArgs a) {
  extern __shared__ float2 sm[];                 // one or two exchange buffers
  constexpr int E = N / kThreads, RL = stk_radix(N, stk_npass(N) - 1);
  constexpr bool BOTH = N <= 4096;               // both transforms' data in registers at once
  const int t = threadIdx.x;
  const int y = blockIdx.x;
  const int level = blockIdx.y;
  const size_t fs = size_t(a.Nyr) * a.ldG;
  const float2* row = a.G + size_t(level) * 4 * fs + size_t(y) * a.ldG;
  float4* out = a.nodes + (size_t(a.lev0 + level) * a.Nyr + y) * N;
  auto pack = [&](float2 (&z)[E], int q) {       // q = 0: U + iV, 1: W + iT
    const float2* A = row + 2 * q * fs;
    const float2* B = A + fs;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int p = t + kThreads * (e / 8) + (e % 8) * (N / 8);
      const bool lo = p < a.Mh, hi = p > N - a.Mh;
      float2 u = make_float2(0.f, 0.f), v = u;
      if (lo || hi) {
        const int mm = lo ? p : N - p;
        u = __ldcg(&A[mm]);
        v = __ldcg(&B[mm]);
      }
      if (p == 0) z[e] = make_float2(u.x, v.x);
      else if (!hi) z[e] = make_float2(u.x - v.y, u.y + v.x);
      else z[e] = make_float2(u.x + v.y, v.x - u.y);
    }
  };
  if constexpr (BOTH) {
    float2 z1[E], z2[E];
    pack(z1, 0);
    pack(z2, 1);
    stkb_fft2<N, kThreads>(z1, z2, a.tw, sm, sm + stk_buf(N), t);
#pragma unroll
    for (int e = 0; e < E; ++e)
      __stcs(&out[t + kThreads * (e / RL) + (e % RL) * (N / RL)], make_float4(z1[e].x, z1[e].y, z2[e].x, z2[e].y));
    __syncthreads();                             // every thread's reads of the rows are done
    discard_rows(row, fs, 4, a.ldG, t, kThreads);
  } else {
    float2* o2 = reinterpret_cast<float2*>(out);
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
      float2 z[E];
      pack(z, q);
      stkb_fft<N, kThreads>(z, a.tw, sm, t);
#pragma unroll
      for (int e = 0; e < E; ++e) __stcs(&o2[2 * (t + kThreads * (e / RL) + (e % RL) * (N / RL)) + q], z[e]);
      __syncthreads();                           // the buffer is reused by the second transform
    }
    discard_rows(row, fs, 4, a.ldG, t, kThreads);  // after the barrier: all reads are done
  }
}

// Row pass over the transposed intermediate with its inputs staged by bulk copies: each warp
// takes `rpw` consecutive rows of one level; lane 0 copies a row's four field segments
// (ldG complex values each, contiguous in G) into the warp's staging buffer with cp.async.bulk
// on the warp's mbarrier, and the next row's copy runs while the current row is transformed.
// A wait that does not complete within its bound sets the device error flag and ends the warp:
// the warp decides together (every lane must have seen its copy complete), waits, also bounded,
// for the copy it still has in flight, and leaves as one. The host reads and clears the flag
// with swense_async_status.
template <int N>
__global__ void __launch_bounds__(256, N >= 1024 ? 1 : 2) k_row_tma(RowArgs a, int rpw) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int E = N / 32, RL = stk_radix(N, stk_npass(N) - 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned span = unsigned(a.ldG) * unsigned(sizeof(float2));      // bytes per field row
  const size_t per_warp = 4 * size_t(span) + size_t(stk_buf(N)) * sizeof(float2);
  float2* stg = reinterpret_cast<float2*>(smraw + warp * per_warp);
  float2* xbuf = reinterpret_cast<float2*>(smraw + warp * per_warp + 4 * size_t(span));
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw + (kThreads / 32) * per_warp) + warp;
  const int level = blockIdx.y;
  const int y0 = (blockIdx.x * (kThreads / 32) + warp) * rpw;
  const int nrows = min(rpw, a.Nyr - y0);
  if (nrows <= 0) return;                        // no block-wide barrier in this kernel
  const size_t fs = size_t(a.Nyr) * a.ldG;
  const float2* Gl = a.G + size_t(level) * 4 * fs;
  if (lane == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    fence_proxy_async();
  }
  __syncwarp();
  auto issue = [&](int i) {
    if (lane == 0) {
      fence_proxy_async();                       // earlier reads of the buffer come first
      mbar_arrive_expect_tx(bar, 4 * span);
      const float2* src = Gl + size_t(y0 + i) * a.ldG;
      if (!a.selftest) {
#pragma unroll
        for (int f = 0; f < 4; ++f) bulk_g2s(stg + f * a.ldG, src + f * fs, span, bar);
      }
    }
  };
  issue(0);
  float2 T[stk_twn(N)];
  stk_init<N>(T, a.tw, lane);
  for (int i = 0; i < nrows; ++i) {
    const bool done = mbar_wait(bar, unsigned(i) & 1u, a.polls);
    if (!__all_sync(0xffffffffu, done)) {        // one lane gave up: the whole warp leaves
      if (lane == 0) atomicExch(&g_async_timeout, 1);
      // the copy waited on is the only one in flight (none in the self-test)
      mbar_wait(bar, unsigned(i) & 1u, a.polls);
      __syncwarp();
      return;
    }
    float2 z1[E], z2[E];
    const float2* U = stg;
    const float2* V = stg + a.ldG;
    const float2* W = stg + 2 * a.ldG;
    const float2* Tt = stg + 3 * a.ldG;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int p = lane + 32 * (e / 8) + (e % 8) * (N / 8);
      const bool lo = p < a.Mh, hi = p > N - a.Mh;
      float2 u = make_float2(0.f, 0.f), v = u, w = u, t = u;
      if (lo || hi) {
        const int mm = lo ? p : N - p;
        u = U[mm];
        v = V[mm];
        w = W[mm];
        t = Tt[mm];
      }
      if (p == 0) {
        z1[e] = make_float2(u.x, v.x);
        z2[e] = make_float2(w.x, t.x);
      } else if (!hi) {
        z1[e] = make_float2(u.x - v.y, u.y + v.x);
        z2[e] = make_float2(w.x - t.y, w.y + t.x);
      } else {
        z1[e] = make_float2(u.x + v.y, v.x - u.y);
        z2[e] = make_float2(w.x + t.y, t.x - w.y);
      }
    }
    __syncwarp();                                // every lane has read the staged row
    // the bulk copy that filled the staging buffer has completed: its global rows are dead
    discard_rows(Gl + size_t(y0 + i) * a.ldG, fs, 4, a.ldG, lane, 32);
    if (i + 1 < nrows) issue(i + 1);
    stk_fft<N>(z1, T, a.tw, xbuf, lane);
    stk_fft<N>(z2, T, a.tw, xbuf, lane);
    float4* out = a.nodes + (size_t(a.lev0 + level) * a.Nyr + y0 + i) * N;
#pragma unroll
    for (int e = 0; e < E; ++e)
      __stcs(&out[lane + 32 * (e / RL) + (e % RL) * (N / RL)], make_float4(z1[e].x, z1[e].y, z2[e].x, z2[e].y));
  }
}

// Launch-shape choices per grid shape (set by swense_autotune_grid or swense_set_grid_tune; defaults
// otherwise).
struct Tune {
  int lpc = -1;                         // levels per column-transform CTA of the transposed pair;
                                        // 0: shared-memory path; -1: default for the shape
  size_t chunk_bytes = kChunkBytes;     // scratch per level chunk
  int rowv = 0;                         // 4: row pass with staged inputs; 5: the pair's passes
                                        // pipelined over two streams; others: one stream
};
std::mutex g_tune_mutex;
std::map<std::array<int64_t, 4>, Tune> g_tune;

Tune tuned(int nx, int ny, int pad, int nz) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  auto it = g_tune.find({nx, ny, pad, nz});
  return it == g_tune.end() ? Tune{} : it->second;
}

// Validated sizes and derived constants of one swense_fields_on_grid request.
struct GridPlan {
  int nx, ny, nz, n_tl, nxh1, Mh, pad, spline;
  int64_t Nxr, Nyr;
  size_t nslot, per_level, geta_bytes;
  bool omega;
  Levels lev;
};

template <int N>
int launch_col_w(const ColArgs& c, const Levels& L, int nl, cudaStream_t stream) {
  using C = ColCfg<N>;
  const size_t smem = (size_t(C::kXch) + N) * sizeof(float2) + size_t(C::E) * C::kThr * sizeof(float);
  const dim3 grid(unsigned((c.Mh + C::kCols - 1) / C::kCols), unsigned((nl + c.lpc - 1) / c.lpc));
  const void* fn = c.depth > 0.f ? (const void*)k_col_w<N, true> : (const void*)k_col_w<N, false>;
  int st = set_smem(fn, smem);
  if (st) return st;
  if (c.depth > 0.f) k_col_w<N, true><<<grid, C::kThr, smem, stream>>>(c, L);
  else k_col_w<N, false><<<grid, C::kThr, smem, stream>>>(c, L);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

template <int N>
int launch_row_w(const RowArgs& r, int nl, cudaStream_t stream) {
  using W = WideRow<N>;
  const int per_sm = W::E == 16 ? 4 : 8;
  const size_t stage = size_t(4) * W::kRows * r.ldG * sizeof(float2), buf = size_t(W::kRows) * W::kBuf * sizeof(float2);
  // 227 KB of shared memory per SM, 1 KB of it reserved per block
  const bool two = !r.selftest && (stage + 2 * buf + 1152) * per_sm <= size_t(227) * 1024;
  const size_t smem = stage + (two ? 2 : 1) * buf + sizeof(uint64_t);
  const auto kernel = r.selftest ? k_row_w<N, false, true> : (two ? k_row_w<N, true> : k_row_w<N, false>);
  int st = set_smem((const void*)kernel, smem);
  if (st) return st;
  int dev = 0, sms = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  SWENSE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int items = nl * (r.Nyr / W::kRows);
  const unsigned grid = unsigned(std::min(items, sms * per_sm));
  kernel<<<grid, W::T * W::kRows, smem, stream>>>(r, items);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

template <int N>
int launch_row_tb(const RowArgs& r, unsigned nl, cudaStream_t stream) {
  const size_t smem = size_t(N <= 4096 ? 2 : 1) * stk_buf(N) * sizeof(float2);
  int st = set_smem((const void*)k_row_tb<N>, smem);
  if (st) return st;
  k_row_tb<N><<<dim3(unsigned(r.Nyr), nl), kThreads, smem, stream>>>(r);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

constexpr int kRowsPerWarp = 2;     // rows a warp of the staged row pass takes in turn

template <int N>
int launch_row_tma(const RowArgs& r, unsigned nl, cudaStream_t stream) {
  const size_t per_warp = 4 * size_t(r.ldG) * sizeof(float2) + size_t(stk_buf(N)) * sizeof(float2);
  const size_t smem = (kThreads / 32) * per_warp + (kThreads / 32) * sizeof(uint64_t);
  int st = set_smem((const void*)k_row_tma<N>, smem);
  if (st) return st;
  const unsigned per_block = (kThreads / 32) * kRowsPerWarp;
  k_row_tma<N><<<dim3((unsigned(r.Nyr) + per_block - 1) / per_block, nl), kThreads, smem, stream>>>(r, kRowsPerWarp);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

// Transposed pair: `which` = 1 the column pass alone, 2 the row pass alone, 0 both; staged: the row
// pass whose inputs arrive by bulk copies (256- to 1024-point rows; others take the plain one).
int launch_pair(const ColArgs& c, const RowArgs& r, const Levels& L, int nl, cudaStream_t s, bool staged = false,
                int which = 0) {
  int st = SWENSE_OK;
  if (which != 2) {
    switch (c.Nyr) {
      case 32: st = launch_col_w<32>(c, L, nl, s); break;
      case 64: st = launch_col_w<64>(c, L, nl, s); break;
      case 128: st = launch_col_w<128>(c, L, nl, s); break;
      case 256: st = launch_col_w<256>(c, L, nl, s); break;
      case 512: st = launch_col_w<512>(c, L, nl, s); break;
      case 1024: st = launch_col_w<1024>(c, L, nl, s); break;
      default: return fail(SWENSE_ERR_UNSUPPORTED, "transposed pair: column length");
    }
  }
  if (st || which == 1) return st;
  if (staged) {
    switch (r.Nxr) {
      case 256: return launch_row_tma<256>(r, unsigned(nl), s);
      case 512: return launch_row_tma<512>(r, unsigned(nl), s);
      case 1024: return launch_row_tma<1024>(r, unsigned(nl), s);
      default: break;
    }
  }
  switch (r.Nxr) {
    case 32: return launch_row_w<32>(r, nl, s);
    case 64: return launch_row_w<64>(r, nl, s);
    case 128: return launch_row_w<128>(r, nl, s);
    case 256: return launch_row_w<256>(r, nl, s);
    case 512: return launch_row_w<512>(r, nl, s);
    case 1024: return launch_row_w<1024>(r, nl, s);
    case 2048: return launch_row_w<2048>(r, nl, s);
    case 4096: return launch_row_tb<4096>(r, unsigned(nl), s);
    case 8192: return launch_row_tb<8192>(r, unsigned(nl), s);
    default: return fail(SWENSE_ERR_UNSUPPORTED, "transposed pair: row length");
  }
}

// The transposed pair covers 3-D grids with 32- to 1024-point columns and rows of 32 points and more.
bool pair_path(int ny, int64_t Nxr, int64_t Nyr) {
  return ny > 1 && Nyr >= 32 && Nyr <= 1024 && Nxr >= 32 && Nxr <= SWENSE_MAX_FFT;
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

int plan_grid(const swense_modes* md, int32_t n_tl, const double* t, const swense_grid_desc* desc,
              const float* nodes, const float* eta, GridPlan* p) {
  if (!md || !desc || !nodes || !eta) return fail(SWENSE_ERR_ARG, "NULL modes, desc or output");
  if (!md->A_eta || !md->A_phi || !md->A_phit) return fail(SWENSE_ERR_ARG, "NULL modal amplitudes");
  const int nx = md->nx, ny = md->ny;
  if (!is_pow2(nx) || nx < 4 || !is_pow2(ny) || (ny != 1 && ny < 4))
    return fail(SWENSE_ERR_SIZE, "nx must be a power of two >= 4, ny 1 or a power of two >= 4");
  const int pad = desc->pad_n;
  if (pad < 1 || pad > 8) return fail(SWENSE_ERR_ARG, "pad_n must lie in 1..8");
  const int64_t Nxr = int64_t(pad) * nx, Nyr = ny > 1 ? int64_t(pad) * ny : 1;
  if (Nxr > SWENSE_MAX_FFT || Nyr > SWENSE_MAX_FFT)
    return fail(SWENSE_ERR_SIZE, "pad_n*nx and pad_n*ny must not exceed SWENSE_MAX_FFT");
  if (!(md->Lx > 0) || !std::isfinite(md->Lx) || (ny > 1 && (!(md->Ly > 0) || !std::isfinite(md->Ly))))
    return fail(SWENSE_ERR_ARG, "domain lengths must be finite and positive");
  if (!std::isfinite(md->depth)) return fail(SWENSE_ERR_ARG, "depth must be finite");
  if (n_tl < 1 || n_tl > 64) return fail(SWENSE_ERR_ARG, "n_tl must be in [1, 64]");
  if (md->omega) {
    if (md->n_snap != 1) return fail(SWENSE_ERR_ARG, "with omega, n_snap must be 1");
    if (!t) return fail(SWENSE_ERR_ARG, "with omega, t[n_tl] is required");
    for (int l = 0; l < n_tl; ++l)
      if (!std::isfinite(t[l])) return fail(SWENSE_ERR_ARG, "non-finite time");
  } else if (md->n_snap != n_tl) {
    return fail(SWENSE_ERR_ARG, "without omega, n_snap must equal n_tl");
  }
  const int nz = desc->nz;
  if (nz < 4 || nz > SWENSE_MAX_LEVELS || !desc->z_levels)
    return fail(SWENSE_ERR_LEVELS, "need 4 <= nz <= SWENSE_MAX_LEVELS levels");
  for (int l = 0; l < nz; ++l) {
    p->lev.z[l] = desc->z_levels[l];
    if (!std::isfinite(p->lev.z[l]) || (l > 0 && !(p->lev.z[l] > p->lev.z[l - 1])))
      return fail(SWENSE_ERR_LEVELS, "z_levels must be finite and strictly increasing");
  }
  if ((reinterpret_cast<uintptr_t>(nodes) & 15) || (reinterpret_cast<uintptr_t>(eta) & 3))
    return fail(SWENSE_ERR_ARG, "nodes must be 16-byte aligned, eta 4-byte aligned");
  if (desc->scheme != SWENSE_LAGRANGE3 && desc->scheme != SWENSE_SPLINE3)
    return fail(SWENSE_ERR_ARG, "unknown interpolation scheme");
  p->spline = desc->scheme == SWENSE_SPLINE3;
  p->nx = nx;
  p->ny = ny;
  p->pad = pad;
  p->nz = nz;
  p->n_tl = n_tl;
  p->nxh1 = nx / 2 + 1;
  p->Mh = nx / 2;
  p->Nxr = Nxr;
  p->Nyr = Nyr;
  p->nslot = size_t(ny) * p->nxh1;
  p->per_level = size_t(4) * Nyr * trans_ld(p->Mh) * sizeof(float2);
  p->omega = md->omega != nullptr;
  p->geta_bytes = ny > 1 ? size_t(Nyr) * p->Mh * sizeof(float2) : 0;
  return SWENSE_OK;
}

// The launch shape of a request: the tuned one of its grid shape, else the transposed pair where it
// applies and the shared-memory path elsewhere.
using Shape = GridShape;

// Whether a launch shape runs the transposed pair, and with eta's transforms among its slots (the
// row passes of 4096 points and more and the staged one take levels only).
bool runs_pair(const GridPlan& p, int lpc) { return lpc > 0 && pair_path(p.ny, p.Nxr, p.Nyr); }
bool eta_inline(const GridPlan& p, const Shape& s) { return runs_pair(p, s.lpc) && p.Nxr <= 2048 && s.rowv != 4; }
// Slots of a request: levels of all time levels (and eta) for the pair, else one time level's levels.
int grid_slots(const GridPlan& p, const Shape& s) {
  return runs_pair(p, s.lpc) ? p.n_tl * (p.nz + (eta_inline(p, s) ? 1 : 0)) : p.nz;
}

int chunk_slots(const GridPlan& p, const Shape& s, size_t bytes) {
  return int(std::max<size_t>(1, std::min<size_t>(size_t(grid_slots(p, s)), bytes / p.per_level)));
}
// Slots of a chunk where no more chunks are taken than need be: all are of this size but the last, which has
// what is left (2048 x 1024 modes, 258 slots: 16 of 16 slots and the two of eta, which are a quarter of the
// work; sizes that differ by one at most were slower there, 7.50 -> 7.54 ms, and at 130 slots, 1615 -> 1620 us).
int even_chunk(const GridPlan& p, const Shape& s, int chunk) {
  const int n = grid_slots(p, s), k = (n + chunk - 1) / chunk;
  return (n + k - 1) / k;
}
Shape grid_shape(const GridPlan& p) {
  const Tune tn = tuned(p.nx, p.ny, p.pad, p.nz);
  Shape s;
  s.lpc = tn.lpc >= 0 ? tn.lpc : (pair_path(p.ny, p.Nxr, p.Nyr) ? kColLevels : 0);
  s.rowv = tn.lpc >= 0 ? tn.rowv : 0;
  s.chunk = p.ny > 1 ? even_chunk(p, s, chunk_slots(p, s, tn.chunk_bytes)) : 0;
  return s;
}

// Scratch bytes of the prepared modes: the pair's modal fields and eta's propagated modes, or the
// three propagated arrays of the shared-memory path.
size_t modes_bytes(const GridPlan& p, bool pair) {
  const size_t own = p.omega ? (pair ? 1 : 3) * p.nslot : 0;
  return size_t(p.n_tl) * (own + (pair ? size_t(5) * p.ny * trans_ld(p.Mh) : 0)) * sizeof(float2);
}

// Scratch bytes for a level chunk of `chunk` levels (0 when no scratch is needed).
size_t scratch_bytes(const GridPlan& p, int chunk, int nbuf, bool pair) {
  const size_t g_bytes = p.ny > 1 ? size_t(chunk) * p.per_level : 0;
  return align256(modes_bytes(p, pair)) + align256(p.geta_bytes) + size_t(nbuf) * align256(g_bytes);
}

// Workspace of a request (`extra` bytes more); where that much cannot be had, or would have to be got
// during a capture, of smaller chunks, down to one slot, and at last of the shared-memory path, whose
// modes take less. First without giving up the present workspace (a smaller chunk is better than a free
// and an allocation on every call), then, should it not even hold one slot, whatever it takes.
constexpr size_t kChunkNeeded = size_t(64) << 20;
int shape_workspace(const GridPlan& p, Shape* s, int nbuf, size_t extra, cudaStream_t stream, void** ws) {
  const Shape first = *s;
  Shape shared = first;
  shared.lpc = 0;
  shared.chunk = chunk_slots(p, shared, kChunkNeeded);
  int st = SWENSE_OK;
  for (int pass = 0; pass < 2; ++pass) {
    for (Shape t : {first, shared}) {
      if (pass == 1) t.chunk = std::min(t.chunk, chunk_slots(p, t, kChunkNeeded));
      for (;; t.chunk = (t.chunk + 1) / 2) {
        const size_t bytes = scratch_bytes(p, t.chunk, nbuf, runs_pair(p, t.lpc)) + extra;
        st = !bytes ? SWENSE_OK : pass == 0 ? workspace_optional(bytes, stream, ws) : workspace(bytes, stream, ws);
        *s = t;
        if (st != SWENSE_ERR_OOM && st != SWENSE_ERR_ARG) return st;   // ARG: growth during a capture
        if (t.chunk <= 1) break;
      }
      if (!runs_pair(p, first.lpc)) break;
    }
  }
  return st;
}

// Self-test of the staged rows' waits, per device (swense_selftest_grid_wait_timeout).
std::mutex g_selftest_mutex;
bool g_selftest[64];
bool g_row_selftest() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(g_selftest_mutex);
  return g_selftest[dev];
}

// Library-internal second stream and events (per device) for the two-stream transform
// pipeline: chunk c's row pass runs on the second stream while chunk c+1's column pass runs on
// the caller's stream, with two intermediate buffers. Created on first use; recording, waiting
// and launching on them inside a stream capture joins them to the capture (fork/join).
struct Pipe {
  cudaStream_t side = nullptr;
  cudaEvent_t col_done[2] = {nullptr, nullptr}, row_done[2] = {nullptr, nullptr};
  // the eta transform runs beside the level transforms on a stream of its own
  cudaStream_t eta_side = nullptr;
  cudaEvent_t eta_fork = nullptr, eta_join = nullptr;
};
std::mutex g_pipe_mutex;
std::map<int, Pipe> g_pipe;

int get_pipe(Pipe** out) {
  int dev = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  Pipe& pp = g_pipe[dev];
  if (!pp.side) {
    SWENSE_CUDA_TRY(cudaStreamCreateWithFlags(&pp.side, cudaStreamNonBlocking));
    for (int b = 0; b < 2; ++b) {
      SWENSE_CUDA_TRY(cudaEventCreateWithFlags(&pp.col_done[b], cudaEventDisableTiming));
      SWENSE_CUDA_TRY(cudaEventCreateWithFlags(&pp.row_done[b], cudaEventDisableTiming));
    }
    SWENSE_CUDA_TRY(cudaStreamCreateWithFlags(&pp.eta_side, cudaStreamNonBlocking));
    SWENSE_CUDA_TRY(cudaEventCreateWithFlags(&pp.eta_fork, cudaEventDisableTiming));
    SWENSE_CUDA_TRY(cudaEventCreateWithFlags(&pp.eta_join, cudaEventDisableTiming));
  }
  *out = &pp;
  return SWENSE_OK;
}

// Enqueue every kernel of the request; `ws` holds scratch_bytes(p, chunk) bytes. eta_side: run
// the eta transform of each time level on the per-device second stream, forked after that time
// level's propagated modes exist and joined back before the call returns (graph-capturable).
int launch_grid(const GridPlan& p, const swense_modes* md, const double* t, float* nodes, float* eta,
                void* ws, const Shape& shape, cudaStream_t stream, bool overlap, bool eta_side) {
  const float2* tw = nullptr;
  {
    int st = twiddles(stream, &tw);
    if (st) return st;
  }
  const int chunk = shape.chunk;
  const int ny = p.ny, nz = p.nz, Mh = p.Mh, nxh1 = p.nxh1;
  const int64_t Nxr = p.Nxr, Nyr = p.Nyr;
  const size_t nslot = p.nslot;
  const bool pair = runs_pair(p, shape.lpc);
  const int ld = trans_ld(Mh);
  float2* prop = static_cast<float2*>(ws);       // pair: eta's modes (with omega), then the modal fields
  float2* form = prop + (pair && md->omega ? size_t(p.n_tl) * nslot : 0);
  const size_t b_modes = align256(modes_bytes(p, pair));
  float2* g_eta = reinterpret_cast<float2*>(static_cast<char*>(ws) + b_modes);
  float2* g_lev = reinterpret_cast<float2*>(static_cast<char*>(ws) + b_modes + align256(p.geta_bytes));
  // second intermediate buffer of the two-stream pipeline
  float2* g_lev2 = reinterpret_cast<float2*>(reinterpret_cast<char*>(g_lev) +
                                             align256(size_t(chunk) * p.per_level));
  Pipe* pipe = nullptr;
  const bool use_pipe = overlap && pair;
  const bool inline_eta = eta_inline(p, shape);
  const bool eta_fork = eta_side && p.ny > 1 && !inline_eta;
  if (use_pipe || eta_fork) {
    int st = get_pipe(&pipe);
    if (st) return st;
  }
  struct EtaJoin {                               // the caller's stream waits for the eta stream
    Pipe* pp;
    cudaStream_t s;
    bool forked;
    ~EtaJoin() {
      if (!pp || !forked) return;
      cudaEventRecord(pp->eta_join, pp->eta_side);
      cudaStreamWaitEvent(s, pp->eta_join, 0);
    }
  } eta_join{eta_fork ? pipe : nullptr, stream, false};
  int chunk_no = 0;                              // chunks issued so far (over all time levels)
  struct Join {                                  // the caller's stream waits for the second one
    Pipe* pp;
    int* n;
    cudaStream_t s;
    ~Join() {
      if (!pp) return;
      for (int b = 0; b < 2 && b < *n; ++b) cudaStreamWaitEvent(s, pp->row_done[b], 0);
    }
  } join{use_pipe ? pipe : nullptr, &chunk_no, stream};

  const float kxs = float(6.283185307179586476925 / md->Lx);
  const float kys = ny > 1 ? float(6.283185307179586476925 / md->Ly) : 0.f;
  const float depth = md->depth > 0 ? float(md->depth) : 0.f;
  const int log2Nxr = ilog2(Nxr), log2Nyr = ilog2(Nyr);

  PropTimes T{};
  for (int l = 0; md->omega && l < p.n_tl; ++l) T.dt[l] = t[l] - md->t_ref;
  const float2 *A_eta = reinterpret_cast<const float2*>(md->A_eta), *A_phi = reinterpret_cast<const float2*>(md->A_phi),
               *A_phit = reinterpret_cast<const float2*>(md->A_phit);
  if (ny == 1) {
    const size_t smem = size_t(2) * Nxr * sizeof(float2);
    int st = set_smem((const void*)k_line, smem);
    if (st) return st;
    const LineArgs a{A_eta, A_phi, A_phit, md->omega, reinterpret_cast<float4*>(nodes), eta, tw, nxh1, Mh, int(Nxr),
                     log2Nxr, nz, p.spline, kxs, depth};
    k_line<<<dim3(unsigned(nz + 1), unsigned(p.n_tl)), kThreads, smem, stream>>>(a, p.lev, T);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);
    return SWENSE_OK;
  }

  // launch shapes
  int fp = 4, cb = 1;
  while (fp > 1 && size_t(fp) * Nyr * sizeof(float2) > kSmemBudget) fp >>= 1;
  cb = int(std::max<size_t>(1, kSmemBudget / (size_t(fp) * Nyr * sizeof(float2))));
  cb = std::min(cb, std::min(64, Mh));
  int cb_eta = int(std::max<size_t>(1, kSmemBudget / (size_t(Nyr) * sizeof(float2))));
  cb_eta = std::min(cb_eta, std::min(64, Mh));
  // the eta transform is a single level: keep about two CTAs per SM busy rather than few wide ones
  cb_eta = std::min(cb_eta, std::max(1, (Mh + 303) / 304));
  const size_t rowb = size_t(2) * Nxr * sizeof(float2);
  int rb = int(std::max<size_t>(1, kSmemBudget / rowb));
  rb = int(std::min<int64_t>(rb, std::min<int64_t>(16, Nyr)));
  int rb_eta = int(std::max<size_t>(1, kSmemBudget / (size_t(Nxr) * sizeof(float2))));
  rb_eta = int(std::min<int64_t>(rb_eta, std::min<int64_t>(16, (Nyr + 1) / 2)));
  rb_eta = int(std::min<int64_t>(rb_eta, std::max<int64_t>(1, ((Nyr + 1) / 2 + 303) / 304)));
  const size_t smem_a = size_t(fp) * cb * Nyr * sizeof(float2);
  const size_t smem_a_eta = size_t(cb_eta) * Nyr * sizeof(float2);
  const size_t smem_b = size_t(rb) * rowb;
  const size_t smem_b_eta = size_t(rb_eta) * Nxr * sizeof(float2);
  {
    int st = set_smem((const void*)k_pass_a, std::max(smem_a, smem_a_eta));
    if (!st) st = set_smem((const void*)k_pass_b, std::max(smem_b, smem_b_eta));
    if (st) return st;
  }

  if (md->omega || pair) {                        // all time levels' modes at once
    const dim3 gm(unsigned((nslot + 255) / 256), unsigned(p.n_tl));
    if (pair) {
      const FormArgs f{A_eta, A_phi, A_phit, md->omega, inline_eta ? nullptr : prop, form, ny, nxh1, ld, int(Nxr), int(Nyr), p.spline, kxs, kys};
      k_form_modes<<<gm, 256, 0, stream>>>(f, T);
    } else {
      k_propagate<<<gm, 256, 0, stream>>>(A_eta, A_phi, A_phit, md->omega, int(nslot), T, prop);
    }
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);
  }
  for (int l = 0; l < p.n_tl && !inline_eta; ++l) {
    const float2 *Ae, *Ap = nullptr, *At = nullptr;
    if (md->omega && pair) {
      Ae = prop + size_t(l) * nslot;
    } else if (md->omega) {
      float2* o = prop + size_t(l) * 3 * nslot;
      Ae = o;
      Ap = o + nslot;
      At = o + 2 * nslot;
    } else {
      Ae = reinterpret_cast<const float2*>(md->A_eta) + size_t(l) * nslot;
      Ap = reinterpret_cast<const float2*>(md->A_phi) + size_t(l) * nslot;
      At = reinterpret_cast<const float2*>(md->A_phit) + size_t(l) * nslot;
    }
    float4* nodes_l = reinterpret_cast<float4*>(nodes) + size_t(l) * nz * Nyr * Nxr;
    float* eta_l = eta + size_t(l) * Nyr * Nxr;

    PassBArgs b{};
    b.nodes = nodes_l;
    b.eta = eta_l;
    b.tw = tw;
    b.Mh = Mh;
    b.Nxr = int(Nxr);
    b.log2Nxr = log2Nxr;
    b.Nyr = int(Nyr);

    PassAArgs a{};
    a.A_phi = Ap;
    a.A_phit = At;
    a.A_eta = Ae;
    a.tw = tw;
    a.ny = ny;
    a.nxh1 = nxh1;
    a.Mh = Mh;
    a.Nyr = int(Nyr);
    a.log2Nyr = log2Nyr;
    a.kxs = kxs;
    a.kys = kys;
    a.depth = depth;
    a.Nxr = int(Nxr);
    a.spline = p.spline;

    // eta: pass A (eta mode) then pass B packing row pairs; on the eta stream when forked (the
    // time levels' eta transforms stay in order there, so they share one intermediate)
    cudaStream_t es = stream;
    if (eta_fork) {
      SWENSE_CUDA_TRY(cudaEventRecord(pipe->eta_fork, stream));
      SWENSE_CUDA_TRY(cudaStreamWaitEvent(pipe->eta_side, pipe->eta_fork, 0));
      eta_join.forked = true;
      es = pipe->eta_side;
    }
    a.G = g_eta;
    a.eta_mode = 1;
    a.fp = 1;
    a.cb = cb_eta;
    a.lev0 = 0;
    k_pass_a<<<dim3((Mh + cb_eta - 1) / cb_eta, 1), kThreads, smem_a_eta, es>>>(a, p.lev);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);
    b.G = g_eta;
    b.mode = B_ETA_G;
    b.rb = rb_eta;
    b.lev0 = 0;
    k_pass_b<<<dim3(unsigned((Nyr + 2 * rb_eta - 1) / (2 * rb_eta)), 1), kThreads, smem_b_eta,
               es>>>(b);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);

    if (pair) continue;                          // the levels of all time levels follow
    a.eta_mode = 0;
    a.fp = fp;
    a.cb = cb;
    a.G = g_lev;
    b.G = g_lev;
    b.mode = B_LEVEL_G;
    b.rb = rb;
    for (int l0 = 0; l0 < nz; l0 += chunk) {
      const int nl = std::min(chunk, nz - l0);
      a.lev0 = l0;
      b.lev0 = l0;
      k_pass_a<<<dim3((Mh + cb - 1) / cb, nl), kThreads, smem_a, stream>>>(a, p.lev);
      SWENSE_CUDA_TRY(cudaGetLastError());
      count_launches(1);
      k_pass_b<<<dim3(unsigned((Nyr + rb - 1) / rb), nl), kThreads, smem_b, stream>>>(b);
      SWENSE_CUDA_TRY(cudaGetLastError());
      count_launches(1);
    }
  }
  if (!pair) return SWENSE_OK;
  ColArgs ca{};
  ca.A = form;
  ca.G = g_lev;
  ca.tw = tw;
  ca.ny = ny;
  ca.Mh = Mh;
  ca.Nyr = int(Nyr);
  ca.nz = nz;
  ca.n_lev = p.n_tl * nz;
  ca.lpc = shape.lpc;
  ca.kxs = kxs;
  ca.kys = kys;
  ca.depth = depth;
  RowArgs ra{};
  ra.G = g_lev;
  ra.nodes = reinterpret_cast<float4*>(nodes);
  ra.eta = eta;
  ra.tw = tw;
  ra.Mh = Mh;
  ra.Nxr = int(Nxr);
  ra.Nyr = int(Nyr);
  ra.n_lev = ca.n_lev;
  const bool selftest = g_row_selftest();
  ra.polls = selftest ? 8 : kMbarPolls;
  ra.selftest = selftest;
  ca.ldG = ra.ldG = ld;
  const int slots = grid_slots(p, shape);
  for (int l0 = 0; l0 < slots; l0 += chunk) {
    const int nl = std::min(chunk, slots - l0);
    ca.lev0 = ra.lev0 = l0;
    ca.nlev = nl;
    if (!use_pipe) {
      int st = launch_pair(ca, ra, p.lev, nl, stream, shape.rowv == 4);
      if (st) return st;
      continue;
    }
    const int b = chunk_no & 1;
    ca.G = b ? g_lev2 : g_lev;
    ra.G = ca.G;
    if (chunk_no >= 2) SWENSE_CUDA_TRY(cudaStreamWaitEvent(stream, pipe->row_done[b], 0));
    int st = launch_pair(ca, ra, p.lev, nl, stream, false, 1);          // column pass
    if (st) return st;
    SWENSE_CUDA_TRY(cudaEventRecord(pipe->col_done[b], stream));
    SWENSE_CUDA_TRY(cudaStreamWaitEvent(pipe->side, pipe->col_done[b], 0));
    st = launch_pair(ca, ra, p.lev, nl, pipe->side, false, 2);          // row pass
    if (st) return st;
    SWENSE_CUDA_TRY(cudaEventRecord(pipe->row_done[b], pipe->side));
    ++chunk_no;
  }
  return SWENSE_OK;
}

}  // namespace
}  // namespace swense

namespace swense {
namespace {

// Zero-padding by a factor that is not a power of two, pad = q p2 with q odd: the refined node
// x_I, I = q J + s, is the p2-refined node x_J moved by s Lx / (pad nx), which is the p2-refined
// transform of the modes times e^{i k_x s Lx / (pad nx)} (the shift theorem; likewise in y).
// So the grid is q^2 (q in 2-D) power-of-two transforms of phase-shifted modes, each scattered
// to every q-th node. The spline prefilter, which depends on the final node spacing, is applied
// here, and the shifted transforms run as Lagrange grids.
__global__ void __launch_bounds__(256) k_shift_modes(const float2* __restrict__ ae, const float2* __restrict__ ap,
                                                     const float2* __restrict__ at, int nx, int ny, int64_t total,
                                                     int sx, int sy, int Nxr, int Nyr, int spline,
                                                     float2* __restrict__ oe, float2* __restrict__ op,
                                                     float2* __restrict__ ot) {
  const int nh1 = nx / 2 + 1;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int m = int(i % nh1);
    const int r = int((i / nh1) % ny);
    const int n = ny == 1 ? 0 : (r < ny / 2 ? r : r - ny);
    // phase in turns, reduced exactly in integers: m sx / Nxr + n sy / Nyr
    const int tx = int((int64_t(m) * sx) % Nxr);
    const int ty = ny == 1 ? 0 : int(((int64_t(n) * sy) % Nyr + Nyr) % Nyr);
    float tau = float(tx) / float(Nxr) + (ny == 1 ? 0.f : float(ty) / float(Nyr));
    tau -= floorf(tau);
    float sn, cs;
    sincospif(2.f * tau, &sn, &cs);
    const float f = spline ? spline_prefilter(m, Nxr, n, Nyr) : 1.f;
    const float c = f * cs, s2 = f * sn;
    const float2 e = __ldg(&ae[i]), p = __ldg(&ap[i]), t = __ldg(&at[i]);
    oe[i] = make_float2(c * e.x - s2 * e.y, c * e.y + s2 * e.x);
    op[i] = make_float2(c * p.x - s2 * p.y, c * p.y + s2 * p.x);
    ot[i] = make_float2(c * t.x - s2 * t.y, c * t.y + s2 * t.x);
  }
}

// Sub-grid node (tl, level, J_y, J_x) -> refined node (tl, level, qy J_y + sy, q J_x + sx).
__global__ void __launch_bounds__(256) k_scatter_grid(const float4* __restrict__ sn, const float* __restrict__ se,
                                                      int64_t n_nodes, int64_t n_eta, int nxs, int nys, int q,
                                                      int qy, int sx, int sy, int64_t Nxr, int64_t Nyr,
                                                      float4* __restrict__ nodes, float* __restrict__ eta) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n_nodes + n_eta;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t k = i < n_nodes ? i : i - n_nodes;
    const int64_t jx = k % nxs, rest = k / nxs;
    const int64_t jy = rest % nys, slab = rest / nys;            // slab: (tl, level) or tl
    const int64_t o = (slab * Nyr + qy * jy + sy) * Nxr + q * jx + sx;
    if (i < n_nodes) nodes[o] = __ldg(&sn[k]);
    else eta[o] = __ldg(&se[k]);
  }
}

}  // namespace
}  // namespace swense

using namespace swense;

namespace swense {
namespace {

int fields_on_grid_shifted(const GridPlan& p, const swense_modes* md, const double* t, float* nodes,
                           float* eta, cudaStream_t stream) {
  int q = p.pad, p2 = 1;
  while (!(q & 1)) {
    q >>= 1;
    p2 <<= 1;
  }
  const int qy = p.ny > 1 ? q : 1;
  // the plan of one shifted power-of-two transform
  GridPlan sp = p;
  sp.pad = p2;
  sp.spline = 0;
  sp.Nxr = int64_t(p2) * p.nx;
  sp.Nyr = p.ny > 1 ? int64_t(p2) * p.ny : 1;
  sp.per_level = size_t(4) * sp.Nyr * trans_ld(sp.Mh) * sizeof(float2);
  sp.geta_bytes = p.ny > 1 ? size_t(sp.Nyr) * sp.Mh * sizeof(float2) : 0;
  Shape shape = grid_shape(sp);                               // one stream for the sub-grids
  const int64_t sub_nodes = int64_t(p.n_tl) * p.nz * sp.Nyr * sp.Nxr;
  const int64_t sub_eta = int64_t(p.n_tl) * sp.Nyr * sp.Nxr;
  const int64_t nmodes = int64_t(md->n_snap) * p.ny * p.nxh1;
  const size_t b_nodes = align256(size_t(sub_nodes) * sizeof(float4));
  const size_t b_eta = align256(size_t(sub_eta) * sizeof(float));
  const size_t b_modes = align256(size_t(nmodes) * sizeof(float2));
  void* ws = nullptr;
  int st = shape_workspace(sp, &shape, 1, b_nodes + b_eta + 3 * b_modes, stream, &ws);
  if (st) return st;
  const size_t scratch = align256(scratch_bytes(sp, shape.chunk, 1, runs_pair(sp, shape.lpc)));
  char* base = static_cast<char*>(ws);
  float4* snodes = reinterpret_cast<float4*>(base + scratch);
  float* seta = reinterpret_cast<float*>(base + scratch + b_nodes);
  float2* sm = reinterpret_cast<float2*>(base + scratch + b_nodes + b_eta);
  swense_modes shifted = *md;
  shifted.A_eta = reinterpret_cast<const float*>(sm);
  shifted.A_phi = reinterpret_cast<const float*>(sm + b_modes / sizeof(float2));
  shifted.A_phit = reinterpret_cast<const float*>(sm + 2 * (b_modes / sizeof(float2)));
  const int threads = 256;
  for (int sy = 0; sy < qy; ++sy) {
    for (int sx = 0; sx < q; ++sx) {
      const int64_t mb = std::min<int64_t>((nmodes + threads - 1) / threads, int64_t(1) << 20);
      k_shift_modes<<<unsigned(mb), threads, 0, stream>>>(
          reinterpret_cast<const float2*>(md->A_eta), reinterpret_cast<const float2*>(md->A_phi),
          reinterpret_cast<const float2*>(md->A_phit), p.nx, p.ny, nmodes, sx, sy, int(p.Nxr), int(p.Nyr),
          p.spline, sm, sm + b_modes / sizeof(float2), sm + 2 * (b_modes / sizeof(float2)));
      SWENSE_CUDA_TRY(cudaGetLastError());
      count_launches(1);
      st = launch_grid(sp, &shifted, t, reinterpret_cast<float*>(snodes), seta, ws, shape, stream, false, false);
      if (st) return st;
      const int64_t tot = sub_nodes + sub_eta;
      const int64_t gb = std::min<int64_t>((tot + threads - 1) / threads, int64_t(152) * 64);
      k_scatter_grid<<<unsigned(gb), threads, 0, stream>>>(snodes, seta, sub_nodes, sub_eta, int(sp.Nxr),
                                                           int(sp.Nyr), q, qy, sx, sy, p.Nxr, p.Nyr,
                                                           reinterpret_cast<float4*>(nodes), eta);
      SWENSE_CUDA_TRY(cudaGetLastError());
      count_launches(1);
    }
  }
  return SWENSE_OK;
}

}  // namespace
}  // namespace swense

using namespace swense;

extern "C" int swense_fields_on_grid(const swense_modes* md, int32_t n_tl, const double* t,
                                     const swense_grid_desc* desc, float* nodes, float* eta,
                                     void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  GridPlan p;
  int st = plan_grid(md, n_tl, t, desc, nodes, eta, &p);
  if (st) return st;
  if (!is_pow2(p.pad)) return fields_on_grid_shifted(p, md, t, nodes, eta, stream);
  Shape shape = grid_shape(p);
  void* ws = nullptr;
  st = shape_workspace(p, &shape, shape.rowv == 5 ? 2 : 1, 0, stream, &ws);
  if (st) return st;
  return launch_grid(p, md, t, nodes, eta, ws, shape, stream, shape.rowv == 5, true);
}

namespace swense {

// Launch shape and scratch of one swense_fields_on_grid call, and the same call
// with that scratch supplied (no library stream: the eta transform and, for variant 5, the row
// passes stay on `stream`), for callers that run several reconstructions concurrently, each in
// its own part of the workspace (swense_batch_run).
int grid_scratch(const swense_modes* md, int32_t n_tl, const double* t, const swense_grid_desc* desc,
                 float* nodes, float* eta, size_t chunk_limit, GridShape* shape, size_t* bytes) {
  GridPlan p;
  int st = plan_grid(md, n_tl, t, desc, nodes, eta, &p);
  if (st) return st;
  if (!is_pow2(p.pad)) return fail(SWENSE_ERR_UNSUPPORTED, "batched grids take power-of-two padding factors");
  *shape = grid_shape(p);
  if (chunk_limit == 0) shape->lpc = 0;
  if (p.ny > 1) shape->chunk = std::min(shape->chunk, chunk_slots(p, *shape, chunk_limit));
  *bytes = scratch_bytes(p, shape->chunk, 1, runs_pair(p, shape->lpc));
  return SWENSE_OK;
}

int grid_with_scratch(const swense_modes* md, int32_t n_tl, const double* t, const swense_grid_desc* desc,
                      float* nodes, float* eta, const GridShape& shape, void* ws, cudaStream_t stream) {
  GridPlan p;
  int st = plan_grid(md, n_tl, t, desc, nodes, eta, &p);
  if (st) return st;
  if (!is_pow2(p.pad)) return fail(SWENSE_ERR_UNSUPPORTED, "batched grids take power-of-two padding factors");
  return launch_grid(p, md, t, nodes, eta, ws, shape, stream, false, false);
}

}  // namespace swense

extern "C" int swense_autotune_grid(const swense_modes* md, int32_t n_tl, const double* t,
                                    const swense_grid_desc* desc, float* nodes, float* eta,
                                    int32_t* lpc_out, int64_t* chunk_bytes_out, int32_t* row_variant_out,
                                    void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  GridPlan p;
  int st = plan_grid(md, n_tl, t, desc, nodes, eta, &p);
  if (st) return st;
  if (!is_pow2(p.pad))
    return fail(SWENSE_ERR_UNSUPPORTED, "autotune the power-of-two factor of the padding instead");
  Tune best{};
  if (p.ny > 1) {
    cudaEvent_t e0, e1;
    SWENSE_CUDA_TRY(cudaEventCreate(&e0));
    SWENSE_CUDA_TRY(cudaEventCreate(&e1));
    float best_ms = 1e30f;
    // Every timed repetition starts from a cold L2, as a solver's step does (its other work
    // evicts the grid): the workspace, sized for the largest candidate and at least twice the
    // L2, is overwritten before each repetition (its contents are scratch).
    constexpr size_t kFlushBytes = size_t(256) << 20;
    const int max_chunk = chunk_slots(p, Shape{0, 1, 0}, kFlushBytes);   // the largest candidate: 256 MB
    bool pp = pair_path(p.ny, p.Nxr, p.Nyr);
    size_t ws_all = 0;
    for (;; pp = false) {                        // the pair's candidates only where its scratch can be had
      const size_t chunks = pp ? scratch_bytes(p, max_chunk, 2, true)
                               : scratch_bytes(p, chunk_slots(p, Shape{0, 0, 0}, kFlushBytes), 1, false);
      ws_all = std::max(chunks, kFlushBytes);
      void* ws = nullptr;
      st = workspace(ws_all, stream, &ws);
      if (st && !(st == SWENSE_ERR_OOM && pp)) {
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        return st;
      }
      if (!st) break;
    }
    for (int lpc : {0, 1, 2, 4})
    for (int rowv : {0, 4, 5}) {
      if (lpc > 0 && !pp) continue;
      if (rowv && lpc == 0) continue;
      if (rowv == 4 && (p.Nxr < 256 || p.Nxr > 1024)) continue;
      for (size_t mb : {16, 32, 64, 96, 128, 256}) {
        const size_t cb = mb << 20;
        Shape shape{0, lpc, rowv};
        shape.chunk = even_chunk(p, shape, chunk_slots(p, shape, cb));
        void* ws = nullptr;
        st = workspace(ws_all, stream, &ws);
        if (!st) st = launch_grid(p, md, t, nodes, eta, ws, shape, stream, rowv == 5, true);   // warm
        // best of five (the fastest repetition is the least disturbed one)
        float ms = 0.f, tot = 1e30f;
        for (int rep = 0; rep < 5 && !st; ++rep) {
          if (cudaMemsetAsync(ws, 0, kFlushBytes, stream) != cudaSuccess) { st = SWENSE_ERR_CUDA; break; }
          if (cudaEventRecord(e0, stream) != cudaSuccess) { st = SWENSE_ERR_CUDA; break; }
          st = launch_grid(p, md, t, nodes, eta, ws, shape, stream, rowv == 5, true);
          if (cudaEventRecord(e1, stream) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
              cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) st = SWENSE_ERR_CUDA;
          tot = std::min(tot, ms);
        }
        if (st) break;
        if (tot < best_ms) {
          best_ms = tot;
          best.lpc = lpc;
          best.chunk_bytes = cb;
          best.rowv = rowv;
        }
      }
      if (st) break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st) return st == SWENSE_ERR_CUDA ? cuda_fail(cudaGetLastError(), "autotune timing") : st;
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    g_tune[{p.nx, p.ny, p.pad, p.nz}] = best;
  }
  if (lpc_out) *lpc_out = best.lpc;
  if (chunk_bytes_out) *chunk_bytes_out = int64_t(best.chunk_bytes);
  if (row_variant_out) *row_variant_out = best.rowv;
  return SWENSE_OK;
}

extern "C" int swense_set_grid_tune(int32_t nx, int32_t ny, int32_t pad_n, int32_t nz, int32_t lpc,
                                    int64_t chunk_bytes, int32_t row_variant) {
  if (lpc != -1 && lpc != 0 && lpc != 1 && lpc != 2 && lpc != 4)
    return fail(SWENSE_ERR_ARG, "lpc must be -1 (default), 0, 1, 2 or 4");
  if (chunk_bytes < (int64_t(1) << 20) || chunk_bytes > (int64_t(1) << 30))
    return fail(SWENSE_ERR_ARG, "chunk_bytes must be in [1 MiB, 1 GiB]");
  if ((row_variant & 15) > 5 || (row_variant >> 4) > 1 || row_variant < 0)
    return fail(SWENSE_ERR_ARG, "row_variant must be 0..5, plus 16 for the one-field column pass");
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  if (lpc == -1) {                      // back to the untuned defaults for this shape
    g_tune.erase({nx, ny, pad_n, nz});
    return SWENSE_OK;
  }
  Tune tn;
  tn.lpc = lpc;
  tn.chunk_bytes = size_t(chunk_bytes);
  tn.rowv = row_variant & 15;           // the one-field column variants (+16) run the same kernel
  g_tune[{nx, ny, pad_n, nz}] = tn;
  return SWENSE_OK;
}

// ---------------------------------------------------------------------------------------------
// Bounded device-side waits report here: the flag of this translation unit (k_row_w, k_row_tma).
namespace swense {

int grid_async_flag(bool reset, int* was_set) {
  int v = 0;
  SWENSE_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_async_timeout, sizeof(int)));
  if (reset && v) {
    const int zero = 0;
    SWENSE_CUDA_TRY(cudaMemcpyToSymbol(g_async_timeout, &zero, sizeof(int)));
  }
  *was_set = v;
  return SWENSE_OK;
}

}  // namespace swense

extern "C" int swense_selftest_grid_wait_timeout(int32_t on) {
  int dev = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SWENSE_ERR_UNSUPPORTED, "device index too large");
  std::lock_guard<std::mutex> lock(g_selftest_mutex);
  g_selftest[dev] = on != 0;
  return SWENSE_OK;
}

extern "C" int swense_selftest_wait_timeout(void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  const float2* tw = nullptr;
  int st = twiddles(stream, &tw);
  if (st) return st;
  // one level of 256-point rows, 16 rows: the bulk copies are never issued, so the first wait of
  // every warp runs out after a few polls; nothing is read or written but the flag
  constexpr int N = 256, rows = 16;
  const size_t g_bytes = size_t(4) * rows * trans_ld(N / 2) * sizeof(float2);
  void* ws = nullptr;
  st = workspace(g_bytes + size_t(rows) * N * sizeof(float4), stream, &ws);
  if (st) return st;
  RowArgs r{};
  r.G = static_cast<const float2*>(ws);
  r.nodes = reinterpret_cast<float4*>(static_cast<char*>(ws) + g_bytes);
  r.tw = tw;
  r.Mh = N / 2;
  r.Nxr = N;
  r.Nyr = rows;
  r.ldG = trans_ld(N / 2);
  r.polls = 8;
  r.selftest = 1;
  return launch_row_tma<N>(r, 1u, stream);
}

// ---------------------------------------------------------------------------------------------
// swense_fields_on_grid_noalloc: the same kernels, with their scratch in a fixed device array
// that is part of the library image instead of the cudaMalloc'ed workspace.
namespace swense {
namespace {

static __device__ __align__(256) unsigned char g_noalloc_scratch[SWENSE_NOALLOC_SCRATCH_BYTES];

std::mutex g_noalloc_mutex;
void* g_noalloc_ptr[64] = {};

// Device address of g_noalloc_scratch on the current device. The host-side symbol is only a
// stand-in, so the address is looked up once per device (with that device current) and cached.
int noalloc_scratch(void** out) {
  int dev = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SWENSE_ERR_UNSUPPORTED, "device index too large");
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return SWENSE_OK;
}

}  // namespace
}  // namespace swense

extern "C" int swense_fields_on_grid_noalloc(const swense_modes* md, int32_t n_tl, const double* t,
                                             const swense_grid_desc* desc, float* nodes,
                                             float* eta, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  GridPlan p;
  int st = plan_grid(md, n_tl, t, desc, nodes, eta, &p);
  if (st) return st;
  if (!is_pow2(p.pad))
    return fail(SWENSE_ERR_UNSUPPORTED, "padding factors that are not powers of two need the workspace (swense_fields_on_grid)");
  const size_t cap = size_t(SWENSE_NOALLOC_SCRATCH_BYTES);
  // the launch shape swense_fields_on_grid would take (tuned, else its default), except that the
  // two-stream pipeline (variant 5) stays on `stream`: the fixed array holds one level chunk, not
  // two, and this call uses no library stream. The limit is that of the shared-memory path, which
  // takes over where the pair's modal fields leave no room for a level.
  Shape shape = grid_shape(p);
  const size_t fixed = scratch_bytes(p, 0, 1, false);
  if (p.ny > 1) {
    if (fixed + p.per_level > cap)
      return fail(SWENSE_ERR_SIZE,
                  "request needs " + std::to_string(fixed + p.per_level) +
                      " bytes of scratch for one level; swense_fields_on_grid_noalloc has " +
                      std::to_string(cap) + " (SWENSE_NOALLOC_SCRATCH_BYTES)");
    if (scratch_bytes(p, 1, 1, runs_pair(p, shape.lpc)) > cap) shape.lpc = 0;
    shape.chunk = grid_slots(p, shape);
    while (shape.chunk > 1 && scratch_bytes(p, shape.chunk, 1, runs_pair(p, shape.lpc)) > cap) --shape.chunk;
  } else if (fixed > cap) {
    return fail(SWENSE_ERR_SIZE, "request needs " + std::to_string(fixed) +
                                     " bytes of scratch; swense_fields_on_grid_noalloc has " +
                                     std::to_string(cap) + " (SWENSE_NOALLOC_SCRATCH_BYTES)");
  }
  void* ws = nullptr;
  st = noalloc_scratch(&ws);
  if (st) return st;
  return launch_grid(p, md, t, nodes, eta, ws, shape, stream, false, false);
}
