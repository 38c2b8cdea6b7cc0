// Direct ("analytical") evaluation of the modal sums at arbitrary points.
//
// Paper: reconstruction section, subsection on the analytical evaluation of u_I and w_I
// (substituting the point coordinates into the modal sums; cost proportional to the number of
// Fourier components per point), with the spectral decomposition of Eqs. whatIsSpectralMethod1
// and whatIsSpectralMethod and Bernoulli for the pressure. Used for small mode counts and for
// near-body points that must not carry interpolation error.
//
// FP32 path: rows n and -n of the one-sided spectrum share |k|, so they are summed together. With
// theta = kx_m x and phi = ky_n y the two modes' contribution to a field is
//   cos(phi) F (P cos(theta) + Q sin(theta)) + sin(phi) F (R cos(theta) + S sin(theta))
// with P, Q, R, S made from the two amplitudes, so the inner loop over m needs one depth factor, one
// rotation of theta and four products per field for two modes. The phase is carried as an exact
// 32-bit fraction of a turn: per point X = frac(x / Lx) * 2^32 and Y = frac(y / Ly) * 2^32 (formed in
// FP64 once per point), per mode the integer product m X (mod 2^32), so the argument error does not
// grow with |k x|. Depth factors use a compensated |k| z product. Sums are accumulated per tile and
// then added to the running totals to limit FP32 round-off growth over many modes.
#include <algorithm>
#include <cmath>

#include "fft.cuh"
#include "internal.cuh"
#include "mma.cuh"

namespace swense {
namespace {

// Weighted coefficients of slot i = r (nx/2 + 1) + m of the one-sided spectrum at time offset dt
// (linear propagation e^{-i omega dt} when omega is given). Nyquist slots return live = false.
struct SlotCoef {
  bool live;
  int m, n;
  float k, invd;
  float2 we, wu, wv, ww, wt;
};

__device__ __forceinline__ SlotCoef slot_coef(int i, const float2* __restrict__ Ae,
                                              const float2* __restrict__ Ap, const float2* __restrict__ At,
                                              const double* __restrict__ omega, double dt, int nx, int ny,
                                              float kxs, float kys, float depth) {
  const int nxh1 = nx / 2 + 1;
  const int r = i / nxh1, m = i - r * nxh1;
  SlotCoef sc{};
  sc.live = !(m >= nx / 2 || (ny > 1 && r == ny / 2));    // Nyquist slots are ignored
  sc.invd = 1.f;
  if (!sc.live) return sc;
  float2 e = Ae[i], p = Ap[i], t = At[i];
  if (omega) {
    const double turns = omega[i] * dt * 0.15915494309189533577;
    const double frac = turns - rint(turns);
    float s, c;
    sincospif(2.f * float(frac), &s, &c);
    e = make_float2(fmaf(e.x, c, e.y * s), fmaf(e.y, c, -e.x * s));
    p = make_float2(fmaf(p.x, c, p.y * s), fmaf(p.y, c, -p.x * s));
    t = make_float2(fmaf(t.x, c, t.y * s), fmaf(t.y, c, -t.x * s));
  }
  const int n = ny > 1 ? (r < ny / 2 ? r : r - ny) : 0;
  const float kx = float(m) * kxs, ky = float(n) * kys;
  const float k = sqrtf(kx * kx + ky * ky);
  const float wgt = m == 0 ? 1.f : 2.f;
  sc.m = m;
  sc.n = n;
  sc.k = k;
  sc.invd = depth > 0.f ? 1.f / (1.f + expf(-2.f * k * depth)) : 1.f;
  sc.we = make_float2(wgt * e.x, wgt * e.y);
  sc.wu = make_float2(-wgt * kx * p.y, wgt * kx * p.x);     // c i kx A^phi
  sc.wv = make_float2(-wgt * ky * p.y, wgt * ky * p.x);     // c i ky A^phi
  sc.ww = make_float2(wgt * k * p.x, wgt * k * p.y);        // c |k| A^phi
  sc.wt = make_float2(wgt * t.x, wgt * t.y);                // c A^phit
  return sc;
}

// Depth factors as depth_factors (fft.cuh) with 1 / (1 + e^{-2 k h}) given.
template <bool FINITE>
__device__ __forceinline__ void direct_depth(float k, float z, float h, float invd, float& F, float& S) {
  const float kz = k * z;
  const float kz_lo = fmaf(k, z, -kz);
  float e1 = expf(kz);
  e1 = fmaf(e1, kz_lo, e1);
  if (!FINITE) {
    F = S = e1;
    return;
  }
  const float e2 = expf(-k * (z + 2.f * h));
  F = (e1 + e2) * invd;
  S = (e1 - e2) * invd;
}

// One (m, |n|) pair of modes, 96 bytes: per field the factors of (cos, sin)(phi) x (cos, sin)(theta),
//   q = (P, R, Q, S): C += F (P cos(theta) + Q sin(theta)), S += F (R cos(theta) + S sin(theta)),
// for eta (F = 1), u, v, w (F = the vertical factor S(z)), dphi/dt; then |k| and, in finite depth,
// 1 / (1 + e^{-2 |k| h}).
struct PairCoef {
  float4 q[5];
  float k, invd, pad_[2];
};
static_assert(sizeof(PairCoef) == 96, "pair record");

constexpr int kDirTile = 64;    // pairs per tile: a part of one row |n|, or whole rows of fewer modes
constexpr int kDirAnchor = 16;  // exact phase of theta every this many modes

// Pairs row by row, entry |n| nx/2 + m, zero past the last of them (n: whole tiles).
__global__ void k_direct_prep(const float2* __restrict__ Ae, const float2* __restrict__ Ap,
                              const float2* __restrict__ At, const double* __restrict__ omega,
                              double dt, int nx, int ny, float kxs, float kys, float depth, int64_t n_pairs, int64_t n,
                              PairCoef* __restrict__ out) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int m = int(i % (nx / 2)), row = int(i / (nx / 2));
  PairCoef pc{};
  pc.invd = 1.f;
  if (i < n_pairs) {
    const int nxh1 = nx / 2 + 1;
    const SlotCoef p = slot_coef(row * nxh1 + m, Ae, Ap, At, omega, dt, nx, ny, kxs, kys, depth);
    SlotCoef o{};                                  // the partner row -n (none for n = 0)
    if (row > 0) o = slot_coef((ny - row) * nxh1 + m, Ae, Ap, At, omega, dt, nx, ny, kxs, kys, depth);
    const float2 a[5] = {p.we, p.wu, p.wv, p.ww, p.wt}, b[5] = {o.we, o.wu, o.wv, o.ww, o.wt};
#pragma unroll
    for (int f = 0; f < 5; ++f)
      pc.q[f] = make_float4(a[f].x + b[f].x, b[f].y - a[f].y, -(a[f].y + b[f].y), b[f].x - a[f].x);
    pc.k = p.k;
    pc.invd = p.invd;
  }
  out[i] = pc;
}

struct DirectArgs {
  const PairCoef* pairs;
  int n_tiles, rows;         // tiles; rows |n|
  int mh, log_mh;            // modes per row |n| (a power of two)
  int tps;                   // tiles per split (blockIdx.y)
  const float* pts;
  float *o_eta, *o_u, *o_v, *o_w, *o_p;
  float* part;               // [splits][5][np] partial sums, or NULL: one split writes the outputs
  int64_t np;
  double inv_lx, inv_ly;
  float depth;
  int p_mode;
  float rho, g;
};

__device__ __forceinline__ void direct_store(const DirectArgs& a, int64_t i, float z, const float (&s)[5]) {
  if (a.o_eta) a.o_eta[i] = s[0];
  if (a.o_u) a.o_u[i] = s[1];
  if (a.o_v) a.o_v[i] = s[2];
  if (a.o_w) a.o_w[i] = s[3];
  if (a.o_p) {
    float p;
    if (a.p_mode == SWENSE_P_PHIT) {
      p = s[4];
    } else {
      p = -a.rho * (s[4] + 0.5f * (s[1] * s[1] + s[2] * s[2] + s[3] * s[3]));
      if (a.p_mode == SWENSE_P_TOTAL) p -= a.rho * a.g * z;
    }
    a.o_p[i] = p;
  }
}

// A tile of 64 pairs holds a part of one row |n| or, where rows are shorter (2 to 32 modes), several whole
// rows in turn; each took a tile of its own before, and a sea of 8 x 1024 modes 4.04 ms where one mode at a
// time had taken 1.28 (100,003 points, deep water; 0.40 now).
// Four points a thread: a pair's 22 coefficients come from shared memory as six 16-byte broadcasts,
// which occupy the shared-memory port for 24 cycles a warp, against about 31 FP32 operations a point;
// with one point a thread the port, not the FP32 pipe, would bound the kernel. blockIdx.y takes a
// contiguous range of tiles, so that few points still fill the GPU; the partial sums are added in
// order by k_direct_finish. 100,003 points x 4,032 modes in finite depth: 1538 -> 396 us (one mode at
// a time, one point a thread, the division of the depth factor per pair before).
constexpr int kDirThreads = 128;
constexpr int kDirPts = 4;

template <bool FINITE>
__global__ void __launch_bounds__(kDirThreads, 4) k_direct_fp32(DirectArgs a) {
  __shared__ PairCoef tile[2][kDirTile];
  const int64_t i0 = int64_t(blockIdx.x) * (kDirThreads * kDirPts) + threadIdx.x;
  unsigned X[kDirPts], Y[kDirPts];
  float z[kDirPts], sst[kDirPts], cst[kDirPts], sn[kDirPts], cs[kDirPts], tot[kDirPts][5];
#pragma unroll
  for (int p = 0; p < kDirPts; ++p) {
    const int64_t i = i0 + p * kDirThreads;
    const int64_t ic = i < a.np ? i : a.np - 1;
    X[p] = turn_fraction(a.pts[3 * ic], a.inv_lx);
    Y[p] = turn_fraction(a.pts[3 * ic + 1], a.inv_ly);
    z[p] = a.pts[3 * ic + 2];
    // e^{i 2 pi x / Lx}: the rotation from mode m to m + 1
    sincospif(2.f * (float(int(X[p])) * 2.3283064365386963e-10f), &sst[p], &cst[p]);
#pragma unroll
    for (int f = 0; f < 5; ++f) tot[p][f] = 0.f;
  }
  const int t0 = blockIdx.y * a.tps, t1 = min(t0 + a.tps, a.n_tiles);
  constexpr int kWords = int(sizeof(PairCoef)) * kDirTile / 16;
  auto load = [&](int t) {
    const uint4* src = reinterpret_cast<const uint4*>(a.pairs + size_t(t) * kDirTile);
    uint4* dst = reinterpret_cast<uint4*>(tile[t & 1]);
    for (int v = threadIdx.x; v < kWords; v += kDirThreads) cp_async16(dst + v, src + v, 16);
    cp_async_commit();
  };
  load(t0);
  for (int t = t0; t < t1; ++t) {
    if (t + 1 < t1) {
      load(t + 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int seg = min(a.mh, kDirTile);           // the tile's modes of one row
#pragma unroll 1
    for (int s0 = 0; s0 < kDirTile; s0 += seg) {
      const PairCoef* tc = tile[t & 1] + s0;
      const int64_t e0 = int64_t(t) * kDirTile + s0;
      const int n = int(e0 >> a.log_mh), m0 = int(e0 & (a.mh - 1));
      if (n >= a.rows) break;
      float2 acc[kDirPts][5];                      // (C, S) of each field
#pragma unroll
      for (int p = 0; p < kDirPts; ++p)
#pragma unroll
        for (int f = 0; f < 5; ++f) acc[p][f] = make_float2(0.f, 0.f);
#pragma unroll 1
      for (int j0 = 0; j0 < seg; j0 += kDirAnchor) {
#pragma unroll
        for (int p = 0; p < kDirPts; ++p)          // exact phase m X (mod 2^32)
          sincospif(2.f * (float(int(unsigned(m0 + j0) * X[p])) * 2.3283064365386963e-10f), &sn[p], &cs[p]);
#pragma unroll 1
        for (int j = j0; j < min(j0 + kDirAnchor, seg); ++j) {
          const PairCoef& c = tc[j];
          const float4 qe = c.q[0], qu = c.q[1], qv = c.q[2], qw = c.q[3], qt = c.q[4];
          const float k = c.k, invd = FINITE ? c.invd : 1.f;
#pragma unroll
          for (int p = 0; p < kDirPts; ++p) {
            float F, S;
            direct_depth<FINITE>(k, z[p], a.depth, invd, F, S);
            auto add = [&](float2& s, const float4& q, float cc, float ss) {
              s = pfma(make_float2(cc, cc), make_float2(q.x, q.y), s);
              s = pfma(make_float2(ss, ss), make_float2(q.z, q.w), s);
            };
            const float fc = F * cs[p], fs = F * sn[p];
            add(acc[p][0], qe, cs[p], sn[p]);
            add(acc[p][1], qu, fc, fs);
            add(acc[p][2], qv, fc, fs);
            add(acc[p][3], qw, FINITE ? S * cs[p] : fc, FINITE ? S * sn[p] : fs);
            add(acc[p][4], qt, fc, fs);
            const float c2 = fmaf(cs[p], cst[p], -sn[p] * sst[p]);
            sn[p] = fmaf(sn[p], cst[p], cs[p] * sst[p]);
            cs[p] = c2;
          }
        }
      }
#pragma unroll
      for (int p = 0; p < kDirPts; ++p) {
        float sy, cy;
        sincospif(2.f * (float(int(unsigned(n) * Y[p])) * 2.3283064365386963e-10f), &sy, &cy);
#pragma unroll
        for (int f = 0; f < 5; ++f) tot[p][f] += fmaf(cy, acc[p][f].x, sy * acc[p][f].y);
      }
    }
    __syncthreads();                               // tile (t & 1) is reloaded next iteration
  }
#pragma unroll
  for (int p = 0; p < kDirPts; ++p) {
    const int64_t i = i0 + p * kDirThreads;
    if (i >= a.np) continue;
    if (a.part) {
#pragma unroll
      for (int f = 0; f < 5; ++f) a.part[(int64_t(blockIdx.y) * 5 + f) * a.np + i] = tot[p][f];
    } else {
      direct_store(a, i, z[p], tot[p]);
    }
  }
}

// Sums of the splits in order, Bernoulli, outputs.
__global__ void __launch_bounds__(256) k_direct_finish(DirectArgs a, int splits) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= a.np) return;
  float s[5];
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    s[f] = a.part[int64_t(f) * a.np + i];
    for (int q = 1; q < splits; ++q) s[f] += a.part[(int64_t(q) * 5 + f) * a.np + i];
  }
  direct_store(a, i, a.pts[3 * i + 2], s);
}

// ------------------------------------------------------------------------------------------------
// Split-BF16 tensor-core path. The sums over modes are a contraction of the points-by-(mode,
// re/im) matrix A[p][2j] = cos(theta_pj) f_j(z_p), A[p][2j+1] = sin(theta_pj) f_j(z_p) with the
// (mode, re/im)-by-field matrix B[2j][c] = Re W_c[j], B[2j+1][c] = -Im W_c[j], c = u, v, w, phi_t
// (columns 4..7 zero). A is generated in registers directly in the m16n8k16 fragment layout (no
// shared-memory round trip) and both operands are split into BF16 hi + lo; three MMAs
// (hi.hi + hi.lo + lo.hi) accumulate in FP32, which leaves a relative error of about 2^-16 per
// product. eta has no depth factor and one column, so it is summed in FP32 on the side from the
// same phases. Finite depth writes the factors as a + b and a - b with a = e^{kz} / (1 + e^{-2kh})
// and b = a e^{-2k(z+h)} (so f = a + b for u, v, phi_t and g = a - b for w): A carries (cos, sin)
// times a and times b, and B's w column takes the sign flip on the b half.
//
// Table: modes in rows of constant n (Nyquist row skipped), m = 0 .. nx/2 - 1 padded with zero
// modes to a multiple of 8, cut into k-steps of KM = 8 modes (deep) or 4 modes (finite depth).
// Lane (g, q) of a k-step holds modes q and q + 4 (deep) or mode q in its a and b halves.
struct SplitStep {
  uint4 b[32];      // per lane: (b0 hi, b1 hi, b0 lo, b1 lo)
  float4 info[8];   // per mode of the step: (|k| log2 e, 1 / (1 + e^{-2kh}), W_eta)
};
static_assert(sizeof(SplitStep) == 640, "split step record");

constexpr int kSplitThreads = 256;
constexpr int kSplitTiles = 2;     // 16-point MMA tiles per warp
constexpr int kSplitStage = 32;    // k-steps per shared-memory stage (double-buffered)
constexpr int kSplitAnchor = 16;   // exact phase every this many k-steps

// 2^x (PTX ex2.approx: relative error about 2^-22, far below the split products' 2^-16)
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float2 pick_w(const SlotCoef& sc, int c) {
  return c == 0 ? sc.wu : c == 1 ? sc.wv : c == 2 ? sc.ww : c == 3 ? sc.wt : make_float2(0.f, 0.f);
}

__global__ void k_direct_prep_split(const float2* __restrict__ Ae, const float2* __restrict__ Ap,
                                    const float2* __restrict__ At, const double* __restrict__ omega,
                                    double dt, int nx, int ny, float kxs, float kys, float depth,
                                    int km, int spr, int nsteps, SplitStep* __restrict__ out) {
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  if (gt >= nsteps * 32) return;
  const int s = gt >> 5, L = gt & 31;
  const int ri = s / spr, m0 = (s - ri * spr) * km;
  const int r = (ny > 1 && ri >= ny / 2) ? ri + 1 : ri;
  const int nxh1 = nx / 2 + 1;
  auto coef = [&](int j) {
    const int m = m0 + j;
    SlotCoef sc{};
    if (m < nx / 2) sc = slot_coef(r * nxh1 + m, Ae, Ap, At, omega, dt, nx, ny, kxs, kys, depth);
    return sc;                                   // not live: all weights zero
  };
  const int g = L >> 2, q = L & 3;
  const SlotCoef s0 = coef(q);
  const float2 w0 = pick_w(s0, g);
  float2 w1;
  if (km == 8) {
    w1 = pick_w(coef(q + 4), g);
  } else {
    w1 = g == 2 ? make_float2(-w0.x, -w0.y) : w0;    // b half: w column changes sign
  }
  unsigned h0, l0, h1, l1;
  bf2_split(w0.x, -w0.y, h0, l0);
  bf2_split(w1.x, -w1.y, h1, l1);
  out[s].b[L] = make_uint4(h0, h1, l0, l1);
  if (L < 8) {
    float4 inf = make_float4(0.f, 1.f, 0.f, 0.f);
    if (L < km) {
      const SlotCoef sc = coef(L);
      if (sc.live) inf = make_float4(sc.k * 1.4426950408889634f, sc.invd, sc.we.x, sc.we.y);
    }
    out[s].info[L] = inf;
  }
}

struct SplitArgs {
  const SplitStep* steps;
  int nsteps, spr, ny;
  const float* pts;
  float *o_eta, *o_u, *o_v, *o_w, *o_p;
  int64_t np;
  double inv_lx, inv_ly;
  float depth;
  int p_mode;
  float rho, g;
  // points sorted by the tensor-core path: output i goes to perm[i], and only the tiles of
  // tile_pts points that tile_bad marks are written (NULL: caller's order, every point)
  const int32_t* perm;
  const uint8_t* tile_bad;
  int tile_pts;
};

template <bool FINITE>
__global__ void __launch_bounds__(kSplitThreads, 2) k_direct_split(SplitArgs a) {
  constexpr int KM = FINITE ? 4 : 8;
  constexpr int TT = kSplitTiles;
  constexpr int JN = FINITE ? 1 : 2;               // modes per lane per k-step
  __shared__ SplitStep stage[2][kSplitStage];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, q = lane & 3;
  const int64_t pbase = (int64_t(blockIdx.x) * (kSplitThreads / 32) + warp) * (16 * TT);
  bool write = true;
  if (a.tile_bad) {
    // the block's points span whole warps of one tile each; leave at once (before any barrier)
    // unless one of the block's tiles is marked
    const int64_t b0 = int64_t(blockIdx.x) * (kSplitThreads / 32) * (16 * TT);
    const int64_t t0 = b0 / a.tile_pts, t1 = (std::min(b0 + (kSplitThreads / 32) * (16 * TT), a.np) - 1) / a.tile_pts;
    bool any = false;
    for (int64_t tt = t0; tt <= t1; ++tt) any |= a.tile_bad[tt] != 0;
    if (!any) return;
    write = pbase < a.np && a.tile_bad[pbase / a.tile_pts] != 0;
  }

  unsigned X[TT][2], Y[TT][2];
  float z[TT][2], stc[TT][2], sts[TT][2];
  float pc[TT][2][JN], ps[TT][2][JN];
#pragma unroll
  for (int t = 0; t < TT; ++t)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t i = pbase + 16 * t + g + 8 * h;
      float x = 0.f, y = 0.f, zz = 0.f;
      if (i < a.np) {
        x = a.pts[3 * i];
        y = a.pts[3 * i + 1];
        zz = a.pts[3 * i + 2];
      }
      X[t][h] = turn_fraction(x, a.inv_lx);
      Y[t][h] = turn_fraction(y, a.inv_ly);
      z[t][h] = zz;
      // phase step for m -> m + KM
      sincospif(2.f * (float(int(unsigned(KM) * X[t][h])) * 2.3283064365386963e-10f), &sts[t][h], &stc[t][h]);
#pragma unroll
      for (int j = 0; j < JN; ++j) pc[t][h][j] = 1.f, ps[t][h][j] = 0.f;
    }
  float run[TT][4], eta_run[TT][2];
#pragma unroll
  for (int t = 0; t < TT; ++t) {
#pragma unroll
    for (int e = 0; e < 4; ++e) run[t][e] = 0.f;
    eta_run[t][0] = eta_run[t][1] = 0.f;
  }

  const int nchunks = (a.nsteps + kSplitStage - 1) / kSplitStage;
  auto load_chunk = [&](int c) {
    const int cnt = min(kSplitStage, a.nsteps - c * kSplitStage);
    const uint4* src = reinterpret_cast<const uint4*>(a.steps + size_t(c) * kSplitStage);
    uint4* dst = reinterpret_cast<uint4*>(stage[c & 1]);
    for (int v = threadIdx.x; v < cnt * 40; v += kSplitThreads) cp_async16(dst + v, src + v, 16);
    cp_async_commit();
  };
  load_chunk(0);
  int ri = 0, sidx = 0;                             // table row and step within it of step s
  for (int c = 0; c < nchunks; ++c) {
    if (c + 1 < nchunks) {
      load_chunk(c + 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const SplitStep* st = stage[c & 1];
    const int cnt = min(kSplitStage, a.nsteps - c * kSplitStage);
    float acc[TT][4], eta_acc[TT][2];
#pragma unroll
    for (int t = 0; t < TT; ++t) {
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[t][e] = 0.f;
      eta_acc[t][0] = eta_acc[t][1] = 0.f;
    }
    for (int sl = 0; sl < cnt; ++sl) {
      if (sidx % kSplitAnchor == 0) {
        // exact phase (m X + n Y) mod 2^32 of this lane's modes
        const int r = (a.ny > 1 && ri >= a.ny / 2) ? ri + 1 : ri;
        const int n = a.ny > 1 ? (r < a.ny / 2 ? r : r - a.ny) : 0;
#pragma unroll
        for (int t = 0; t < TT; ++t)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < JN; ++j) {
              const unsigned m = unsigned(sidx * KM + q + 4 * j);
              const unsigned ph = m * X[t][h] + unsigned(n) * Y[t][h];
              sincospif(2.f * (float(int(ph)) * 2.3283064365386963e-10f), &ps[t][h][j], &pc[t][h][j]);
            }
      } else {
#pragma unroll
        for (int t = 0; t < TT; ++t)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < JN; ++j) {
              const float c2 = fmaf(pc[t][h][j], stc[t][h], -ps[t][h][j] * sts[t][h]);
              ps[t][h][j] = fmaf(ps[t][h][j], stc[t][h], pc[t][h][j] * sts[t][h]);
              pc[t][h][j] = c2;
            }
      }
      const uint4 bf = st[sl].b[lane];
      float4 inf[JN];
#pragma unroll
      for (int j = 0; j < JN; ++j) inf[j] = st[sl].info[q + 4 * j];
#pragma unroll
      for (int t = 0; t < TT; ++t) {
        float v[2][2][2];                          // [register pair][h][cos/sin]
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float zz = z[t][h];
          if constexpr (!FINITE) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const float f = ex2(inf[j].x * zz);
              v[j][h][0] = pc[t][h][j] * f;
              v[j][h][1] = ps[t][h][j] * f;
              eta_acc[t][h] = fmaf(inf[j].z, pc[t][h][j], fmaf(-inf[j].w, ps[t][h][j], eta_acc[t][h]));
            }
          } else {
            const float k = inf[0].x;
            const float fa = ex2(k * zz) * inf[0].y;
            const float fb = fa * ex2(-2.f * k * (zz + a.depth));
            v[0][h][0] = pc[t][h][0] * fa;
            v[0][h][1] = ps[t][h][0] * fa;
            v[1][h][0] = pc[t][h][0] * fb;
            v[1][h][1] = ps[t][h][0] * fb;
            eta_acc[t][h] = fmaf(inf[0].z, pc[t][h][0], fmaf(-inf[0].w, ps[t][h][0], eta_acc[t][h]));
          }
        }
        unsigned ahi[4], alo[4];
        bf2_split(v[0][0][0], v[0][0][1], ahi[0], alo[0]);   // (g, 2q..2q+1)
        bf2_split(v[0][1][0], v[0][1][1], ahi[1], alo[1]);   // (g+8, 2q..2q+1)
        bf2_split(v[1][0][0], v[1][0][1], ahi[2], alo[2]);   // (g, 2q+8..2q+9)
        bf2_split(v[1][1][0], v[1][1][1], ahi[3], alo[3]);   // (g+8, 2q+8..2q+9)
        mma16816(acc[t], ahi, bf.x, bf.y);
        mma16816(acc[t], ahi, bf.z, bf.w);
        mma16816(acc[t], alo, bf.x, bf.y);
      }
      if (++sidx == a.spr) {                       // next step: next table row
        sidx = 0;
        ++ri;
      }
    }
#pragma unroll
    for (int t = 0; t < TT; ++t) {
#pragma unroll
      for (int e = 0; e < 4; ++e) run[t][e] += acc[t][e];
      eta_run[t][0] += eta_acc[t][0];
      eta_run[t][1] += eta_acc[t][1];
    }
    __syncthreads();                               // stage (c & 1) is reloaded next iteration
  }

#pragma unroll
  for (int t = 0; t < TT; ++t) {
    float e0 = eta_run[t][0], e1 = eta_run[t][1];
    e0 += __shfl_xor_sync(0xffffffffu, e0, 1);
    e0 += __shfl_xor_sync(0xffffffffu, e0, 2);
    e1 += __shfl_xor_sync(0xffffffffu, e1, 1);
    e1 += __shfl_xor_sync(0xffffffffu, e1, 2);
    // lane q = 0 holds (u, v) of rows g and g + 8, lane q = 1 holds (w, phi_t)
    const float w0 = __shfl_down_sync(0xffffffffu, run[t][0], 1);
    const float t0 = __shfl_down_sync(0xffffffffu, run[t][1], 1);
    const float w1 = __shfl_down_sync(0xffffffffu, run[t][2], 1);
    const float t1 = __shfl_down_sync(0xffffffffu, run[t][3], 1);
    if (q != 0 || !write) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t ii = pbase + 16 * t + g + 8 * h;
      if (ii >= a.np) continue;
      const int64_t i = a.perm ? int64_t(a.perm[ii]) : ii;
      const float uu = run[t][2 * h], vv = run[t][2 * h + 1];
      const float ww = h ? w1 : w0, tt = h ? t1 : t0;
      if (a.o_eta) a.o_eta[i] = h ? e1 : e0;
      if (a.o_u) a.o_u[i] = uu;
      if (a.o_v) a.o_v[i] = vv;
      if (a.o_w) a.o_w[i] = ww;
      if (a.o_p) {
        float p;
        if (a.p_mode == SWENSE_P_PHIT) {
          p = tt;
        } else {
          p = -a.rho * (tt + 0.5f * (uu * uu + vv * vv + ww * ww));
          if (a.p_mode == SWENSE_P_TOTAL) p -= a.rho * a.g * z[t][h];
        }
        a.o_p[i] = p;
      }
    }
  }
}

}  // namespace
}  // namespace swense

using namespace swense;

namespace {

int direct_split_impl(const swense_modes* md, double t, const float* pts, const int32_t* perm,
                      const uint8_t* tile_bad, int tile_pts, int64_t np, float* eta, float* u,
                      float* v, float* w, float* p, int32_t p_mode, double rho, double grav,
                      cudaStream_t stream, size_t ws_offset) {
  const int nx = md->nx, ny = md->ny;
  const bool finite = md->depth > 0;
  const int km = finite ? 4 : 8;
  const int rm = ((nx / 2 + 7) / 8) * 8;        // modes per table row, padded to a multiple of 8
  const int spr = rm / km;
  const int nrows = ny > 1 ? ny - 1 : 1;        // Nyquist row skipped
  const int64_t nsteps = int64_t(nrows) * spr;
  if (nsteps * 32 >= (int64_t(1) << 31)) return fail(SWENSE_ERR_SIZE, "too many modes for the split table");
  void* ws = nullptr;
  int st = workspace(ws_offset + size_t(nsteps) * sizeof(SplitStep), stream, &ws);
  if (st) return st;
  SplitStep* steps = reinterpret_cast<SplitStep*>(static_cast<char*>(ws) + ws_offset);
  const float depth = finite ? float(md->depth) : 0.f;
  k_direct_prep_split<<<unsigned((nsteps * 32 + 255) / 256), 256, 0, stream>>>(
      reinterpret_cast<const float2*>(md->A_eta), reinterpret_cast<const float2*>(md->A_phi),
      reinterpret_cast<const float2*>(md->A_phit), md->omega, t - md->t_ref, nx, ny,
      float(6.283185307179586476925 / md->Lx), ny > 1 ? float(6.283185307179586476925 / md->Ly) : 0.f,
      depth, km, spr, int(nsteps), steps);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  SplitArgs a{};
  a.steps = steps;
  a.nsteps = int(nsteps);
  a.spr = spr;
  a.ny = ny;
  a.pts = pts;
  a.o_eta = eta;
  a.o_u = u;
  a.o_v = v;
  a.o_w = w;
  a.o_p = p;
  a.np = np;
  a.inv_lx = 1.0 / md->Lx;
  a.inv_ly = ny > 1 ? 1.0 / md->Ly : 0.0;
  a.depth = depth;
  a.p_mode = p_mode;
  a.rho = float(rho);
  a.g = float(grav);
  a.perm = perm;
  a.tile_bad = tile_bad;
  a.tile_pts = tile_pts;
  const int64_t per_cta = int64_t(kSplitThreads / 32) * 16 * kSplitTiles;
  const int64_t blocks = (np + per_cta - 1) / per_cta;
  if (blocks >= (int64_t(1) << 31)) return fail(SWENSE_ERR_SIZE, "too many points for one call");
  if (finite) k_direct_split<true><<<unsigned(blocks), kSplitThreads, 0, stream>>>(a);
  else k_direct_split<false><<<unsigned(blocks), kSplitThreads, 0, stream>>>(a);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

}  // namespace

namespace swense {

size_t split_table_bytes(const swense_modes* md) {
  const int km = md->depth > 0 ? 4 : 8;
  const int rm = ((md->nx / 2 + 7) / 8) * 8;
  const int nrows = md->ny > 1 ? md->ny - 1 : 1;
  return size_t(nrows) * (rm / km) * sizeof(SplitStep);
}

int direct_split_sorted(const swense_modes* md, double t, const float* srt, const int32_t* perm,
                        const uint8_t* tile_bad, int tile_pts, int64_t np, float* eta, float* u, float* v,
                        float* w, float* p, int32_t p_mode, double rho, double grav, cudaStream_t stream,
                        size_t ws_offset) {
  static_assert((kSplitThreads / 32) * 16 * kSplitTiles % 32 == 0, "warps of 32 points");
  if (tile_pts % (16 * kSplitTiles)) return fail(SWENSE_ERR_ARG, "tile size");
  // the workspace already holds the sorted points and the tensor-core path's tables, which this
  // launch reads: its own table goes at ws_offset, after them (the caller sized the workspace for
  // both, so that nothing here grows it and frees the buffers in use)
  return direct_split_impl(md, t, srt, perm, tile_bad, tile_pts, np, eta, u, v, w, p, p_mode, rho, grav,
                           stream, ws_offset);
}

}  // namespace swense

extern "C" int swense_direct(const swense_modes* md, double t, const float* pts, int64_t np,
                             float* eta, float* u, float* v, float* w, float* p, int32_t p_mode,
                             double rho, double grav, int32_t precision, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (!md || !md->A_eta || !md->A_phi || !md->A_phit) return fail(SWENSE_ERR_ARG, "NULL modes");
  if (np < 0) return fail(SWENSE_ERR_ARG, "np must be >= 0");
  if (np > 0 && !pts) return fail(SWENSE_ERR_ARG, "NULL pts");
  const int nx = md->nx, ny = md->ny;
  if (!is_pow2(nx) || nx < 4 || !is_pow2(ny) || (ny != 1 && ny < 4) || nx > (1 << 16) || ny > (1 << 16))
    return fail(SWENSE_ERR_SIZE, "nx must be a power of two in [4, 65536], ny 1 or a power of two in [4, 65536]");
  if (md->n_snap != 1) return fail(SWENSE_ERR_ARG, "swense_direct takes one snapshot (n_snap = 1)");
  if (!(md->Lx > 0) || !std::isfinite(md->Lx) || (ny > 1 && (!(md->Ly > 0) || !std::isfinite(md->Ly))))
    return fail(SWENSE_ERR_ARG, "domain lengths must be finite and positive");
  if (!std::isfinite(t) || !std::isfinite(md->depth) || !std::isfinite(rho) || !std::isfinite(grav))
    return fail(SWENSE_ERR_ARG, "non-finite t, depth, rho or g");
  if (p_mode != SWENSE_P_DYN && p_mode != SWENSE_P_PHIT && p_mode != SWENSE_P_TOTAL)
    return fail(SWENSE_ERR_ARG, "unknown p_mode");
  if (precision != SWENSE_DIRECT_FP32 && precision != SWENSE_DIRECT_SPLIT_BF16 &&
      precision != SWENSE_DIRECT_SPLIT_BF16_PAIRWISE)
    return fail(SWENSE_ERR_ARG, "unknown precision");
  if (np == 0) return SWENSE_OK;
  if (precision == SWENSE_DIRECT_SPLIT_BF16)
    return direct_tc(md, t, pts, np, eta, u, v, w, p, p_mode, rho, grav, stream);
  if (precision == SWENSE_DIRECT_SPLIT_BF16_PAIRWISE)
    return direct_split_impl(md, t, pts, nullptr, nullptr, 0, np, eta, u, v, w, p, p_mode, rho, grav, stream, 0);
  const int rows = ny > 1 ? ny / 2 : 1;           // |n| = 0 .. ny/2 - 1 (the Nyquist row is ignored)
  const int64_t n_pairs = int64_t(rows) * (nx / 2), n_tiles = (n_pairs + kDirTile - 1) / kDirTile;
  if (n_tiles >= (int64_t(1) << 31)) return fail(SWENSE_ERR_SIZE, "too many modes for one call");
  const int64_t blocks = (np + kDirThreads * kDirPts - 1) / (kDirThreads * kDirPts);
  if (blocks >= (int64_t(1) << 31)) return fail(SWENSE_ERR_SIZE, "too many points for one call");
  int dev = 0, sms = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  SWENSE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // four blocks fit an SM: split the modes until the grid fills the GPU about three times over (a
  // partly filled last wave then costs little), at least one tile a split
  const int64_t want = std::max<int64_t>(1, (int64_t(sms) * 12 + blocks - 1) / blocks);
  const int64_t tps = (n_tiles + std::min(want, n_tiles) - 1) / std::min(want, n_tiles);
  const int splits = int((n_tiles + tps - 1) / tps);
  const size_t b_pairs = size_t(n_tiles) * kDirTile * sizeof(PairCoef);
  const size_t b_part = splits > 1 ? size_t(splits) * 5 * size_t(np) * sizeof(float) : 0;
  void* ws = nullptr;
  int st = workspace(b_pairs + b_part, stream, &ws);
  if (st) return st;
  PairCoef* pairs = static_cast<PairCoef*>(ws);
  const float depth = md->depth > 0 ? float(md->depth) : 0.f;
  k_direct_prep<<<unsigned((n_tiles * kDirTile + 255) / 256), 256, 0, stream>>>(
      reinterpret_cast<const float2*>(md->A_eta), reinterpret_cast<const float2*>(md->A_phi),
      reinterpret_cast<const float2*>(md->A_phit), md->omega, t - md->t_ref, nx, ny,
      float(6.283185307179586476925 / md->Lx), ny > 1 ? float(6.283185307179586476925 / md->Ly) : 0.f,
      depth, n_pairs, n_tiles * kDirTile, pairs);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  DirectArgs a{};
  a.pairs = pairs;
  a.n_tiles = int(n_tiles);
  a.mh = nx / 2;
  a.log_mh = ilog2(nx / 2);
  a.rows = rows;
  a.tps = int(tps);
  a.pts = pts;
  a.o_eta = eta;
  a.o_u = u;
  a.o_v = v;
  a.o_w = w;
  a.o_p = p;
  a.part = splits > 1 ? reinterpret_cast<float*>(static_cast<char*>(ws) + b_pairs) : nullptr;
  a.np = np;
  a.inv_lx = 1.0 / md->Lx;
  a.inv_ly = ny > 1 ? 1.0 / md->Ly : 0.0;
  a.depth = depth;
  a.p_mode = p_mode;
  a.rho = float(rho);
  a.g = float(grav);
  const dim3 grid{unsigned(blocks), unsigned(splits), 1u};
  if (depth > 0.f) k_direct_fp32<true><<<grid, kDirThreads, 0, stream>>>(a);
  else k_direct_fp32<false><<<grid, kDirThreads, 0, stream>>>(a);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  if (splits > 1) {
    k_direct_finish<<<unsigned((np + 255) / 256), 256, 0, stream>>>(a, splits);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);
  }
  return SWENSE_OK;
}
