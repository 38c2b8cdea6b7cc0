// Stage 2 of the reconstruction: grid fields -> arbitrary points (cell and face centres).
//
// Paper: reconstruction section, step "Interpolation" (HOS grid -> CFD mesh). Scheme: tensor
// product 4-point Lagrange in x, y (uniform, periodic) and z (arbitrary levels, stencil shifted
// inside the level range at the ends), Lagrange over the stored time levels, then Bernoulli.
//
// A point's horizontal cell is located with a compensated FP32 product (x * nx_r / Lx as hi + lo) so
// the in-cell offset keeps ~1e-7 absolute accuracy even for points hundreds of cells from the origin.
// Points come in chunks of 1024 neighbours: a chunk whose stencils fit a tile gathers from shared memory
// (k_interp_box), others straight from the grid, four lanes a point (k_interp_global), or, many points on
// a fine grid, from planes collapsed in z that the chunks of a layer share (k_interp_planes).
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <vector>

#include "internal.cuh"
#include "mlp.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace swense {
namespace {

// z lookup: ZLUT equal buckets over [z_0, z_{nz-1}]; lut[b] = largest level index j with
// z_j <= z_0 + b h. A point starts its search one bucket below its own (so rounding of the
// bucket index cannot place it past its level) and steps up: one or two steps for any level
// spacing that is not much finer than h.
constexpr int ZLUT = 256;

// Level tables, built on the host once per call and passed as a kernel parameter: levels,
// inverse Lagrange denominators of each 4-level window (inv[j] for nodes j..j+3) and the lookup.
struct Levels {
  float z[SWENSE_MAX_LEVELS];
  float4 inv[SWENSE_MAX_LEVELS];
  unsigned lut4[ZLUT / 4];          // lut bytes, four per word
  float z0, inv_h;
};

struct InterpArgs {
  const float4* nodes;   // [TL][nz][Nyr][Nxr]
  const float* eta;      // [TL][Nyr][Nxr]
  const float* pts;      // [np][3]
  float* o_eta;
  float* o_u;
  float* o_v;
  float* o_w;
  float* o_p;
  unsigned long long* n_oor;
  const int32_t* perm;   // output index of each point (NULL: identity); points are pre-sorted
  int64_t np;
  int Nxr, Nyr, nz, n_tl;
  float sx_hi, sx_lo, sy_hi, sy_lo;   // nx_r / Lx and ny_r / Ly as hi + lo
  float wt[SWENSE_MAX_TL];            // time weights
  int p_mode;
  float rho, g;
  int spline;            // cubic B-spline weights in x and y (grid holds spline coefficients)
  int p2;                // both node counts are powers of two (mask wrap; the kernels' <true>)
};

// Periodic node index i mod n. Grids whose horizontal node counts are powers of two (every
// grid zero-padded by a power of two) wrap with a mask; the others (padding factors 3, 5, 6, 7)
// take the remainder. The kernels are instantiated for both, so the mask path is unchanged.
template <bool P2>
__device__ __forceinline__ int wrapi(int i, int n) {
  if constexpr (P2) {
    return i & (n - 1);
  } else {
    const int r = i % n;
    return r < 0 ? r + n : r;
  }
}

// Cell index (mod n) and in-cell offset f in [0, 1] of coordinate x for the node spacing
// 1 / (s_hi + s_lo); the product is carried as an unevaluated sum (fma residual).
template <bool P2 = true>
__device__ __forceinline__ void locate(float x, float s_hi, float s_lo, int n, int& i0, float& f) {
  const float p = x * s_hi;
  const float e = fmaf(x, s_hi, -p);
  const float lo = fmaf(x, s_lo, e);
  const float fl = floorf(p);
  f = (p - fl) + lo;
  int i = int(fl);
  if (f < 0.f) {
    f += 1.f;
    i -= 1;
  } else if (f >= 1.f) {
    f -= 1.f;
    i += 1;
  }
  i0 = wrapi<P2>(i, n);
}

// Uniform cubic B-spline basis of the coefficients -1, 0, 1, 2 at f.
__device__ __forceinline__ void bspline4(float f, float w[4]) {
  const float g = 1.f - f, f2 = f * f, f3 = f2 * f;
  w[0] = g * g * g * (1.f / 6.f);
  w[1] = fmaf(0.5f * f3, 1.f, fmaf(-f2, 1.f, 2.f / 3.f));      // (3f^3 - 6f^2 + 4) / 6
  w[2] = fmaf(-0.5f, f3, fmaf(0.5f, f2, fmaf(0.5f, f, 1.f / 6.f)));   // (-3f^3 + 3f^2 + 3f + 1) / 6
  w[3] = f3 * (1.f / 6.f);
}

// Lagrange basis of the nodes -1, 0, 1, 2 at f.
__device__ __forceinline__ void lagrange4_uniform(float f, float w[4]) {
  const float fm1 = f - 1.f, fm2 = f - 2.f, fp1 = f + 1.f;
  w[0] = -f * fm1 * fm2 * (1.f / 6.f);
  w[1] = 0.5f * fp1 * fm1 * fm2;
  w[2] = -0.5f * fp1 * f * fm2;
  w[3] = fp1 * f * fm1 * (1.f / 6.f);
}

// Lagrange basis of the 4 arbitrary nodes zn at z; inv holds 1 / prod_{b != a} (zn[a] - zn[b]).
__device__ __forceinline__ void lagrange4(const float zn[4], float4 inv, float z, float w[4]) {
  const float d0 = z - zn[0], d1 = z - zn[1], d2 = z - zn[2], d3 = z - zn[3];
  w[0] = (d1 * d2 * d3) * inv.x;
  w[1] = (d0 * d2 * d3) * inv.y;
  w[2] = (d0 * d1 * d3) * inv.z;
  w[3] = (d0 * d1 * d2) * inv.w;
}

// Shared-memory copy of the levels and, per stencil start j0, the inverse Lagrange
// denominators of the levels j0 .. j0+3 (computed once per CTA: no divisions per point).
struct LevelTables {
  float z[SWENSE_MAX_LEVELS];
  float4 inv[SWENSE_MAX_LEVELS];
  alignas(4) unsigned char lut[ZLUT];
  float z0, inv_h;
};
static_assert(sizeof(LevelTables) == sizeof(Levels) && sizeof(Levels) % 16 == 0 &&
                  offsetof(LevelTables, inv) == offsetof(Levels, inv) && offsetof(LevelTables, lut) == offsetof(Levels, lut4) &&
                  offsetof(LevelTables, z0) == offsetof(Levels, z0),
              "the same layout");

// The level tables of a kernel parameter by a generic pointer: loads through it are ordinary cached
// loads, where per-thread indices into the parameter itself serialise on the constant bank, a lane
// at a time.
__device__ __forceinline__ const LevelTables* level_tables(const Levels& L) {
  const LevelTables* p = reinterpret_cast<const LevelTables*>(&L);
  asm volatile("" : "+l"(p));
  return p;
}

// Copy of the level tables in shared memory.
__device__ __forceinline__ void fill_level_tables(LevelTables& T, const Levels& L) {
  const uint4* src = reinterpret_cast<const uint4*>(level_tables(L));
  uint4* dst = reinterpret_cast<uint4*>(&T);
  for (int i = threadIdx.x; i < int(sizeof(LevelTables) / 16); i += blockDim.x) dst[i] = src[i];
}

struct PointCell {
  int ix, iy, j0;       // first stencil node in x, y (before the -1 shift) and first level
  float wx[4], wy[4], wz[4];
  bool inside;
};

// Horizontal part of a point's cell: first stencil nodes and weights in x and y.
template <bool P2 = true>
__device__ __forceinline__ void point_xy(const InterpArgs& a, float x, float y, PointCell& c) {
  float fx;
  locate<P2>(x, a.sx_hi, a.sx_lo, a.Nxr, c.ix, fx);
  if (a.spline) bspline4(fx, c.wx); else lagrange4_uniform(fx, c.wx);
  c.iy = 0;
  c.wy[0] = 1.f;
  c.wy[1] = c.wy[2] = c.wy[3] = 0.f;
  if (a.Nyr > 1) {
    float fy;
    locate<P2>(y, a.sy_hi, a.sy_lo, a.Nyr, c.iy, fy);
    if (a.spline) bspline4(fy, c.wy); else lagrange4_uniform(fy, c.wy);
  }
}

// Vertical part: first stencil level j0, level weights and whether z lies inside the levels.
__device__ __forceinline__ void point_level(const InterpArgs& a, const LevelTables& T, float z,
                                            PointCell& c) {
  const float* zs = T.z;
  // bracket: largest j with zs[j] <= z, clamped to [0, nz-2]; stencil j0 = clamp(j-1, 0, nz-4)
  const int nz = a.nz;
  c.inside = (z >= zs[0]) && (z <= zs[nz - 1]);
  const float bf = fminf(fmaxf((z - T.z0) * T.inv_h, 0.f), float(ZLUT - 1));   // NaN -> 0
  int jj = T.lut[max(int(bf) - 1, 0)];
  while (jj + 1 < nz && zs[jj + 1] <= z) ++jj;
  const int j = min(jj, nz - 2);
  c.j0 = min(max(j - 1, 0), nz - 4);
  float zn[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) zn[q] = zs[c.j0 + q];
  lagrange4(zn, T.inv[c.j0], z, c.wz);
}

template <bool P2 = true>
__device__ __forceinline__ PointCell point_cell(const InterpArgs& a, const LevelTables& T, float x,
                                                float y, float z) {
  PointCell c;
  point_xy<P2>(a, x, y, c);
  point_level(a, T, z, c);
  return c;
}

__device__ __forceinline__ void store_point(const InterpArgs& a, int64_t i, float4 acc,
                                            float acc_eta, float z, bool inside) {
  if (a.perm) i = a.perm[i];
  if (!inside) {
    const float qnan = __int_as_float(0x7fc00000);
    acc = make_float4(qnan, qnan, qnan, qnan);
    if (a.n_oor) atomicAdd(a.n_oor, 1ULL);
  }
  if (a.o_eta) a.o_eta[i] = acc_eta;
  if (a.o_u) a.o_u[i] = acc.x;
  if (a.o_v) a.o_v[i] = acc.y;
  if (a.o_w) a.o_w[i] = acc.z;
  if (a.o_p) {
    float p;
    if (a.p_mode == SWENSE_P_PHIT) {
      p = acc.w;
    } else {
      const float q2 = acc.x * acc.x + acc.y * acc.y + acc.z * acc.z;
      p = -a.rho * (acc.w + 0.5f * q2);
      if (a.p_mode == SWENSE_P_TOTAL) p -= a.rho * a.g * z;
    }
    a.o_p[i] = p;
  }
}

// Box-staged gather for spatially coherent point sets (mesh order). Each CTA takes BOX_PTS
// consecutive points, finds the bounding box of their stencils, loads that box of the grid into
// shared memory already blended in time (sum_t w_t G_t, exact reordering of the linear sums),
// then evaluates every point from shared memory, where threads of a warp mostly share cells
// (broadcast reads). A CTA whose box exceeds BOX_NODES falls back to global gathers.
constexpr int BOX_THREADS = 256;
constexpr int BOX_PPT = 4;                         // points per thread
constexpr int BOX_PTS = BOX_THREADS * BOX_PPT;
constexpr int BOX_NODES = 4096;                    // float4 nodes (64 KB; 99 % of the 1024-point mesh chunks fit)
constexpr int BOX_COLS = BOX_NODES / 4;             // eta columns (a box has at least 4 levels)
constexpr size_t BOX_SMEM = size_t(BOX_NODES) * sizeof(float4) + size_t(BOX_COLS) * sizeof(float);
// Tile of the batched gather: points binned in rows of tiles put 1024 of them in a box of
// (256 / d + 3) x 7 x 4 nodes at d points per node, or of whole rows of a narrow grid; 6400 nodes
// (two CTAs per SM) hold that from d = 1.1 on, 4096 only from 1.8 on.
constexpr int BATCH_NODES = 6400, BATCH_COLS = BATCH_NODES / 4;
constexpr size_t BATCH_SMEM = size_t(BATCH_NODES) * sizeof(float4) + size_t(BATCH_COLS) * sizeof(float);
// Level-flat chunks (every point at the same z, as the cell and face centres of one layer of an
// extruded mesh) stage one z-collapsed plane instead of the box: float4 columns and eta.
constexpr int FLAT_COLS = 3456;
static_assert(size_t(FLAT_COLS) * (sizeof(float4) + sizeof(float)) <= BOX_SMEM, "flat plane fits the tile");
// Chunks whose points lie at two z values (a chunk that straddles two layers) stage two
// collapsed planes and one eta plane.
constexpr int FLAT2_COLS = 1920;
static_assert(size_t(FLAT2_COLS) * (2 * sizeof(float4) + sizeof(float)) <= BOX_SMEM, "two planes fit the tile");

// One chunk's plan, 16 bytes: x0, y0 (first staged node, wrapped), l0 | FLAT_BIT, extents.
//   3-D box:  w = bx | by << 11 | bz << 22 (bz >= 4), z = l0
//   flat:     w = bx | by << 12 (4 levels from l0), z = l0 | FLAT_BIT
//   two z:    w = bx | by << 12, z = FLAT_BIT | FLAT2_BIT (the z values are those of the chunk's
//             first and last points; their level windows are looked up by the gather)
//   neither fits the tile: w < 0 (global gathers): -1, or for one or two z values the extents all the
//             same, w = 1 << 31 | bx | by << 14, z = FLAT_BIT (| FLAT2_BIT); ROWS_BIT of z besides where the
//             points follow one another along the grid's rows
constexpr int FLAT_BIT = 1 << 30;
constexpr int FLAT2_BIT = 1 << 29;
constexpr int ROWS_BIT = 1 << 28;
// ROWS_BIT: the chunk's box spans half the grid's row length and more, and its first 32 points go ROWS_RATIO times
// as far along x as along y. So do layers (45 and more), and points binned by rows of tiles (18 and more); points
// close by in all directions (Morton order, the cells of a mesh) and points in no order do not.
constexpr int ROWS_RATIO = 6;
struct BoxPlan {
  int x0, y0, l0, bx, by, bz;
  bool flat;     // z-collapsed plane
  bool two;      // two z-collapsed planes (flat is set too)
  bool box3d;    // the 3-D box fits BOX_NODES / BOX_COLS
};
__device__ __forceinline__ BoxPlan decode_plan(int4 pl) {
  BoxPlan b;
  b.x0 = pl.x;
  b.y0 = pl.y;
  b.flat = pl.w >= 0 && (pl.z & FLAT_BIT);
  b.two = b.flat && (pl.z & FLAT2_BIT);
  b.l0 = pl.z & 0xffff;
  if (b.flat) {
    b.bx = pl.w & 4095;
    b.by = (pl.w >> 12) & 4095;
    b.bz = 4;
  } else {
    b.bx = pl.w & 2047;
    b.by = (pl.w >> 11) & 2047;
    b.bz = (pl.w >> 22) & 511;
  }
  const int sbx = b.bx + ((4 - b.bx) & 7);
  b.box3d = pl.w >= 0 && !b.two && (!b.flat || (sbx * b.by * 4 <= BOX_NODES && sbx * b.by <= BOX_COLS));
  return b;
}

// Level-plane stride of the box (unpadded: padding it to separate z-neighbours' bank groups
// removed only 6 % of the wavefronts and made more chunks miss the tile).
__host__ __device__ __forceinline__ int box_zstride(int sbx, int by) { return by * sbx; }

template <bool P2 = true>
__device__ __forceinline__ int wrap_rel(int i, int ref, int n) {
  // i - ref folded into [-n/2, n/2)
  return wrapi<P2>(i - ref + (n >> 1), n) - (n >> 1);
}

// Two FP32 lanes packed in 64 bits for the Blackwell paired FMA (fma.rn.f32x2).
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  return (unsigned long long)__float_as_uint(a) | ((unsigned long long)__float_as_uint(b) << 32);
}
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long w, unsigned long long v) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(w), "l"(v));
}
__device__ __forceinline__ float lo2(unsigned long long v) { return __uint_as_float(unsigned(v)); }
__device__ __forceinline__ float hi2(unsigned long long v) { return __uint_as_float(unsigned(v >> 32)); }

// One stencil row of four staged nodes summed along x: (u, v) and (w, phi_t) pairs with the
// x weights given as (w, w) pairs, and (second form) the row's eta values with the same weights.
__device__ __forceinline__ void row_sum(const float4* row, const unsigned long long (&wx2)[4],
                                        unsigned long long& ruv, unsigned long long& rwt) {
  ruv = pack2(0.f, 0.f);
  rwt = pack2(0.f, 0.f);
#pragma unroll
  for (int kx = 0; kx < 4; ++kx) {
    const float4 gv = row[kx];
    fma2(ruv, wx2[kx], pack2(gv.x, gv.y));
    fma2(rwt, wx2[kx], pack2(gv.z, gv.w));
  }
}
__device__ __forceinline__ void row_sum(const float4* row, const float* erow,
                                        const unsigned long long (&wx2)[4], const float (&wx)[4],
                                        unsigned long long& ruv, unsigned long long& rwt, float& re) {
  row_sum(row, wx2, ruv, rwt);
  re = 0.f;
#pragma unroll
  for (int kx = 0; kx < 4; ++kx) re = fmaf(wx[kx], erow[kx], re);
}

// Points whose stencils are gathered straight from global memory (L1/L2): one record per point,
// 80 bytes so that the eight records a warp reads at once lie in different banks.
struct alignas(16) GatherRec {
  int4 cell;             // first stencil node in x and y (before the -1 shift), first level, inside
  float4 wy, wz;
  float wx[4];           // the four gathered fields overwrite the x weights
  float eta, pad_[3];
};
static_assert(sizeof(GatherRec) == 80, "GatherRec layout");

// A quad's sum over its four columns (lane k's sums (u, v), (w, dphi/dt), eta times its x weight) into
// the point's record: field k from lane k.
__device__ __forceinline__ void quad_sum(unsigned long long uv, unsigned long long wt, float e, float wxk, int k,
                                         GatherRec& r) {
  const float f0 = wxk * lo2(uv), f1 = wxk * hi2(uv), f2 = wxk * lo2(wt), f3 = wxk * hi2(wt);
  e *= wxk;
  e += __shfl_xor_sync(0xffffffffu, e, 1);
  e += __shfl_xor_sync(0xffffffffu, e, 2);
  // transposing reduction: lanes k and k ^ 1 swap the halves they do not keep, then k and k ^ 2
  const bool odd = k & 1, high = k & 2;
  float g0 = odd ? f1 : f0, g1 = odd ? f3 : f2;
  g0 += __shfl_xor_sync(0xffffffffu, odd ? f0 : f1, 1);
  g1 += __shfl_xor_sync(0xffffffffu, odd ? f2 : f3, 1);
  const float h = (high ? g1 : g0) + __shfl_xor_sync(0xffffffffu, high ? g0 : g1, 2);
  __syncwarp();                                    // every lane of the quad has read the record
  r.wx[k] = h;
  if (k == 0) r.eta = e;
}

// Stencil sums of points p0 .. p0 + WPTS - 1 by one warp, four lanes a point, lane k the stencil's x
// node k. A warp load then covers the 64-byte stencil rows of eight points (8 to 16 L1 lines), where
// one point a lane touches 32 lines with every load: the L1's line rate is what bounds scattered
// points (74 % of its data pipe on the first workload below, 87 % on the second). Each lane sums its
// column over y, z and time; the quad's x sum is a shuffle reduction that leaves field k with lane k.
// 16 M scattered points on the 8.6 GB grid of 2048 x 1024 modes and 128 levels: 5.17 -> 3.28 ms; 8.2 M
// mesh points on the four-fold padded 512 x 256-mode grid: 1.45 -> 1.02 ms (one point a lane before).
template <bool P2, int WPTS>
__device__ __forceinline__ void gather_warp(const InterpArgs& a, const LevelTables& zs, int64_t p0, GatherRec* rec) {
  const size_t plane = size_t(a.Nyr) * a.Nxr;
  const size_t tl_stride = size_t(a.nz) * plane;
  const int lane = threadIdx.x & 31, k = lane & 3;
  const bool two_d = a.Nyr == 1;
  const int64_t i = p0 + lane;
  float z = 0.f;
  if (WPTS == 32 || lane < WPTS) {
    const int64_t ic = i < a.np ? i : a.np - 1;    // lanes past the end repeat the last point
    z = __ldg(&a.pts[3 * ic + 2]);
    const PointCell c = point_cell<P2>(a, zs, __ldg(&a.pts[3 * ic]), __ldg(&a.pts[3 * ic + 1]), z);
    GatherRec& r = rec[lane];
    r.cell = make_int4(c.ix, c.iy, c.j0, c.inside);
    r.wy = make_float4(c.wy[0], c.wy[1], c.wy[2], c.wy[3]);
    r.wz = make_float4(c.wz[0], c.wz[1], c.wz[2], c.wz[3]);
    *reinterpret_cast<float4*>(r.wx) = make_float4(c.wx[0], c.wx[1], c.wx[2], c.wx[3]);
  }
  __syncwarp();
#pragma unroll 1
  for (int s = 0; s < WPTS / 8; ++s) {
    GatherRec& r = rec[8 * s + (lane >> 2)];
    const int4 c = r.cell;
    const float4 wy = r.wy, wz = r.wz;
    const float wxk = r.wx[k];
    const int xk = wrapi<P2>(c.x - 1 + k, a.Nxr);
    int row[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) row[b] = xk + (two_d ? 0 : wrapi<P2>(c.y - 1 + b, a.Nyr) * a.Nxr);
    const float wyb[4] = {wy.x, wy.y, wy.z, wy.w}, wzq[4] = {wz.x, wz.y, wz.z, wz.w};
    unsigned long long uv = 0ull, wt = 0ull;       // (u, v) and (w, dphi/dt)
    float e = 0.f;
    for (int tl = 0; tl < a.n_tl; ++tl) {
      const float wtl = a.wt[tl];
      const float4* base = a.nodes + size_t(tl) * tl_stride + size_t(c.z) * plane;
      const float* et = a.eta + size_t(tl) * plane;
      if (two_d) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 g = __ldg(&base[q * plane + row[0]]);
          const float w = wtl * wzq[q];
          fma2(uv, pack2(w, w), pack2(g.x, g.y));
          fma2(wt, pack2(w, w), pack2(g.z, g.w));
        }
        e = fmaf(wtl, __ldg(&et[row[0]]), e);
        continue;
      }
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        unsigned long long ruv = 0ull, rwt = 0ull;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float4 g = __ldg(&base[q * plane + row[b]]);
          const unsigned long long w2 = pack2(wyb[b], wyb[b]);
          fma2(ruv, w2, pack2(g.x, g.y));
          fma2(rwt, w2, pack2(g.z, g.w));
        }
        const float w = wtl * (q == 0 ? wz.x : q == 1 ? wz.y : q == 2 ? wz.z : wz.w);
        fma2(uv, pack2(w, w), ruv);
        fma2(wt, pack2(w, w), rwt);
      }
      float re = 0.f;
#pragma unroll
      for (int b = 0; b < 4; ++b) re = fmaf(wyb[b], __ldg(&et[row[b]]), re);
      e = fmaf(wtl, re, e);
    }
    quad_sum(uv, wt, e, wxk, k, r);
  }
  __syncwarp();
  if ((WPTS == 32 || lane < WPTS) && i < a.np) {
    const float4 f = *reinterpret_cast<const float4*>(rec[lane].wx);
    store_point(a, i, f, rec[lane].eta, z, rec[lane].cell.w != 0);
  }
  __syncwarp();                                    // the records are rewritten by the next call
}

// Time-blended box of grid nodes x0..x0+bx-1, y0..y0+by-1 (wrapped), levels l0..l0+bz-1 into
// shared memory (row stride sbx, level-plane stride zst float4), and the eta rows (stride sbx).
// Rows (ly, lz) over warps, two rows per warp at a time (more loads in flight), x over lanes;
// the time blend happens here, once per node.
template <bool P2 = true>
__device__ __forceinline__ void stage_box(const InterpArgs& a, int x0, int y0, int l0, int bx, int by,
                                          int bz, int sbx, int zst, float4* sbox, float* seta) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const size_t plane = size_t(a.Nyr) * a.Nxr;
  const size_t tl_stride = size_t(a.nz) * plane;
  const int nrows = by * bz;
  for (int r0 = warp; r0 < nrows; r0 += 2 * nw) {
    const int r1 = min(r0 + nw, nrows - 1);       // a duplicate of r0's last row when past the end
    const int lz0 = r0 / by, ly0 = r0 - lz0 * by, lz1 = r1 / by, ly1 = r1 - lz1 * by;
    const float4* src0 = a.nodes + size_t(l0 + lz0) * plane + size_t(wrapi<P2>(y0 + ly0, a.Nyr)) * a.Nxr;
    const float4* src1 = a.nodes + size_t(l0 + lz1) * plane + size_t(wrapi<P2>(y0 + ly1, a.Nyr)) * a.Nxr;
    for (int lx = lane; lx < bx; lx += 32) {
      const int gx = wrapi<P2>(x0 + lx, a.Nxr);
      float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
      for (int tl = 0; tl < a.n_tl; ++tl) {
        const float4 g0 = __ldg(&src0[size_t(tl) * tl_stride + gx]);
        const float4 g1 = __ldg(&src1[size_t(tl) * tl_stride + gx]);
        const float w = a.wt[tl];
        v0.x = fmaf(w, g0.x, v0.x);
        v0.y = fmaf(w, g0.y, v0.y);
        v0.z = fmaf(w, g0.z, v0.z);
        v0.w = fmaf(w, g0.w, v0.w);
        v1.x = fmaf(w, g1.x, v1.x);
        v1.y = fmaf(w, g1.y, v1.y);
        v1.z = fmaf(w, g1.z, v1.z);
        v1.w = fmaf(w, g1.w, v1.w);
      }
      sbox[lz0 * zst + ly0 * sbx + lx] = v0;
      sbox[lz1 * zst + ly1 * sbx + lx] = v1;       // same value when r1 repeats a row
    }
  }
  for (int ly = warp; ly < by; ly += nw) {
    const float* src = a.eta + size_t(wrapi<P2>(y0 + ly, a.Nyr)) * a.Nxr;
    for (int lx = lane; lx < bx; lx += 32) {
      const int gx = wrapi<P2>(x0 + lx, a.Nxr);
      float v = 0.f;
      for (int tl = 0; tl < a.n_tl; ++tl) v = fmaf(a.wt[tl], __ldg(&src[size_t(tl) * plane + gx]), v);
      seta[ly * sbx + lx] = v;
    }
  }
}

// Level-flat chunk: the z-collapsed, time-blended plane P = sum_t w_t sum_q wz_q G_t[l0 + q] of
// columns x0..x0+bx-1, y0..y0+by-1 (wrapped) into shared memory (row stride sbx), and the eta
// rows. Columns over all threads (index -> (ly, lx)), so every thread has 4 x n_tl node loads
// and n_tl eta loads of one column in flight.
template <bool P2 = true>
__device__ __forceinline__ void stage_plane(const InterpArgs& a, int x0, int y0, int l0, int bx,
                                            int by, int sbx, const float wz[4], float4* splane,
                                            float* seta, bool with_eta = true) {
  const size_t plane = size_t(a.Nyr) * a.Nxr;
  const size_t tl_stride = size_t(a.nz) * plane;
  const int ncol = bx * by;
  for (int c = threadIdx.x; c < ncol; c += blockDim.x) {
    const int ly = c / bx, lx = c - ly * bx;
    const size_t col = size_t(wrapi<P2>(y0 + ly, a.Nyr)) * a.Nxr + wrapi<P2>(x0 + lx, a.Nxr);
    const float4* src = a.nodes + size_t(l0) * plane + col;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    float e = 0.f;
#pragma unroll
    for (int tl = 0; tl < SWENSE_MAX_TL; ++tl) {
      if (tl >= a.n_tl) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 g = __ldg(&src[size_t(tl) * tl_stride + size_t(q) * plane]);
        const float w = a.wt[tl] * wz[q];
        v.x = fmaf(w, g.x, v.x);
        v.y = fmaf(w, g.y, v.y);
        v.z = fmaf(w, g.z, v.z);
        v.w = fmaf(w, g.w, v.w);
      }
      if (with_eta) e = fmaf(a.wt[tl], __ldg(&a.eta[size_t(tl) * plane + col]), e);
    }
    splane[ly * sbx + lx] = v;
    if (with_eta) seta[ly * sbx + lx] = e;
  }
}

// Box plan of one 1024-point chunk: box origin (grid node indices, wrapped) and extents, or
// dims = -1 when the box does not fit the shared-memory tile (the chunk then gathers from
// global memory). Computed by its own kernel so the gather kernel can start its box load at
// once, without first waiting for its points. One warp per chunk (32 points per lane, loads
// coalesced across the lanes): the chunk's reductions stay in the warp, with no block barrier
// and no single-thread tail, and eight chunks of a block share one copy of the level tables.
constexpr int PLAN_WARPS = BOX_THREADS / 32;
__host__ __device__ __forceinline__ int64_t plan_blocks(int64_t np) {
  return ((np + BOX_PTS - 1) / BOX_PTS + PLAN_WARPS - 1) / PLAN_WARPS;
}

// Plan of chunk `chunk` of the points of `a`, by one warp (no block barrier), for tiles of NODES nodes.
template <bool P2, int NODES = BOX_NODES>
__device__ __forceinline__ void plan_chunk(const InterpArgs& a, const LevelTables& zs, int64_t chunk,
                                           int4* __restrict__ plan, int lane) {
  const int64_t p0 = chunk * BOX_PTS;
  if (p0 >= a.np) return;
  // every lane derives the chunk's reference cell (its first point's) itself: broadcast loads
  int refx, refy, refj0;
  const float refz = __ldg(&a.pts[3 * p0 + 2]);
  {
    const PointCell c = point_cell<P2>(a, zs, __ldg(&a.pts[3 * p0]), __ldg(&a.pts[3 * p0 + 1]), refz);
    refx = c.ix;
    refy = c.iy;
    refj0 = c.j0;
  }
  int same_z = 1;                                   // every point of the chunk at z == refz (bitwise)
  int two_z = 1;                                    // every point at refz or at the last point's z
  const float lastz = __ldg(&a.pts[3 * ((p0 + BOX_PTS < a.np ? p0 + BOX_PTS : a.np) - 1) + 2]);
  int mn[3] = {1 << 30, 1 << 30, 1 << 30}, mx[3] = {-(1 << 30), -(1 << 30), -(1 << 30)};
  int first_x = 0, first_y = 0;                     // the lane's point of the chunk's first 32
  // four points per lane per round, their twelve loads issued before any of them is used
  constexpr int PU = 4;
  static_assert((BOX_PTS / 32) % PU == 0, "whole rounds");
#pragma unroll 1
  for (int k0 = 0; k0 < BOX_PTS / 32; k0 += PU) {
    float qx[PU], qy[PU], qz[PU];
#pragma unroll
    for (int u = 0; u < PU; ++u) {
      const int64_t i = p0 + (k0 + u) * 32 + lane;
      const int64_t ic = i < a.np ? i : a.np - 1;     // in-bounds duplicate past the end, unused
      qx[u] = __ldg(&a.pts[3 * ic]);
      qy[u] = __ldg(&a.pts[3 * ic + 1]);
      qz[u] = __ldg(&a.pts[3 * ic + 2]);
    }
#pragma unroll
    for (int u = 0; u < PU; ++u) {
      const int64_t i = p0 + (k0 + u) * 32 + lane;
      if (i < a.np) {
        const float pz = qz[u];
        PointCell c;
        point_xy<P2>(a, qx[u], qy[u], c);
        // the level window only where z differs from the chunk's first point (a layer of an
        // extruded mesh shares one z)
        const bool zeq = __float_as_int(pz) == __float_as_int(refz);
        same_z &= zeq;
        two_z &= zeq || __float_as_int(pz) == __float_as_int(lastz);
        if (zeq) c.j0 = refj0;
        else point_level(a, zs, pz, c);
        const int rx = wrap_rel<P2>(c.ix, refx, a.Nxr);
        const int ry = a.Nyr > 1 ? wrap_rel<P2>(c.iy, refy, a.Nyr) : 0;
        mn[0] = min(mn[0], rx);
        mx[0] = max(mx[0], rx);
        mn[1] = min(mn[1], ry);
        mx[1] = max(mx[1], ry);
        mn[2] = min(mn[2], c.j0);
        mx[2] = max(mx[2], c.j0);
        if (k0 == 0 && u == 0) {
          first_x = rx;
          first_y = ry;
        }
      }
    }
  }
  const int far_x = __reduce_max_sync(0xffffffffu, first_x) - __reduce_min_sync(0xffffffffu, first_x);
  const int far_y = __reduce_max_sync(0xffffffffu, first_y) - __reduce_min_sync(0xffffffffu, first_y);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    for (int o = 16; o > 0; o >>= 1) {
      mn[d] = min(mn[d], __shfl_xor_sync(0xffffffffu, mn[d], o));
      mx[d] = max(mx[d], __shfl_xor_sync(0xffffffffu, mx[d], o));
    }
  }
  const bool flat = __all_sync(0xffffffffu, same_z);
  const bool flat2 = !flat && __all_sync(0xffffffffu, two_z);
  if (lane != 0) return;
  // box: x nodes rel (mn0-1) .. (mx0+2), y likewise (one row in 2-D), levels mn2 .. mx2+3; one that laps
  // the periodic grid is the whole period and three nodes more, so that every stencil is contiguous
  const int bx = min(mx[0] - mn[0] + 4, a.Nxr + 3);
  const int sbx = bx + ((4 - bx) & 7);
  const int by = a.Nyr > 1 ? min(mx[1] - mn[1] + 4, a.Nyr + 3) : 1;
  const int bz = mx[2] - mn[2] + 4;
  const int zst = box_zstride(sbx, by);
  const bool fits = int64_t(zst) * bz <= NODES && int64_t(sbx) * by <= NODES / 4 && bx < 2048 && by < 2048;
  const bool fits_flat = flat && int64_t(sbx) * by <= FLAT_COLS;
  const bool fits_two = flat2 && int64_t(sbx) * by <= FLAT2_COLS;
  const int rows = 2 * bx >= a.Nxr && far_x > ROWS_RATIO * far_y ? ROWS_BIT : 0;
  const int x0 = wrapi<P2>(refx + mn[0] - 1, a.Nxr);
  const int y0 = a.Nyr > 1 ? wrapi<P2>(refy + mn[1] - 1, a.Nyr) : 0;
  plan[chunk] = fits_flat  ? make_int4(x0, y0, mn[2] | FLAT_BIT, bx | (by << 12))
              : fits_two   ? make_int4(x0, y0, FLAT_BIT | FLAT2_BIT, bx | (by << 12))
              : fits       ? make_int4(x0, y0, mn[2], bx | (by << 11) | (bz << 22))
              : flat || flat2
                  ? make_int4(x0, y0, rows | (flat ? FLAT_BIT : FLAT_BIT | FLAT2_BIT), int(0x80000000u | unsigned(bx) | unsigned(by) << 14))
                  : make_int4(x0, y0, rows | mn[2], -1);
}

template <bool P2>
__global__ void __launch_bounds__(BOX_THREADS) k_interp_plan(const __grid_constant__ InterpArgs a, const __grid_constant__ Levels L, int4* __restrict__ plan) {
  __shared__ LevelTables zs;
  fill_level_tables(zs, L);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  plan_chunk<P2>(a, zs, int64_t(blockIdx.x) * PLAN_WARPS + warp, plan, lane);
}

// True when a chunk's plan stages no tile (or is a plan made for another level list): its points
// gather their stencils from global memory.
__device__ __forceinline__ bool plan_is_global(const int4 pl, int nz) {
  if (pl.w < 0) return true;
  const BoxPlan bp = decode_plan(pl);
  return bp.l0 + bp.bz > nz;
}

// Chunks for k_interp_lanes, where that runs.
__device__ __forceinline__ bool plan_is_lanes(const int4 pl, int nz) { return plan_is_global(pl, nz) && pl.w < 0 && (pl.z & ROWS_BIT); }

// The chunk's points gathered from global memory, 32 at a time by each warp; rec: 32 records per warp.
static_assert(BOX_THREADS * sizeof(GatherRec) <= BOX_SMEM, "the records fit the tile's shared memory");
template <bool P2>
__device__ __forceinline__ void global_points(const InterpArgs& a, const LevelTables& zs, int64_t p0,
                                              GatherRec* rec) {
#pragma unroll 1
  for (int k = 0; k < BOX_PPT; ++k) {
    const int64_t i0 = p0 + k * BOX_THREADS + (threadIdx.x & ~31);
    if (i0 >= a.np) break;                         // uniform over the warp
    gather_warp<P2, 32>(a, zs, i0, rec + (threadIdx.x & ~31));
  }
}

// Gather of chunk `chunk` of the points of `a` with its plan `pl`, by the whole CTA; the level
// tables zs are complete after the first barrier inside. kGlobal: also the chunks without a
// staged tile (else those are left to k_interp_global).
template <bool P2, bool kGlobal = true>
__device__ __forceinline__ void box_chunk(const InterpArgs& a, const LevelTables& zs, int64_t chunk,
                                          const int4 pl, float4* sbox, float* seta) {
  const int64_t p0 = chunk * BOX_PTS;
  // the first point's coordinates are in flight during the box load; each later point's while
  // the previous one is processed
  float nx_ = 0.f, ny_ = 0.f, nz_ = 0.f;
  {
    const int64_t i = p0 + threadIdx.x;
    if (i < a.np) {
      nx_ = __ldg(&a.pts[3 * i]);
      ny_ = __ldg(&a.pts[3 * i + 1]);
      nz_ = __ldg(&a.pts[3 * i + 2]);
    }
  }
  const BoxPlan bp = decode_plan(pl);
  if (plan_is_global(pl, a.nz)) {                  // no tile, or a plan of another level list
    __syncthreads();
    if (kGlobal) global_points<P2>(a, zs, p0, reinterpret_cast<GatherRec*>(sbox));
    return;
  }
  const int bx = bp.bx, by = bp.by, bz = bp.bz;
  // shared-memory row stride = 4 (mod 8) float4: reads of neighbouring cells (dx, dy in {0, 1})
  // by one quarter-warp fall into different bank groups
  const int sbx = bx + ((4 - bx) & 7);
  const int x0 = bp.x0, y0 = bp.y0, l0 = bp.l0;
  const int nys = a.Nyr > 1 ? 4 : 1;
  if (bp.flat) {
    // one z (or two: a chunk across two layers) for the whole chunk: level weights once per z
    // (from the level tables, so after the barrier that completes them), the z-collapsed
    // plane(s) and the eta plane, then a 2-D gather of 16 float4 per point
    const bool two = bp.two;
    const float zc = __ldg(&a.pts[3 * p0 + 2]);
    const float zc2 = two ? __ldg(&a.pts[3 * ((p0 + BOX_PTS < a.np ? p0 + BOX_PTS : a.np) - 1) + 2]) : zc;
    __syncthreads();
    PointCell cz, cz2;
    point_level(a, zs, zc, cz);
    if (two) point_level(a, zs, zc2, cz2);
    else cz2 = cz;
    float4* planeB = two ? sbox + FLAT2_COLS : sbox;
    float* fe = reinterpret_cast<float*>(sbox + (two ? 2 * FLAT2_COLS : FLAT_COLS));
    stage_plane<P2>(a, x0, y0, cz.j0, bx, by, sbx, cz.wz, sbox, fe);
    if (two) stage_plane<P2>(a, x0, y0, cz2.j0, bx, by, sbx, cz2.wz, planeB, fe, false);
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k < BOX_PPT; ++k) {
      const int64_t i = p0 + k * BOX_THREADS + threadIdx.x;
      if (i >= a.np) break;
      const float px = nx_, py = ny_, pz = nz_;
      if (k + 1 < BOX_PPT && i + BOX_THREADS < a.np) {
        nx_ = __ldg(&a.pts[3 * (i + BOX_THREADS)]);
        ny_ = __ldg(&a.pts[3 * (i + BOX_THREADS) + 1]);
        if (two) nz_ = __ldg(&a.pts[3 * (i + BOX_THREADS) + 2]);
      }
      const bool onA = !two || __float_as_int(pz) == __float_as_int(zc);
      PointCell c;
      point_xy<P2>(a, px, py, c);
      const int lx = min(max(wrapi<P2>(c.ix - 1 - x0, a.Nxr), 0), bx - 4);
      const int ly = a.Nyr > 1 ? min(max(wrapi<P2>(c.iy - 1 - y0, a.Nyr), 0), by - 4) : 0;
      const float4* base = (onA ? sbox : planeB) + ly * sbx + lx;
      const float* ebase = fe + ly * sbx + lx;
      // separable tensor product: each stencil row summed along x with the paired x weights,
      // then the rows combined with the y weights
      unsigned long long wx2[4];
#pragma unroll
      for (int kx = 0; kx < 4; ++kx) wx2[kx] = pack2(c.wx[kx], c.wx[kx]);
      unsigned long long uv = pack2(0.f, 0.f), wt = pack2(0.f, 0.f);
      float acc_eta = 0.f;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if (b >= nys) break;
        unsigned long long ruv, rwt;
        float re;
        row_sum(base + b * sbx, ebase + b * sbx, wx2, c.wx, ruv, rwt, re);
        const unsigned long long wy2 = pack2(c.wy[b], c.wy[b]);
        fma2(uv, wy2, ruv);
        fma2(wt, wy2, rwt);
        acc_eta = fmaf(c.wy[b], re, acc_eta);
      }
      store_point(a, i, make_float4(lo2(uv), hi2(uv), lo2(wt), hi2(wt)), acc_eta, pz,
                  onA ? cz.inside : cz2.inside);
    }
    return;
  }
  const int zst = box_zstride(sbx, by);
  stage_box<P2>(a, x0, y0, l0, bx, by, bz, sbx, zst, sbox, seta);
  __syncthreads();
  const int zstride = zst;
#pragma unroll 1
  for (int k = 0; k < BOX_PPT; ++k) {
    const int64_t i = p0 + k * BOX_THREADS + threadIdx.x;
    if (i >= a.np) break;                          // later points of this thread are past np too
    const float px = nx_, py = ny_, pz = nz_;
    if (k + 1 < BOX_PPT && i + BOX_THREADS < a.np) {
      nx_ = __ldg(&a.pts[3 * (i + BOX_THREADS)]);
      ny_ = __ldg(&a.pts[3 * (i + BOX_THREADS) + 1]);
      nz_ = __ldg(&a.pts[3 * (i + BOX_THREADS) + 2]);
    }
    const PointCell c = point_cell<P2>(a, zs, px, py, pz);
    // node offsets inside the box; the plan kernel bounded them with the same point_cell, and
    // the clamps keep every shared-memory read inside the box regardless
    const int lx = min(max(wrapi<P2>(c.ix - 1 - x0, a.Nxr), 0), bx - 4);
    const int ly = a.Nyr > 1 ? min(max(wrapi<P2>(c.iy - 1 - y0, a.Nyr), 0), by - 4) : 0;
    const int lz = min(max(c.j0 - l0, 0), bz - 4);
    const float4* base = sbox + lz * zst + ly * sbx + lx;
    // separable tensor product: rows along x, then y within each level, then the levels in z
    unsigned long long wx2[4];
#pragma unroll
    for (int kx = 0; kx < 4; ++kx) wx2[kx] = pack2(c.wx[kx], c.wx[kx]);
    unsigned long long uv = pack2(0.f, 0.f), wt = pack2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      unsigned long long quv = pack2(0.f, 0.f), qwt = pack2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if (b >= nys) break;
        unsigned long long ruv, rwt;
        row_sum(base + q * zstride + b * sbx, wx2, ruv, rwt);
        const unsigned long long wy2 = pack2(c.wy[b], c.wy[b]);
        fma2(quv, wy2, ruv);
        fma2(qwt, wy2, rwt);
      }
      const unsigned long long wz2 = pack2(c.wz[q], c.wz[q]);
      fma2(uv, wz2, quv);
      fma2(wt, wz2, qwt);
    }
    float acc_eta = 0.f;
    const float* ebase = seta + ly * sbx + lx;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if (b >= nys) break;
      float re = 0.f;
#pragma unroll
      for (int kx = 0; kx < 4; ++kx) re = fmaf(c.wx[kx], ebase[b * sbx + kx], re);
      acc_eta = fmaf(c.wy[b], re, acc_eta);
    }
    store_point(a, i, make_float4(lo2(uv), hi2(uv), lo2(wt), hi2(wt)), acc_eta, pz, c.inside);
  }
}

// The chunks with a staged tile (box, plane or two planes); kSplit: k_interp_global takes the
// others, else this kernel gathers them too (from global memory, with L1 reduced by the tile).
template <bool P2, bool kSplit>
__global__ void __launch_bounds__(BOX_THREADS, 3) k_interp_box(const __grid_constant__ InterpArgs a, const __grid_constant__ Levels L,
                                                                const int4* __restrict__ plan) {
  extern __shared__ float4 sbox[];
  float* seta = reinterpret_cast<float*>(sbox + BOX_NODES);
  __shared__ LevelTables zs;
  const int4 pl = plan[blockIdx.x];
  if (kSplit && plan_is_global(pl, a.nz)) return;   // uniform over the CTA
  fill_level_tables(zs, L);
  box_chunk<P2, !kSplit>(a, zs, blockIdx.x, pl, sbox, seta);
}

// The chunks without a staged tile (scattered points: the stencils of a 1024-point chunk span
// more nodes than shared memory holds). No dynamic shared memory, so that L1 keeps the rows
// neighbouring points share: launched apart from k_interp_box, whose 68 KB tile per CTA would
// leave L1 a fifth of its size.
// A warp per GLOBAL_WPTS points, CTAs in point order and without a block barrier: with 16 points a
// warp the points in flight span half the grid that 32 would (their shared rows stay in L2 until both
// have read them: 3.5 -> 3.3 ms on the scattered points above), with 8 the idle lanes of the cell
// search cost more than that gives (3.4 ms). Four loads in flight a lane (a rolled level loop, 48
// registers, five CTAs per SM): more of them evict each other's lines from L1 (5.8 ms with sixteen).
constexpr int GLOBAL_WPTS = 16;
constexpr int GLOBAL_PTS = GLOBAL_WPTS * (BOX_THREADS / 32);     // points per CTA
template <bool P2, bool LANES = false>
__global__ void __launch_bounds__(BOX_THREADS, 5) k_interp_global(const __grid_constant__ InterpArgs a,
                                                                       const __grid_constant__ Levels L,
                                                                       const int4* __restrict__ plan,
                                                                       const int* __restrict__ n_global,
                                                                       const int2* __restrict__ chunk_slot, int rounds) {
  __shared__ GatherRec rec[GLOBAL_PTS];
  const int warp = threadIdx.x >> 5;
  int64_t p0 = int64_t(blockIdx.x) * rounds * GLOBAL_PTS + warp * GLOBAL_WPTS;
  // uniform over the warp; no plan: every point is gathered here. n_global, chunk_slot: of the gather
  // by kinds (NULL otherwise), whose other kernels took the chunks with a plane
  if (n_global && *n_global == 0) return;
  if (p0 >= a.np || (plan && !plan_is_global(plan[p0 / BOX_PTS], a.nz))) return;
  if (LANES && plan_is_lanes(plan[p0 / BOX_PTS], a.nz)) return;   // k_interp_lanes takes those
  if (chunk_slot && chunk_slot[p0 / BOX_PTS].x >= 0) return;
#pragma unroll 1
  for (int r = 0; r < rounds && p0 < a.np; ++r, p0 += GLOBAL_PTS)   // within one chunk
    gather_warp<P2, GLOBAL_WPTS>(a, *level_tables(L), p0, rec + warp * GLOBAL_WPTS);
}

// Untiled chunks whose points follow the grid's rows, on grids whose four levels of all time levels exceed
// L2: a point a lane. Nothing is met again in L1 or L2 there, so DRAM bounds them, and a lane's load asks
// for one sector where a quad's asks for the two or three of a stencil row, which L2 fetches in pairs: 77
// instead of 112 bytes a row (2 M binned points on the four-fold padded 512 x 256 grid: 2.46 against 3.57
// GB of DRAM reads, 440 against 541 us a time level). Points in no order pay for a lane's 32 pages a load
// (1.74 ms by quads, 3.27 by lanes, the same grid), points close by in all directions meet in L1 (16 M in
// Morton order on the large sea: 2.9 against 5.2 ms), and on grids that fit L2 quads win too.
template <bool P2>
__device__ __forceinline__ void lane_point(const InterpArgs& a, const LevelTables& T, int64_t i) {
  const float z = __ldg(&a.pts[3 * i + 2]);
  const PointCell c = point_cell<P2>(a, T, __ldg(&a.pts[3 * i]), __ldg(&a.pts[3 * i + 1]), z);
  const size_t plane = size_t(a.Nyr) * a.Nxr;
  int xi[4], yo[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    xi[q] = wrapi<P2>(c.ix - 1 + q, a.Nxr);
    yo[q] = wrapi<P2>(c.iy - 1 + q, a.Nyr) * a.Nxr;
  }
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float e = 0.f;
  for (int tl = 0; tl < a.n_tl; ++tl) {
    const float wtl = a.wt[tl];
    const float4* base = a.nodes + (size_t(tl) * a.nz + c.j0) * plane;
    const float* et = a.eta + size_t(tl) * plane;
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
      const float wq = wtl * (q == 0 ? c.wz[0] : q == 1 ? c.wz[1] : q == 2 ? c.wz[2] : c.wz[3]);
#pragma unroll 1
      for (int b = 0; b < 4; ++b) {                // a select, so that the weights stay in registers
        const float wqy = wq * (b == 0 ? c.wy[0] : b == 1 ? c.wy[1] : b == 2 ? c.wy[2] : c.wy[3]);
        const float4* row = base + size_t(q) * plane + (b == 0 ? yo[0] : b == 1 ? yo[1] : b == 2 ? yo[2] : yo[3]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 g = __ldg(&row[xi[k]]);
          const float w = wqy * c.wx[k];
          acc.x = fmaf(w, g.x, acc.x);
          acc.y = fmaf(w, g.y, acc.y);
          acc.z = fmaf(w, g.z, acc.z);
          acc.w = fmaf(w, g.w, acc.w);
        }
      }
    }
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
      const float wy = wtl * (b == 0 ? c.wy[0] : b == 1 ? c.wy[1] : b == 2 ? c.wy[2] : c.wy[3]);
      const float* row = et + (b == 0 ? yo[0] : b == 1 ? yo[1] : b == 2 ? yo[2] : yo[3]);
#pragma unroll
      for (int k = 0; k < 4; ++k) e = fmaf(wy * c.wx[k], __ldg(&row[xi[k]]), e);
    }
  }
  store_point(a, i, acc, e, z, c.inside);
}

// A quarter of a chunk a block, in point order: what the points in flight read then spans few enough of them that
// the next level's, one slab of tiles or layer on, still find it in L2 (the 2 M points above 0.95 ms; whole
// chunks a block 1.48, quarters by persistent blocks in turn 1.09). list: the gather by kinds, its chunks by
// ticket, so that an empty list costs a launch; else every chunk, by its plan.
constexpr int LANE_PARTS = BOX_PTS / BOX_THREADS;
// Fewer chunks than one wave of blocks (a few whose box happens to span the grid, of points in Morton order) take
// one chain of loads, 32 us, however few they are.
constexpr int LANE_FEW = 152;
template <bool P2>
__global__ void __launch_bounds__(BOX_THREADS, 4) k_interp_lanes(const __grid_constant__ InterpArgs a,
                                                                  const __grid_constant__ Levels L,
                                                                  const int4* __restrict__ plan,
                                                                  const int* __restrict__ list,
                                                                  const int* __restrict__ n_list, unsigned* ticket) {
  if (!list) {
    const int64_t chunk = blockIdx.x / LANE_PARTS, i = int64_t(blockIdx.x) * BOX_THREADS + threadIdx.x;
    if (plan_is_lanes(plan[chunk], a.nz) && i < a.np) lane_point<P2>(a, *level_tables(L), i);
    return;
  }
  __shared__ unsigned s_item;
  const unsigned n = unsigned(*n_list) * LANE_PARTS;
  if (n == 0) return;
  for (;;) {
    __syncthreads();                               // the item before has been read
    if (threadIdx.x == 0) s_item = atomicAdd(ticket, 1u);
    __syncthreads();
    const unsigned item = s_item;
    if (item >= n) return;                         // uniform over the block
    const int64_t i = int64_t(list[item / LANE_PARTS]) * BOX_PTS + (item % LANE_PARTS) * BOX_THREADS + threadIdx.x;
    if (i < a.np) lane_point<P2>(a, *level_tables(L), i);
  }
}

// ---------------------------------------------------------------------------------------------
// Gather of many points on a grid much finer than they are (LAYER_POINTS and more; the rule of `split`):
// the layers of an extruded mesh put many chunks at one z, and their stencil boxes are too wide for a
// tile. All chunks of a z share one z-collapsed, time-blended plane of the columns that their stencils
// cover, made once in scratch memory (k_plane_collapse), and a point then reads 16 of its nodes where
// the grid itself would be 64 n_tl. k_gather_register enters each such chunk's z and box in a hash
// table; k_gather_lists sizes the planes (those that pay, within the scratch given), groups them by
// their levels and lists the chunks that read planes and those with a staged tile, for persistent
// kernels, so that an empty list costs a launch; k_interp_global takes the rest in point order.
// 8.2 M mesh points on the four-fold padded 512 x 256 grid: 1.02 ms straight from the grid, 0.46 ms so (planes 0.13, gather 0.22 of it);
// from 2^21 points on, where the lists' fixed cost pays (2 M mesh points: 178 against 235 us there with one time level,
// 288 and 300 with two; 4 M: 512 against 428 with two).
// 3-D grids only: a 2-D one has too few nodes for the rule.
constexpr int64_t LAYER_POINTS = int64_t(1) << 21;
constexpr int PLANE_SLOTS = 4096;                  // planes at most (hash table entries)
constexpr int PLANE_UNIT = BOX_THREADS;            // a plane's columns are padded to whole units
constexpr unsigned PLANE_BIAS = 0x40000000u;
struct PlaneSlot {
  unsigned key;          // ~(bits of z); 0: free (NaN is never entered)
  unsigned cnt;          // points
  unsigned x0, x1, y0, y1;   // box relative to chunk 0's: BIAS - first, BIAS + one past the last (maxima)
  int off;               // first column of the plane, -1: none
  int pad_;
};
struct GatherCounts {
  unsigned long long oor;
  int groups, units, n_plane, n_tile, n_global, n_lanes;
  unsigned lane_ticket;
};
static_assert(sizeof(GatherCounts) <= 256, "the counters' part of the workspace");
// Planes whose z has the same four levels and whose boxes lie close (their union no larger than their
// sum) are made together: a column's nodes are loaded once for all. Others form groups of one.
struct PlaneGroup {
  int unit0, first, n, pad_;     // first unit of the group's box; its planes in `members`
  int rx, ry, bx, by;            // union of their boxes
};
struct GatherLists {
  GatherCounts* n;
  PlaneSlot* slots;      // [PLANE_SLOTS]
  PlaneGroup* groups;    // [PLANE_SLOTS]
  int* members;          // [PLANE_SLOTS] slots, group by group
  int2* chunk_slot;      // [chunks] slots of the chunk's first and last z, x = -1: not from planes
  // [chunks] chunks from planes, and of the others those with a staged tile and those for k_interp_lanes
  int *l_plane, *l_tile, *l_lanes;
  int lanes;             // whether that runs
  float4* cols;          // [max_units * PLANE_UNIT]
  float* etas;
  int max_units;
};

__device__ __forceinline__ int plane_enter(PlaneSlot* slots, float z, int cnt, int rx, int bx, int ry, int by) {
  const unsigned key = ~__float_as_uint(z);
  if (z != z) return -1;
  unsigned h = (key * 2654435761u) >> 20;          // 12 bits
  for (int probe = 0; probe < 32; ++probe, h = (h + 1) & (PLANE_SLOTS - 1)) {
    const unsigned old = atomicCAS(&slots[h].key, 0u, key);
    if (old != 0u && old != key) continue;
    atomicAdd(&slots[h].cnt, unsigned(cnt));
    atomicMax(&slots[h].x0, PLANE_BIAS - unsigned(rx));
    atomicMax(&slots[h].x1, PLANE_BIAS + unsigned(rx + bx));
    atomicMax(&slots[h].y0, PLANE_BIAS - unsigned(ry));
    atomicMax(&slots[h].y1, PLANE_BIAS + unsigned(ry + by));
    return int(h);
  }
  return -1;
}

template <bool P2>
__global__ void __launch_bounds__(256) k_gather_register(const __grid_constant__ InterpArgs a,
                                                         const int4* __restrict__ plan, int chunks, GatherLists g) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= chunks) return;
  const int4 pl = plan[c];
  int2 sl = make_int2(-1, -1);
  const int bx = pl.w >= 0 ? pl.w & 4095 : pl.w & 16383, by = pl.w >= 0 ? (pl.w >> 12) & 4095 : (pl.w >> 14) & 16383;
  // (a plan of another grid may hold boxes that no stencil of this one fits)
  if (pl.w != -1 && (pl.z & FLAT_BIT) && bx >= 4 && by >= 4) {
    const int rx = wrap_rel<P2>(pl.x, plan[0].x, a.Nxr), ry = wrap_rel<P2>(pl.y, plan[0].y, a.Nyr);
    const int64_t p0 = int64_t(c) * BOX_PTS, p1 = p0 + BOX_PTS < a.np ? p0 + BOX_PTS : a.np;
    const int n = int(p1 - p0);
    const bool two = pl.z & FLAT2_BIT;
    sl.x = plane_enter(g.slots, __ldg(&a.pts[3 * p0 + 2]), two ? n / 2 : n, rx, bx, ry, by);
    sl.y = two ? plane_enter(g.slots, __ldg(&a.pts[3 * (p1 - 1) + 2]), n / 2, rx, bx, ry, by) : sl.x;
  }
  g.chunk_slot[c] = sl;
}

// Extents of a plane's box; none when it laps the periodic grid.
__device__ __forceinline__ bool plane_box(const InterpArgs& a, const PlaneSlot& s, int& rx, int& ry, int& bx, int& by) {
  rx = -int(s.x0 - PLANE_BIAS);
  ry = -int(s.y0 - PLANE_BIAS);
  bx = int(s.x1 - PLANE_BIAS) - rx;
  by = int(s.y1 - PLANE_BIAS) - ry;
  return bx <= a.Nxr && by <= a.Nyr;
}

// Exclusive prefix sum of v over the block of 1024 threads; total returned in `sum`.
__device__ __forceinline__ long long block_scan(long long v, long long* warp_sums, long long& sum) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();                                 // the previous scan's sums have been read
  if (lane == 31) warp_sums[w] = x;
  __syncthreads();
  if (w == 0) {
    long long y = warp_sums[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long q = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += q;
    }
    warp_sums[lane] = y;
  }
  __syncthreads();
  sum = warp_sums[31];
  return x - v + (w ? warp_sums[w - 1] : 0);
}

// One block. A plane pays when its columns (4 n_tl coalesced loads, shared within its group) are at most
// four times its points (each 16 loads instead of 64 n_tl).
__global__ void __launch_bounds__(1024) k_gather_lists(const __grid_constant__ InterpArgs a,
                                                       const __grid_constant__ Levels L,
                                                       const int4* __restrict__ plan, int chunks, GatherLists g) {
  __shared__ long long ws[32];
  __shared__ int gcnt[SWENSE_MAX_LEVELS], gx0[SWENSE_MAX_LEVELS], gx1[SWENSE_MAX_LEVELS], gy0[SWENSE_MAX_LEVELS],
      gy1[SWENSE_MAX_LEVELS], gsum[SWENSE_MAX_LEVELS], gpos[SWENSE_MAX_LEVELS];
  constexpr int PER = PLANE_SLOTS / 1024;
  long long mine[PER], units = 0, sum;
  int lev[PER];
  if (threadIdx.x < SWENSE_MAX_LEVELS) {
    gcnt[threadIdx.x] = gsum[threadIdx.x] = 0;
    gx0[threadIdx.x] = gy0[threadIdx.x] = 1 << 30;
    gx1[threadIdx.x] = gy1[threadIdx.x] = -(1 << 30);
  }
  for (int k = 0; k < PER; ++k) {
    const PlaneSlot s = g.slots[threadIdx.x * PER + k];
    int rx, ry, bx, by;
    mine[k] = 0;
    if (s.key && plane_box(a, s, rx, ry, bx, by)) {
      const long long cols = (long long)bx * by;
      if (cols <= 4ll * s.cnt) mine[k] = (cols + PLANE_UNIT - 1) / PLANE_UNIT;
    }
    units += mine[k];
  }
  long long u = block_scan(units, ws, sum);        // (its barriers also order the group tables above)
  for (int k = 0; k < PER; ++k) {                  // planes that pass the scratch's end are left out
    if (u + mine[k] > g.max_units) mine[k] = 0;
    const int i = threadIdx.x * PER + k;
    g.slots[i].off = mine[k] ? int(u) * PLANE_UNIT : -1;
    u += mine[k];
    if (!mine[k]) continue;
    const PlaneSlot s = g.slots[i];
    int rx, ry, bx, by;
    plane_box(a, s, rx, ry, bx, by);
    PointCell pc;
    point_level(a, *level_tables(L), __uint_as_float(~s.key), pc);
    lev[k] = pc.j0;
    atomicAdd(&gcnt[pc.j0], 1);
    atomicAdd(&gsum[pc.j0], int(mine[k]));
    atomicMin(&gx0[pc.j0], rx);
    atomicMin(&gy0[pc.j0], ry);
    atomicMax(&gx1[pc.j0], rx + bx);
    atomicMax(&gy1[pc.j0], ry + by);
  }
  __syncthreads();
  // joint groups, a thread per first level; then the planes of the other levels, each on its own
  const int t = threadIdx.x;
  int cnt = t < SWENSE_MAX_LEVELS ? gcnt[t] : 0;
  const int gbx = cnt ? gx1[t] - gx0[t] : 0, gby = cnt ? gy1[t] - gy0[t] : 0;
  long long gu = ((long long)gbx * gby + PLANE_UNIT - 1) / PLANE_UNIT;
  if (cnt && gu > gsum[t]) {
    cnt = 0;
    gu = 0;
    gpos[t] = -1;                                  // not joint
  }
  const int first = int(block_scan(cnt, ws, sum)), joint = int(sum);
  const int id = int(block_scan(cnt ? 1 : 0, ws, sum));
  int groups = int(sum);
  const int u0 = int(block_scan(gu, ws, sum));
  int gunits = int(sum);
  if (cnt) {
    g.groups[id] = PlaneGroup{u0, first, cnt, 0, gx0[t], gy0[t], gbx, gby};
    gpos[t] = first;
  }
  __syncthreads();
  int alone = 0;
  long long aunits = 0;
  for (int k = 0; k < PER; ++k) {
    if (!mine[k]) continue;
    if (gpos[lev[k]] >= 0) {
      g.members[atomicAdd(&gpos[lev[k]], 1)] = t * PER + k;
    } else {
      ++alone;
      aunits += mine[k];
    }
  }
  int ai = int(block_scan(alone, ws, sum));
  const int n_alone = int(sum);
  int au = gunits + int(block_scan(aunits, ws, sum));
  gunits += int(sum);
  for (int k = 0; k < PER; ++k) {
    if (!mine[k] || gpos[lev[k]] >= 0) continue;
    const int i = t * PER + k;
    const PlaneSlot s = g.slots[i];
    int rx, ry, bx, by;
    plane_box(a, s, rx, ry, bx, by);
    g.members[joint + ai] = i;
    g.groups[groups + ai] = PlaneGroup{au, joint + ai, 1, 0, rx, ry, bx, by};
    au += int(mine[k]);
    ++ai;
  }
  groups += n_alone;
  __threadfence_block();
  __syncthreads();
  int np = 0, nt = 0, ng = 0, nl = 0;
  for (int c0 = 0; c0 < chunks; c0 += 1024) {
    const int c = c0 + t;
    int kind = -1;
    if (c < chunks) {
      const int2 sl = g.chunk_slot[c];
      kind = sl.x >= 0 && sl.y >= 0 && g.slots[sl.x].off >= 0 && g.slots[sl.y].off >= 0 ? 0
             : !plan_is_global(plan[c], a.nz)                                           ? 1
             : g.lanes && plan_is_lanes(plan[c], a.nz)                                  ? 3
                                                                                        : 2;
      // (x >= 0: not for k_interp_global)
      if (kind != 0) g.chunk_slot[c] = make_int2(kind == 3 ? 0 : -1, -1);
    }
    const long long pre = block_scan(kind < 0 ? 0 : 1ll << (16 * kind), ws, sum);
    if (kind == 0) g.l_plane[np + int(pre & 0xffff)] = c;
    if (kind == 1) g.l_tile[nt + int(pre >> 16 & 0xffff)] = c;
    if (kind == 3) g.l_lanes[nl + int(pre >> 48 & 0xffff)] = c;
    np += int(sum & 0xffff);
    nt += int(sum >> 16 & 0xffff);
    ng += int(sum >> 32 & 0xffff);
    nl += int(sum >> 48 & 0xffff);
  }
  if (nl < LANE_FEW) {                             // not worth a launch's wait: left to k_interp_global
    __threadfence_block();
    __syncthreads();
    for (int i = t; i < nl; i += 1024) g.chunk_slot[g.l_lanes[i]] = make_int2(-1, -1);
    ng += nl;
    nl = 0;
  }
  if (t == 0) {
    g.n->groups = groups;
    g.n->units = gunits;
    g.n->n_plane = np;
    g.n->n_tile = nt;
    g.n->n_global = ng;
    g.n->n_lanes = nl;
    g.n->lane_ticket = 0;
  }
}

// The planes: a thread per column of a group's box, its four levels blended in time once, then a
// weighted sum and a store for each of the group's planes that holds the column.
template <bool P2>
__global__ void __launch_bounds__(BOX_THREADS, 4) k_plane_collapse(const __grid_constant__ InterpArgs a,
                                                                    const __grid_constant__ Levels L,
                                                                    const int4* __restrict__ plan, GatherLists g) {
  const int groups = g.n->groups, units = groups ? g.n->units : 0;
  if (units == 0) return;
  const int4 ref = plan[0];
  const size_t plane = size_t(a.Nyr) * a.Nxr, tl_stride = size_t(a.nz) * plane;
  const LevelTables& T = *level_tables(L);
  constexpr int BATCH = 64;                        // planes whose weights and boxes are in shared memory
  __shared__ float4 swz[BATCH];
  __shared__ int4 sbx[BATCH];                      // rx, ry, bx, by
  __shared__ int soff[BATCH];
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    int lo = 0, hi = groups - 1;                   // last group whose first unit <= u
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (g.groups[mid].unit0 <= u) lo = mid;
      else hi = mid - 1;
    }
    const PlaneGroup e = g.groups[lo];
    // threads past the box's end repeat its last column and store nothing
    const int ci = (u - e.unit0) * PLANE_UNIT + int(threadIdx.x), c = min(ci, e.bx * e.by - 1);
    const int cy = e.ry + c / e.bx, cx = e.rx + c % e.bx;     // relative to chunk 0's box
    const size_t col = size_t(wrapi<P2>(ref.y + cy, a.Nyr)) * a.Nxr + wrapi<P2>(ref.x + cx, a.Nxr);
    PointCell pc;
    point_level(a, T, __uint_as_float(~g.slots[g.members[e.first]].key), pc);
    const float4* src = a.nodes + size_t(pc.j0) * plane + col;
    float4 v[4];
    float et = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int tl = 0; tl < a.n_tl; ++tl) {
      const float w = a.wt[tl];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 n = __ldg(&src[size_t(tl) * tl_stride + size_t(q) * plane]);
        v[q].x = fmaf(w, n.x, v[q].x);
        v[q].y = fmaf(w, n.y, v[q].y);
        v[q].z = fmaf(w, n.z, v[q].z);
        v[q].w = fmaf(w, n.w, v[q].w);
      }
      et = fmaf(w, __ldg(&a.eta[size_t(tl) * plane + col]), et);
    }
    for (int k0 = 0; k0 < e.n; k0 += BATCH) {
      const int nk = min(BATCH, e.n - k0);
      __syncthreads();                             // the previous batch has been read
      if (threadIdx.x < nk) {
        const PlaneSlot& s = g.slots[g.members[e.first + k0 + threadIdx.x]];
        int rx, ry, bx, by;
        plane_box(a, s, rx, ry, bx, by);
        point_level(a, T, __uint_as_float(~s.key), pc);
        swz[threadIdx.x] = make_float4(pc.wz[0], pc.wz[1], pc.wz[2], pc.wz[3]);
        sbx[threadIdx.x] = make_int4(rx, ry, bx, by);
        soff[threadIdx.x] = s.off;
      }
      __syncthreads();
      for (int k = 0; k < nk; ++k) {
        const int4 b = sbx[k];
        const int lx = cx - b.x, ly = cy - b.y;
        if (ci != c || lx < 0 || lx >= b.z || ly < 0 || ly >= b.w) continue;
        const float4 w = swz[k];
        float4 o = make_float4(w.x * v[0].x, w.x * v[0].y, w.x * v[0].z, w.x * v[0].w);
        const float wq[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int q = 1; q < 4; ++q) {
          o.x = fmaf(wq[q], v[q].x, o.x);
          o.y = fmaf(wq[q], v[q].y, o.y);
          o.z = fmaf(wq[q], v[q].z, o.z);
          o.w = fmaf(wq[q], v[q].w, o.w);
        }
        const int i = soff[k] + ly * b.z + lx;
        g.cols[i] = o;
        g.etas[i] = et;
      }
    }
  }
}

// WPTS points from their planes by one warp, four lanes a point (as gather_warp).
template <bool P2, int WPTS>
__device__ __forceinline__ void plane_warp(const InterpArgs& a, const Levels& L, const GatherLists& g, int4 ref, int2 sl,
                                           int64_t p0, GatherRec* rec) {
  const int lane = threadIdx.x & 31, k = lane & 3;
  const int64_t i = p0 + lane;
  float z = 0.f;
  if (WPTS == 32 || lane < WPTS) {
    const int64_t ic = i < a.np ? i : a.np - 1;    // lanes past the end repeat the last point
    z = __ldg(&a.pts[3 * ic + 2]);
    PointCell c;
    point_xy<P2>(a, __ldg(&a.pts[3 * ic]), __ldg(&a.pts[3 * ic + 1]), c);
    const PlaneSlot& s = g.slots[~__float_as_uint(z) == g.slots[sl.x].key ? sl.x : sl.y];
    int rx, ry, bx, by;
    plane_box(a, s, rx, ry, bx, by);
    const int lx = min(max(wrapi<P2>(c.ix - 1 - (ref.x + rx), a.Nxr), 0), bx - 4);
    const int ly = min(max(wrapi<P2>(c.iy - 1 - (ref.y + ry), a.Nyr), 0), by - 4);
    GatherRec& r = rec[lane];
    r.cell = make_int4(s.off + ly * bx + lx, bx, 0, 0);
    r.wy = make_float4(c.wy[0], c.wy[1], c.wy[2], c.wy[3]);
    *reinterpret_cast<float4*>(r.wx) = make_float4(c.wx[0], c.wx[1], c.wx[2], c.wx[3]);
  }
  __syncwarp();
#pragma unroll
  for (int s = 0; s < WPTS / 8; ++s) {
    GatherRec& r = rec[8 * s + (lane >> 2)];
    const int4 c = r.cell;
    const float4 wy = r.wy;
    const float wxk = r.wx[k];
    const float wyb[4] = {wy.x, wy.y, wy.z, wy.w};
    unsigned long long uv = 0ull, wt = 0ull;
    float e = 0.f;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int o = c.x + b * c.y + k;
      const float4 v = __ldg(&g.cols[o]);
      const unsigned long long w2 = pack2(wyb[b], wyb[b]);
      fma2(uv, w2, pack2(v.x, v.y));
      fma2(wt, w2, pack2(v.z, v.w));
      e = fmaf(wyb[b], __ldg(&g.etas[o]), e);
    }
    quad_sum(uv, wt, e, wxk, k, r);
  }
  __syncwarp();
  if ((WPTS == 32 || lane < WPTS) && i < a.np) {
    const float4 f = *reinterpret_cast<const float4*>(rec[lane].wx);
    store_point(a, i, f, rec[lane].eta, z, z >= L.z[0] && z <= L.z[a.nz - 1]);
  }
}

// The chunks that read planes, from their list.
template <bool P2>
__global__ void __launch_bounds__(BOX_THREADS, 5) k_interp_planes(const __grid_constant__ InterpArgs a,
                                                                   const __grid_constant__ Levels L,
                                                                   const int4* __restrict__ plan,
                                                                   const __grid_constant__ GatherLists g) {
  __shared__ GatherRec rec[BOX_THREADS];
  const int n = g.n->n_plane;
  for (int li = blockIdx.x; li < n; li += gridDim.x) {
    const int chunk = g.l_plane[li];
    const int2 sl = g.chunk_slot[chunk];
#pragma unroll 1
    for (int k = 0; k < BOX_PPT; ++k) {
      const int64_t p0 = int64_t(chunk) * BOX_PTS + k * BOX_THREADS + (threadIdx.x & ~31);
      if (p0 >= a.np) break;                       // uniform over the warp
      plane_warp<P2, 32>(a, L, g, plan[0], sl, p0, rec + (threadIdx.x & ~31));
      __syncwarp();                                // the records are rewritten by the next turn
    }
  }
}

// The chunks with a staged tile, taken from their list.
template <bool P2>
__global__ void __launch_bounds__(BOX_THREADS, 3) k_interp_tiles(const __grid_constant__ InterpArgs a,
                                                                  const __grid_constant__ Levels L,
                                                                  const int4* __restrict__ plan, GatherLists g) {
  extern __shared__ float4 sbox[];
  float* seta = reinterpret_cast<float*>(sbox + BOX_NODES);
  __shared__ LevelTables zs;
  const int n = g.n->n_tile;
  if (int(blockIdx.x) >= n) return;
  fill_level_tables(zs, L);
  for (int li = blockIdx.x; li < n; li += gridDim.x) {
    __syncthreads();                               // shared memory free for the next chunk
    const int chunk = g.l_tile[li];
    box_chunk<P2, false>(a, zs, chunk, plan[chunk], sbox, seta);
  }
}

// ---------------------------------------------------------------------------------------------
// Batched gather (many instances, swense_batch_run): the point chunks of every instance form
// one list. One launch plans them all (a warp per chunk, the warp's own copy of its instance's
// arguments and level tables), then one persistent launch gathers them: each CTA takes the next
// chunk from a device counter and reloads the instance's arguments and level tables only when
// the instance changes (chunks are listed instance by instance, so rarely).
struct BatchInst {
  InterpArgs a;
  Levels L;
};

__device__ __forceinline__ int batch_instance(const int64_t* chunk0, int n, int64_t c) {
  int lo = 0, hi = n - 1;                           // last instance whose first chunk <= c
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (chunk0[mid] <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void copy_words(void* dst, const void* src, int bytes, int t, int nt) {
  const int* s = static_cast<const int*>(src);
  int* d = static_cast<int*>(dst);
  for (int i = t; i < bytes / 4; i += nt) d[i] = __ldg(&s[i]);
}

__global__ void __launch_bounds__(BOX_THREADS) k_interp_plan_batch(const BatchInst* __restrict__ inst,
                                                                   const int64_t* __restrict__ chunk0, int n,
                                                                   int4* __restrict__ plan) {
  extern __shared__ unsigned char smb[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  InterpArgs* sa = reinterpret_cast<InterpArgs*>(smb) + warp;
  LevelTables* zs = reinterpret_cast<LevelTables*>(smb + PLAN_WARPS * sizeof(InterpArgs)) + warp;
  const int64_t c = int64_t(blockIdx.x) * PLAN_WARPS + warp;
  if (c >= chunk0[n]) return;                       // no block barrier in this kernel
  const int i = batch_instance(chunk0, n, c);
  copy_words(sa, &inst[i].a, int(sizeof(InterpArgs)), lane, 32);
  copy_words(zs, &inst[i].L, int(sizeof(LevelTables)), lane, 32);
  __syncwarp();
  plan_chunk<true, BATCH_NODES>(*sa, *zs, c - chunk0[i], plan + chunk0[i], lane);
}

// The chunks with a staged tile, by persistent blocks.
__global__ void __launch_bounds__(BOX_THREADS, 2) k_interp_box_batch(const BatchInst* __restrict__ inst,
                                                                      const int64_t* __restrict__ chunk0, int n,
                                                                      const int4* __restrict__ plan,
                                                                      unsigned* __restrict__ counter) {
  extern __shared__ float4 sbox[];
  float* seta = reinterpret_cast<float*>(sbox + BATCH_NODES);
  __shared__ LevelTables zs;
  __shared__ InterpArgs sa;
  __shared__ int64_t s_item;
  const int64_t total = chunk0[n];
  int cur = -1;
  for (;;) {
    if (threadIdx.x == 0) {                         // the next chunk with a tile
      int64_t c = int64_t(atomicAdd(counter, 1u));
      while (c < total && plan_is_global(plan[c], inst[batch_instance(chunk0, n, c)].a.nz)) c = int64_t(atomicAdd(counter, 1u));
      s_item = c;
    }
    __syncthreads();
    const int64_t c = s_item;
    if (c >= total) break;                          // uniform over the CTA
    const int i = batch_instance(chunk0, n, c);
    if (i != cur) {
      copy_words(&sa, &inst[i].a, int(sizeof(InterpArgs)), threadIdx.x, blockDim.x);
      fill_level_tables(zs, inst[i].L);
      cur = i;
    }
    __syncthreads();                                // arguments and tables in place
    box_chunk<true, false>(sa, zs, c - chunk0[i], plan[c], sbox, seta);
    __syncthreads();                                // shared memory free for the next chunk
  }
}

// The others, straight from the grid in point order (as k_interp_global): without a tile's shared
// memory L1 holds the rows that neighbouring points share. Eight uneven instances, 4.2 M points at
// four time levels: 1.84 -> 1.06 ms, 0.35 of it the tiles of the dense instance (3.1 M points).
__global__ void __launch_bounds__(BOX_THREADS, 5) k_interp_global_batch(const BatchInst* __restrict__ inst,
                                                                         const int64_t* __restrict__ chunk0, int n,
                                                                         const int4* __restrict__ plan) {
  __shared__ GatherRec rec[GLOBAL_PTS];
  __shared__ InterpArgs sa;
  constexpr int SUB = BOX_PTS / GLOBAL_PTS;
  const int64_t c = blockIdx.x / SUB;
  const int i = batch_instance(chunk0, n, c);
  if (!plan_is_global(plan[c], inst[i].a.nz)) return;   // uniform over the block
  copy_words(&sa, &inst[i].a, int(sizeof(InterpArgs)), threadIdx.x, blockDim.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  const int64_t p0 = (c - chunk0[i]) * BOX_PTS + (blockIdx.x % SUB) * GLOBAL_PTS + warp * GLOBAL_WPTS;
  if (p0 >= sa.np) return;                          // uniform over the warp
  gather_warp<true, GLOBAL_WPTS>(sa, *level_tables(inst[i].L), p0, rec + warp * GLOBAL_WPTS);
}

// ---------------------------------------------------------------------------------------------
// Fused learned gather: the plain Lagrange gather, the network's inputs and its three layers in
// one kernel, per 1024-point chunk. The chunk's stencils come from the staged box (as in
// k_interp_box) when it fits, else from per-point stencil arrays gathered from global memory in the
// same shared memory. Each of the block's two warpgroups takes half of the chunk, some points at a time:
//   A (one thread per point): cell, Lagrange weights, offsets, eta, stencil base -> LPoint;
//   B (one thread per row = point and field, 32 points at a time): stencil values, Lagrange value and
//     max |value|; the normalised values (hi + lo BF16) go to tensor memory as the A operand of layer 1,
//     its accumulators come back through GELU as the A operand of layer 2, and layer 3's one output of
//     the row is an FP32 dot product; lagrange + s_f * out_scale * y[f] is the result;
//   C (one thread per point): Bernoulli, NaN outside the levels, stores.
// Bound by instruction issue (51 % of cycles, 17 % of the tensor cores'): 55 % of it GELU and the splits.
// A row per thread and the fifth-generation tensor cores leave about 850 issue slots per 16 rows where
// fragments of warp MMAs took 1260 and another 1140 cycles of the MMA pipe that did not overlap with them:
// 8.2 M mesh points 4.45 -> 3.00 ms. Two warpgroups a block and two blocks an SM fill one another's waits.
// Offsets and biases are a k-step of their own: a row's inputs 64..79 are the hi halves of dx, dy, dz,
// their lo halves and three ones, against the offsets' weights twice and the bias in three BF16 parts
// (its 24 bits); layer 2 repeats it with weights of zero.
struct alignas(16) LPoint {
  float w[12];              // wx[4], wy[4], wz[4]; the corrected fields overwrite w[0..3]
  float off[3];             // dx, dy in the cell; dz in the stencil's middle level interval
  int base;                 // staged node index of stencil node (x 0, y 0, level 0)
  float eta, z;
  int inside, pad_;
};
static_assert(sizeof(LPoint) == 80, "eight neighbouring records start in eight different groups of banks");

using mlpnet::PackedFwd;

constexpr int LRN_WG = BOX_THREADS / 128;              // warpgroups
constexpr int LRN_SB = 64, LRN_SB_PP = 32;             // points per step of a warpgroup: staged box, per-point stencils
constexpr int LRN_K = 16 * 5, LRN_LBO = mlpnet::NH / 8 * 128;   // bytes between neighbouring core matrices along K
constexpr uint32_t LRN_COLS = 128;                     // tensor-memory columns a warpgroup: A hi 0, A lo 32, D 64
constexpr uint32_t LRN_IDESC = tc::idesc_bf16_f32(128, mlpnet::NH);
static_assert(LRN_WG * LRN_SB_PP * 64 <= BOX_NODES, "per-point stencils fit the box area");
static_assert(mlpnet::KIN == LRN_K && mlpnet::NIN == 67 && mlpnet::NH == 64 && mlpnet::NOUT == 4, "the layout above");

struct LearnedSmem {
  unsigned char w1[LRN_K / 8 * LRN_LBO], w2[LRN_K / 8 * LRN_LBO];   // K-major core matrices
  unsigned char xo[LRN_WG + 1][128 * 16];              // inputs 64..71 of a warpgroup's rows; last: 72..79 of any
  float4 w3[mlpnet::NH / 4][mlpnet::NOUT];
  float b3[mlpnet::NOUT];
  float out_scale;
  uint32_t tmem;
  alignas(8) uint64_t bar[LRN_WG];
};
constexpr size_t LRN_SMEM = size_t(BOX_NODES) * sizeof(float4) + size_t(BOX_COLS) * sizeof(float) +
                            size_t(LRN_WG) * LRN_SB * sizeof(LPoint) + sizeof(LearnedSmem);
static_assert(2 * (LRN_SMEM + 1024) <= 228 * 1024, "two blocks an SM");

// Set when a wait for the tensor cores gives up; the host reads and clears it with swense_async_status.
__device__ int g_learned_timeout;

// Limit of those waits; withhold: no MMA is issued, so that every wait runs out (self-test).
struct LearnedWaits {
  int polls, withhold;
};

__device__ __forceinline__ void wg_sync(int wg) { asm volatile("bar.sync %0, 128;" ::"r"(1 + wg) : "memory"); }

// Eight inputs (k-chunk kc) of output n of a layer with K plain inputs and 16 more for offsets and bias.
__device__ __forceinline__ uint4 learned_weights(const __nv_bfloat16* w, const float* bias, bool offsets, int ldw, int n, int kc) {
  if (kc < 8) return __ldg(reinterpret_cast<const uint4*>(w + n * ldw) + kc);
  const float b = __ldg(&bias[n]);
  unsigned h, l, l2, unused;
  bf2_split(b, 0.f, h, l);
  bf2_split(b - __uint_as_float(h << 16) - __uint_as_float(l << 16), 0.f, l2, unused);
  if (kc == 9) return make_uint4(l2 & 0xffffu, 0u, 0u, 0u);
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (offsets) v = mlpnet::repeat_offsets(__ldg(reinterpret_cast<const uint4*>(w + n * ldw) + kc));
  v.w = (h & 0xffffu) | (l << 16);
  return v;
}

// One layer of a warpgroup's 128 rows, by one thread: D = [A hi + A lo | offsets] x W.
__device__ __forceinline__ void learned_mma(uint32_t ta, const unsigned char* w, const unsigned char* xo, uint32_t xo_lbo,
                                            uint64_t* bar) {
  tc::fence_after();
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    const uint64_t wd = tc::smem_desc(w + 2 * ks * LRN_LBO, LRN_LBO, 128u);
    tc::mma_ts(ta + 64u, ta + 8u * ks, wd, LRN_IDESC, ks > 0 ? 1u : 0u);
    tc::mma_ts(ta + 64u, ta + 32u + 8u * ks, wd, LRN_IDESC, 1u);
  }
  tc::mma_ss(ta + 64u, tc::smem_desc(xo, xo_lbo, 128u), tc::smem_desc(w + 8 * LRN_LBO, LRN_LBO, 128u), LRN_IDESC, 1u);
  tc::commit(bar);
}

// Accumulators 32 hf .. 32 hf + 31 of this thread's row after GELU, in pairs.
__device__ __forceinline__ void learned_activations(uint32_t lanes, int hf, float2 (&g)[16]) {
  uint32_t r0[16], r1[16];
  tc::ld_x16(lanes + 64u + 32u * hf, r0);
  tc::ld_x16(lanes + 64u + 32u * hf + 16u, r1);
  tc::wait_ld();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    g[i] = mlpnet::gelu_fast2(make_float2(__uint_as_float(r0[2 * i]), __uint_as_float(r0[2 * i + 1])));
    g[8 + i] = mlpnet::gelu_fast2(make_float2(__uint_as_float(r1[2 * i]), __uint_as_float(r1[2 * i + 1])));
  }
}

// 32 values of a row (pairs) as hi and lo BF16 halves into the A operand's words 16 hf .. 16 hf + 15.
__device__ __forceinline__ void learned_store_a(uint32_t lanes, int hf, const float2 (&g)[16]) {
  uint32_t hi[16], lo[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) bf2_split(g[i], hi[i], lo[i]);
  tc::st_x16(lanes + 16u * hf, hi);
  tc::st_x16(lanes + 32u + 16u * hf, lo);
}

// PARTS: `parts` blocks a chunk (learned_parts), each with its share of the points and its own tile.
template <bool PARTS>
__global__ void __launch_bounds__(BOX_THREADS, 2) k_interp_learned(const __grid_constant__ InterpArgs a, const __grid_constant__ Levels L,
                                                                    const int4* __restrict__ plan,
                                                                    const PackedFwd* __restrict__ Wg, LearnedWaits waits, int parts) {
  using namespace mlpnet;
  const int chunk = PARTS ? int(blockIdx.x) / parts : int(blockIdx.x);
  const int per = BOX_PTS / (LRN_WG * (PARTS ? parts : 1));   // points of a warpgroup
  const int64_t p0 = int64_t(chunk) * BOX_PTS, pb = PARTS ? p0 + int64_t(int(blockIdx.x) % parts) * (LRN_WG * per) : p0;
  if (PARTS && pb >= a.np) return;                     // uniform over the block
  extern __shared__ float4 sbox[];
  float* seta = reinterpret_cast<float*>(sbox + BOX_NODES);
  LPoint* recs = reinterpret_cast<LPoint*>(seta + BOX_COLS);
  LearnedSmem& W = *reinterpret_cast<LearnedSmem*>(recs + LRN_WG * LRN_SB);
  const LevelTables& zs = *level_tables(L);
  for (int i = threadIdx.x; i < NH * (LRN_K / 8); i += blockDim.x) {
    const int n = i / (LRN_K / 8), kc = i % (LRN_K / 8), o = kc * LRN_LBO + (n / 8) * 128 + (n % 8) * 16;
    *reinterpret_cast<uint4*>(W.w1 + o) = learned_weights(&Wg->w1[0][0], Wg->b1, true, KIN, n, kc);
    *reinterpret_cast<uint4*>(W.w2 + o) = learned_weights(&Wg->w2[0][0], Wg->b2, false, NH, n, kc);
  }
  if (threadIdx.x < 128)                               // input 72 is 1, 73..79 are 0
    *reinterpret_cast<uint4*>(W.xo[LRN_WG] + 16 * threadIdx.x) = make_uint4(0x3f80u, 0u, 0u, 0u);
  if (threadIdx.x < NH) {
    const int k4 = threadIdx.x / NOUT, f = threadIdx.x % NOUT;
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(&Wg->w3[f][4 * k4]));
    W.w3[k4][f] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                              __uint_as_float(w.y & 0xffff0000u));
  }
  if (threadIdx.x < NOUT) W.b3[threadIdx.x] = __ldg(&Wg->b3[threadIdx.x]);
  if (threadIdx.x == 0) {
    W.out_scale = __ldg(&Wg->out_scale);
    for (int i = 0; i < LRN_WG; ++i) mbar_init(&W.bar[i], 1);
    fence_mbar_init();
  }
  __syncwarp();
  if (threadIdx.x < 32) {
    tc::alloc(&W.tmem, LRN_WG * LRN_COLS);
    tc::relinquish();
  }
  const int4 pl = plan[chunk];
  const BoxPlan bp = decode_plan(pl);
  const int bx = bp.bx, by = bp.by;
  const int sbx = bx + ((4 - bx) & 7);
  const int zst = box_zstride(sbx, by);
  int l0 = bp.l0, bz = bp.bz;
  bool box3d = bp.box3d;
  if (bp.two) {
    // a chunk across two layers: the box spans the level windows of its first and last point's z
    PointCell ca, cb;
    point_level(a, zs, __ldg(&a.pts[3 * p0 + 2]), ca);
    point_level(a, zs, __ldg(&a.pts[3 * ((p0 + BOX_PTS < a.np ? p0 + BOX_PTS : a.np) - 1) + 2]), cb);
    l0 = min(ca.j0, cb.j0);
    bz = abs(ca.j0 - cb.j0) + 4;
    box3d = int64_t(zst) * bz <= BOX_NODES && int64_t(sbx) * by <= BOX_COLS;
  }
  const bool boxed = box3d && l0 + bz <= a.nz;
  const int x0 = bp.x0, y0 = bp.y0;
  const size_t plane = size_t(a.Nyr) * a.Nxr;
  if (boxed) stage_box(a, x0, y0, l0, bx, by, bz, sbx, zst, sbox, seta);
  fence_proxy_async();                                 // the weights, read by the tensor cores
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const int wg = threadIdx.x >> 7, t = threadIdx.x & 127, f = t & 3;
  const uint32_t ta = W.tmem + uint32_t(wg) * LRN_COLS, lanes = ta + (uint32_t(t & 96) << 16);
  unsigned char* xo = W.xo[wg];
  const uint32_t xo_lbo = uint32_t(LRN_WG - wg) * uint32_t(sizeof(W.xo[0]));
  uint64_t* bar = &W.bar[wg];
  LPoint* rec = recs + wg * LRN_SB;
  float4* own = sbox + wg * (LRN_SB_PP * 64);          // the warpgroup's per-point stencils
  const float* nf = reinterpret_cast<const float*>(boxed ? sbox : own) + f;
  const int SY = boxed ? sbx : 4, SZ = boxed ? zst : 16;
  const int SB = boxed ? LRN_SB : LRN_SB_PP;
  const int64_t q0 = pb + int64_t(wg) * per;
  unsigned ph = 0;
  bool bad = false;
  // every thread of the warpgroup has its share of the operands in place -> the accumulators are ready
  auto run_layer = [&](const unsigned char* w) {
    tc::wait_st();
    fence_proxy_async();
    tc::fence_before();
    wg_sync(wg);
    if (t == 0 && !bad && !waits.withhold) learned_mma(ta, w, xo, xo_lbo, bar);
    __syncwarp();
    if (!bad) bad = !mbar_wait(bar, ph, waits.polls);
    if (!bad) ph ^= 1u;                                // a thread that gave up stays at the phase it gave up on
    __syncwarp();
    tc::fence_after();
  };
  for (int s0 = 0; s0 < per; s0 += SB) {
    int npts = int(a.np - (q0 + s0) < int64_t(SB) ? a.np - (q0 + s0) : int64_t(SB));
    if (PARTS) npts = min(npts, per - s0);
    if (npts <= 0) break;                              // uniform over the warpgroup
    // ---- A
    auto record = [&](LPoint& P, const PointCell& c, float px, float py, float pz, int base, float e) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        P.w[k] = c.wx[k];
        P.w[4 + k] = c.wy[k];
        P.w[8 + k] = c.wz[k];
      }
      float fx, fy;
      int ixx, iyy;
      locate(px, a.sx_hi, a.sx_lo, a.Nxr, ixx, fx);
      locate(py, a.sy_hi, a.sy_lo, a.Nyr, iyy, fy);
      const float z1 = zs.z[c.j0 + 1], z2 = zs.z[c.j0 + 2];
      P.off[0] = fx;
      P.off[1] = fy;
      P.off[2] = (pz - z1) / (z2 - z1);
      P.base = base;
      P.eta = e;
      P.z = pz;
      P.inside = c.inside;
    };
    if (boxed) {
      if (t < npts) {
        const int64_t i = q0 + s0 + t;
        const float px = __ldg(&a.pts[3 * i]), py = __ldg(&a.pts[3 * i + 1]), pz = __ldg(&a.pts[3 * i + 2]);
        const PointCell c = point_cell(a, zs, px, py, pz);
        const int lx = min(max((c.ix - 1 - x0) & (a.Nxr - 1), 0), bx - 4);
        const int ly = min(max((c.iy - 1 - y0) & (a.Nyr - 1), 0), by - 4);
        const int lz = min(max(c.j0 - l0, 0), bz - 4);
        float e = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int k = 0; k < 4; ++k) e = fmaf(c.wy[b] * c.wx[k], seta[(ly + b) * sbx + lx + k], e);
        record(rec[t], c, px, py, pz, lz * zst + ly * sbx + lx, e);
      }
    } else {
      // per-point stencils: four threads per point, each blends 16 of its 64 nodes
      const int j = t >> 2, qq = t & 3;
      if (j < npts) {
        const int64_t i = q0 + s0 + j;
        const float px = __ldg(&a.pts[3 * i]), py = __ldg(&a.pts[3 * i + 1]), pz = __ldg(&a.pts[3 * i + 2]);
        const PointCell c = point_cell(a, zs, px, py, pz);
        const size_t tl_stride = size_t(a.nz) * plane;
#pragma unroll 4
        for (int kk = 0; kk < 16; ++kk) {
          const int node = 16 * qq + kk, zq = node >> 4, b = (node >> 2) & 3, k = node & 3;
          const size_t gi = size_t(c.j0 + zq) * plane + size_t((c.iy - 1 + b) & (a.Nyr - 1)) * a.Nxr +
                            size_t((c.ix - 1 + k) & (a.Nxr - 1));
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int tl = 0; tl < a.n_tl; ++tl) {
            const float4 gv = __ldg(&a.nodes[size_t(tl) * tl_stride + gi]);
            const float w = a.wt[tl];
            v.x = fmaf(w, gv.x, v.x);
            v.y = fmaf(w, gv.y, v.y);
            v.z = fmaf(w, gv.z, v.z);
            v.w = fmaf(w, gv.w, v.w);
          }
          own[64 * j + node] = v;
        }
        if (qq == 0) {
          float e = 0.f;
          for (int tl = 0; tl < a.n_tl; ++tl)
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
              for (int k = 0; k < 4; ++k)
                e = fmaf(a.wt[tl] * c.wy[b] * c.wx[k],
                         __ldg(&a.eta[size_t(tl) * plane + size_t((c.iy - 1 + b) & (a.Nyr - 1)) * a.Nxr +
                                      ((c.ix - 1 + k) & (a.Nxr - 1))]), e);
          record(rec[j], c, px, py, pz, 64 * j, e);
        }
      }
    }
    wg_sync(wg);
    // ---- B (rows past the last point repeat it and are not kept)
    for (int g0 = 0; g0 < npts; g0 += 32) {
      const int j = g0 + (t >> 2);
      float lag = 0.f, mx = 0.f;
      {
        const LPoint& P = rec[min(j, npts - 1)];
        const float4 w4x = *reinterpret_cast<const float4*>(&P.w[0]), w4y = *reinterpret_cast<const float4*>(&P.w[4]),
                     w4z = *reinterpret_cast<const float4*>(&P.w[8]), o4 = *reinterpret_cast<const float4*>(&P.off[0]);
        const float wx[4] = {w4x.x, w4x.y, w4x.z, w4x.w}, wy[4] = {w4y.x, w4y.y, w4y.z, w4y.w},
                    wz[4] = {w4z.x, w4z.y, w4z.z, w4z.w};
        const float* src = nf + 4 * __float_as_int(o4.w);
        float2 v[2][16];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          float sy = 0.f;
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            float x[4], sx = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              x[k] = src[4 * (kk * SZ + b * SY + k)];
              sx = fmaf(wx[k], x[k], sx);
              mx = fmaxf(mx, fabsf(x[k]));
            }
            sy = fmaf(wy[b], sx, sy);
            v[kk >> 1][8 * (kk & 1) + 2 * b] = make_float2(x[0], x[1]);
            v[kk >> 1][8 * (kk & 1) + 2 * b + 1] = make_float2(x[2], x[3]);
          }
          lag = fmaf(wz[kk], sy, lag);
        }
        mx += 1e-30f;
        const float inv = 1.f / mx;
        __syncwarp();
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[hf][i] = pmul(v[hf][i], make_float2(inv, inv));
          learned_store_a(lanes, hf, v[hf]);
        }
        unsigned h, l, hz, lz;
        bf2_split(o4.x, o4.y, h, l);
        bf2_split(o4.z, 0.f, hz, lz);
        *reinterpret_cast<uint4*>(xo + 16 * t) =
            make_uint4(h, (hz & 0xffffu) | (l << 16), (l >> 16) | (lz << 16), 0x3f803f80u);
      }
      run_layer(W.w1);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        float2 g[16];
        learned_activations(lanes, hf, g);
        learned_store_a(lanes, hf, g);
      }
      run_layer(W.w2);
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        float2 g[16];
        learned_activations(lanes, hf, g);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 w = W.w3[8 * hf + i][f];
          acc = pfma(g[2 * i], make_float2(w.x, w.y), acc);
          acc = pfma(g[2 * i + 1], make_float2(w.z, w.w), acc);
        }
      }
      const float y = acc.x + acc.y + W.b3[f];
      if (j < npts) rec[j].w[f] = bad ? __int_as_float(0x7fc00000) : fmaf(mx * W.out_scale, y, lag);
    }
    wg_sync(wg);
    // ---- C
    if (t < npts) {
      const LPoint& P = rec[t];
      store_point(a, q0 + s0 + t, make_float4(P.w[0], P.w[1], P.w[2], P.w[3]), P.eta, P.z, P.inside != 0);
    }
    wg_sync(wg);
  }
  if (bad) {
    atomicExch(&g_learned_timeout, 1);
    // thread 0 issues a layer only after it has seen the one before complete, so the MMAs that may still be
    // in flight are those of the phase it gave up on
    if (t == 0) mbar_wait(bar, ph, waits.polls);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (threadIdx.x < 32) tc::dealloc(W.tmem, LRN_WG * LRN_COLS);
}

void split(double v, float& hi, float& lo) {
  hi = float(v);
  lo = float(v - double(hi));
}

}  // namespace
}  // namespace swense

// ---------------------------------------------------------------------------------------------
// Inputs of the learned correction: per point and field f in (u, v, w, dphi/dt) one row
//   x = [stencil_f / s_f (64 time-blended node values, x fastest, then y, then z), dx, dy, dz, 0]
// with s_f = max |stencil_f| + 1e-30 and dz the offset in the stencil's middle level interval,
// plus s_f, the plain Lagrange value of f, and the plain eta.
namespace swense {
namespace {

constexpr int MLP_XLD = 68;

struct FeatArgs {
  InterpArgs a;          // grid, points, time weights (o_* unused)
  float* x;              // [4 np][68]
  float* scale;          // [4 np]
  float* lag;            // [4 np]
  float* eta_out;        // [np] or NULL
};

__global__ void __launch_bounds__(128) k_mlp_features(FeatArgs f, const __grid_constant__ Levels L) {
  __shared__ LevelTables zs;
  const InterpArgs& a = f.a;
  fill_level_tables(zs, L);
  __syncthreads();
  const size_t plane = size_t(a.Nyr) * a.Nxr;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < a.np;
       i += int64_t(gridDim.x) * blockDim.x) {
    const float px = a.pts[3 * i], py = a.pts[3 * i + 1], pz = a.pts[3 * i + 2];
    const PointCell c = point_cell(a, zs, px, py, pz);
    float fx, fy;
    int ixx, iyy;
    locate(px, a.sx_hi, a.sx_lo, a.Nxr, ixx, fx);
    locate(py, a.sy_hi, a.sy_lo, a.Nyr, iyy, fy);
    const float z1 = zs.z[c.j0 + 1], z2 = zs.z[c.j0 + 2];
    const float fz = (pz - z1) / (z2 - z1);
    int xi[4], yi[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      xi[q] = (c.ix - 1 + q) & (a.Nxr - 1);
      yi[q] = (c.iy - 1 + q) & (a.Nyr - 1);
    }
    if (f.eta_out) {
      float e = 0.f;
      for (int tl = 0; tl < a.n_tl; ++tl)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            e = fmaf(a.wt[tl] * c.wy[b] * c.wx[k], __ldg(&a.eta[tl * plane + size_t(yi[b]) * a.Nxr + xi[k]]), e);
      f.eta_out[i] = e;
    }
#pragma unroll 1
    for (int fld = 0; fld < 4; ++fld) {
      float* xr = f.x + (4 * i + fld) * MLP_XLD;
      float smax = 0.f, lagv = 0.f;
      // pass 1: time-blended stencil values -> row (unscaled), max, Lagrange value
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const float wzq = q == 0 ? c.wz[0] : q == 1 ? c.wz[1] : q == 2 ? c.wz[2] : c.wz[3];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const size_t node = size_t(c.j0 + q) * plane + size_t(yi[b]) * a.Nxr + xi[k];
            float v = 0.f;
            for (int tl = 0; tl < a.n_tl; ++tl)
              v = fmaf(a.wt[tl], __ldg(reinterpret_cast<const float*>(&a.nodes[tl * a.nz * plane + node]) + fld), v);
            xr[(q * 4 + b) * 4 + k] = v;
            smax = fmaxf(smax, fabsf(v));
            lagv = fmaf(wzq * c.wy[b] * c.wx[k], v, lagv);
          }
        }
      }
      const float s = smax + 1e-30f;
      const float inv = 1.f / s;
      for (int k = 0; k < 64; ++k) xr[k] *= inv;
      xr[64] = fx;
      xr[65] = fy;
      xr[66] = fz;
      xr[67] = 0.f;
      f.scale[4 * i + fld] = s;
      f.lag[4 * i + fld] = lagv;
    }
  }
}

// Validate a grid request and fill the launch arguments shared by the interpolation entry points.
int prepare_interp(const swense_grid* g, double t, const float* pts, int64_t np, int32_t p_mode,
                   double rho, double grav, InterpArgs* a, Levels* lev) {
  if (!g || !g->nodes || !g->eta || !g->z_levels || !g->t_levels)
    return fail(SWENSE_ERR_ARG, "NULL grid, grid arrays or level lists");
  if (np < 0) return fail(SWENSE_ERR_ARG, "np must be >= 0");
  if (np > 0 && !pts) return fail(SWENSE_ERR_ARG, "NULL pts");
  // node counts: even in [4, MAX] (powers of two, or a non-power-of-two padding factor times
  // one); ny_r = 1 for a 2-D grid
  if ((g->nx_r & 1) || g->nx_r < 4 || g->nx_r > SWENSE_MAX_FFT ||
      (g->ny_r != 1 && ((g->ny_r & 1) || g->ny_r < 4)) || g->ny_r > SWENSE_MAX_FFT)
    return fail(SWENSE_ERR_SIZE, "nx_r must be even in [4, MAX], ny_r 1 or even in [4, MAX]");
  if (g->nz < 4 || g->nz > SWENSE_MAX_LEVELS) return fail(SWENSE_ERR_LEVELS, "need 4 <= nz <= SWENSE_MAX_LEVELS");
  if (g->n_tl < 1 || g->n_tl > SWENSE_MAX_TL) return fail(SWENSE_ERR_ARG, "n_tl must be in [1, SWENSE_MAX_TL]");
  if (p_mode != SWENSE_P_DYN && p_mode != SWENSE_P_PHIT && p_mode != SWENSE_P_TOTAL)
    return fail(SWENSE_ERR_ARG, "unknown p_mode");
  if (!(g->Lx > 0) || !std::isfinite(g->Lx) || (g->ny_r > 1 && (!(g->Ly > 0) || !std::isfinite(g->Ly))))
    return fail(SWENSE_ERR_ARG, "domain lengths must be finite and positive");
  if (!std::isfinite(t) || !std::isfinite(rho) || !std::isfinite(grav))
    return fail(SWENSE_ERR_ARG, "non-finite t, rho or g");
  if (reinterpret_cast<uintptr_t>(g->nodes) & 15) return fail(SWENSE_ERR_ARG, "nodes must be 16-byte aligned");
  for (int l = 0; l < g->nz; ++l) {
    lev->z[l] = g->z_levels[l];
    if (!std::isfinite(lev->z[l]) || (l > 0 && !(lev->z[l] > lev->z[l - 1])))
      return fail(SWENSE_ERR_LEVELS, "z_levels must be finite and strictly increasing");
  }
  {
    const int nz = g->nz;
    for (int j = 0; j + 3 < nz; ++j) {
      double zn[4], d[4];
      for (int q = 0; q < 4; ++q) zn[q] = lev->z[j + q];
      for (int q = 0; q < 4; ++q) {
        d[q] = 1.0;
        for (int r = 0; r < 4; ++r)
          if (r != q) d[q] *= zn[q] - zn[r];
      }
      lev->inv[j] = make_float4(float(1.0 / d[0]), float(1.0 / d[1]), float(1.0 / d[2]), float(1.0 / d[3]));
    }
    const double z0 = lev->z[0], h = (double(lev->z[nz - 1]) - z0) / ZLUT;
    lev->z0 = lev->z[0];
    lev->inv_h = float(1.0 / h);
    unsigned char lut[ZLUT];
    int j = 0;
    for (int b = 0; b < ZLUT; ++b) {
      const double zb = z0 + b * h;
      while (j + 1 < nz && double(lev->z[j + 1]) <= zb) ++j;
      lut[b] = (unsigned char)j;
    }
    std::memcpy(lev->lut4, lut, sizeof(lut));
  }
  for (int l = 0; l < g->n_tl; ++l) {
    if (!std::isfinite(g->t_levels[l]) || (l > 0 && !(g->t_levels[l] > g->t_levels[l - 1])))
      return fail(SWENSE_ERR_ARG, "t_levels must be finite and strictly increasing");
  }
  *a = InterpArgs{};
  for (int l = 0; l < g->n_tl; ++l) {
    double wl = 1.0;
    for (int m = 0; m < g->n_tl; ++m)
      if (m != l) wl *= (t - g->t_levels[m]) / (g->t_levels[l] - g->t_levels[m]);
    a->wt[l] = float(wl);
  }
  a->nodes = reinterpret_cast<const float4*>(g->nodes);
  a->eta = g->eta;
  a->pts = pts;
  a->np = np;
  a->Nxr = g->nx_r;
  a->Nyr = g->ny_r;
  a->nz = g->nz;
  a->n_tl = g->n_tl;
  split(double(g->nx_r) / g->Lx, a->sx_hi, a->sx_lo);
  if (g->ny_r > 1) split(double(g->ny_r) / g->Ly, a->sy_hi, a->sy_lo);
  a->p_mode = p_mode;
  a->rho = float(rho);
  a->g = float(grav);
  if (g->scheme != SWENSE_LAGRANGE3 && g->scheme != SWENSE_SPLINE3)
    return fail(SWENSE_ERR_ARG, "unknown interpolation scheme");
  a->spline = g->scheme == SWENSE_SPLINE3;
  a->p2 = is_pow2(g->nx_r) && is_pow2(g->ny_r);
  return SWENSE_OK;
}

}  // namespace
}  // namespace swense

using namespace swense;

extern "C" int swense_mlp_features(const swense_grid* g, double t, const float* pts, int64_t np,
                                   float* x, float* scale, float* lagrange, float* eta,
                                   void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  InterpArgs a;
  Levels lev;
  int st = prepare_interp(g, t, pts, np, SWENSE_P_DYN, 1.0, 1.0, &a, &lev);
  if (st) return st;
  if (g->ny_r < 4) return fail(SWENSE_ERR_UNSUPPORTED, "the learned correction needs a 3-D grid");
  if (a.spline) return fail(SWENSE_ERR_UNSUPPORTED, "the learned correction is defined on LAGRANGE3 grids");
  if (!a.p2) return fail(SWENSE_ERR_UNSUPPORTED, "the learned correction needs power-of-two node counts");
  if (np == 0) return SWENSE_OK;
  if (!x || !scale || !lagrange) return fail(SWENSE_ERR_ARG, "NULL feature outputs");
  FeatArgs f{a, x, scale, lagrange, eta};
  const unsigned blocks = unsigned(std::min<int64_t>((np + 127) / 128, 152 * 64));
  k_mlp_features<<<blocks, 128, 0, stream>>>(f, lev);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

namespace swense {
namespace {

std::mutex g_learned_selftest_mutex;
bool g_learned_selftest[64];      // per device (swense_selftest_learned_wait_timeout)

// Blocks a chunk. A chunk is a chain of sixteen 32-point steps for each warpgroup, 0.19 ms, which a set of few
// chunks waits for whole (500 points: 191 us, with warp MMAs 150 before; 30 us in 16 parts), and a grid of one
// wave of blocks and a little takes two. So chunks are split, down to one step a warpgroup, up to five waves
// of blocks: 400,000 points in two parts 622 -> 485 us, 200,000 in four 346 -> 264. More waves would still
// help points of their own stencils, but every part stages its chunk's box again (400,000 points on a grid of
// 64 x 32 nodes: 195 us whole, 197 in two parts, 209 in four).
int learned_parts(int64_t chunks, int64_t slots) {
  int parts = 1;
  while (parts < BOX_PTS / (LRN_WG * 32) && chunks * parts * 2 <= 5 * slots) parts *= 2;
  return parts;
}

int learned_waits(LearnedWaits* w) {
  int dev = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(g_learned_selftest_mutex);
  const bool on = dev >= 0 && dev < 64 && g_learned_selftest[dev];
  *w = on ? LearnedWaits{8, 1} : LearnedWaits{kMbarPolls, 0};
  return SWENSE_OK;
}

}  // namespace

int learned_async_flag(bool reset, int* was_set) {
  int v = 0;
  SWENSE_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_learned_timeout, sizeof(int)));
  if (reset && v) {
    const int zero = 0;
    SWENSE_CUDA_TRY(cudaMemcpyToSymbol(g_learned_timeout, &zero, sizeof(int)));
  }
  *was_set = v;
  return SWENSE_OK;
}

}  // namespace swense

extern "C" int swense_selftest_learned_wait_timeout(int32_t on) {
  int dev = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SWENSE_ERR_UNSUPPORTED, "device index too large");
  std::lock_guard<std::mutex> lock(g_learned_selftest_mutex);
  g_learned_selftest[dev] = on != 0;
  return SWENSE_OK;
}

extern "C" int swense_interp_learned(const swense_grid* g, double t, const float* pts, int64_t np,
                                     float* eta, float* u, float* v, float* w, float* p,
                                     int32_t p_mode, double rho, double grav, const void* packed,
                                     int64_t* n_out_of_range, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  InterpArgs a;
  Levels lev;
  int st = prepare_interp(g, t, pts, np, p_mode, rho, grav, &a, &lev);
  if (st) return st;
  if (g->ny_r < 4) return fail(SWENSE_ERR_UNSUPPORTED, "the learned correction needs a 3-D grid");
  if (a.spline) return fail(SWENSE_ERR_UNSUPPORTED, "the learned correction is defined on LAGRANGE3 grids");
  if (!a.p2) return fail(SWENSE_ERR_UNSUPPORTED, "the learned correction needs power-of-two node counts");
  if (!packed) return fail(SWENSE_ERR_ARG, "NULL packed weights");
  if (reinterpret_cast<uintptr_t>(packed) & 15) return fail(SWENSE_ERR_ARG, "packed weights must be 16-byte aligned");
  // workspace: [0, 256) out-of-range counter, then one int4 box plan per 1024-point chunk
  const int64_t blocks = (np + BOX_PTS - 1) / BOX_PTS;
  if (blocks >= (int64_t(1) << 31)) return fail(SWENSE_ERR_SIZE, "too many points for one call");
  void* ws = nullptr;
  st = workspace(256 + size_t(blocks) * sizeof(int4), stream, &ws);
  if (st) return st;
  unsigned long long* d_count = static_cast<unsigned long long*>(ws);
  if (n_out_of_range) SWENSE_CUDA_TRY(cudaMemsetAsync(d_count, 0, sizeof(unsigned long long), stream));
  if (np > 0) {
    a.o_eta = eta;
    a.o_u = u;
    a.o_v = v;
    a.o_w = w;
    a.o_p = p;
    a.n_oor = n_out_of_range ? d_count : nullptr;
    int4* plan = reinterpret_cast<int4*>(static_cast<char*>(ws) + 256);
    k_interp_plan<true><<<unsigned(plan_blocks(np)), BOX_THREADS, 0, stream>>>(a, lev, plan);
    SWENSE_CUDA_TRY(cudaGetLastError());
    int dev = 0, sms = 0;
    SWENSE_CUDA_TRY(cudaGetDevice(&dev));
    SWENSE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int parts = learned_parts(blocks, 2 * sms);
    const auto kernel = parts > 1 ? k_interp_learned<true> : k_interp_learned<false>;
    SWENSE_CUDA_TRY(cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(LRN_SMEM)));
    LearnedWaits waits;
    st = learned_waits(&waits);
    if (st) return st;
    kernel<<<unsigned(blocks * parts), BOX_THREADS, LRN_SMEM, stream>>>(
        a, lev, plan, static_cast<const PackedFwd*>(packed), waits, parts);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(2);
  }
  if (n_out_of_range) {
    unsigned long long h = 0;
    SWENSE_CUDA_TRY(cudaMemcpyAsync(&h, d_count, sizeof(h), cudaMemcpyDeviceToHost, stream));
    SWENSE_CUDA_TRY(cudaStreamSynchronize(stream));
    *n_out_of_range = int64_t(h);
  }
  return SWENSE_OK;
}

namespace swense {
namespace {

size_t up256(size_t b) { return (b + 255) & ~size_t(255); }

// Scratch of the gather by kinds of chunks, after the counters and the plan: 2 columns per point, at
// most 2^26, which holds a mesh's planes with room to spare.
int plane_units(int64_t np) { return int(std::min<int64_t>(2 * np, int64_t(1) << 26) / PLANE_UNIT); }
size_t lists_bytes(int64_t np, int64_t chunks) {
  const size_t cols = size_t(plane_units(np)) * PLANE_UNIT;
  return up256(PLANE_SLOTS * sizeof(PlaneSlot)) + up256(PLANE_SLOTS * sizeof(PlaneGroup)) +
         up256(PLANE_SLOTS * sizeof(int)) + up256(chunks * sizeof(int2)) + 3 * up256(chunks * sizeof(int)) + up256(cols * sizeof(float4)) + up256(cols * sizeof(float));
}
GatherLists lists_in(char* c, int64_t np, int64_t chunks, void* counts, bool lanes) {
  const size_t cols = size_t(plane_units(np)) * PLANE_UNIT;
  GatherLists g;
  auto take = [&](size_t b) { char* q = c; c += up256(b); return q; };
  g.n = static_cast<GatherCounts*>(counts);
  g.slots = reinterpret_cast<PlaneSlot*>(take(PLANE_SLOTS * sizeof(PlaneSlot)));
  g.groups = reinterpret_cast<PlaneGroup*>(take(PLANE_SLOTS * sizeof(PlaneGroup)));
  g.members = reinterpret_cast<int*>(take(PLANE_SLOTS * sizeof(int)));
  g.chunk_slot = reinterpret_cast<int2*>(take(chunks * sizeof(int2)));
  g.l_plane = reinterpret_cast<int*>(take(chunks * sizeof(int)));
  g.l_tile = reinterpret_cast<int*>(take(chunks * sizeof(int)));
  g.l_lanes = reinterpret_cast<int*>(take(chunks * sizeof(int)));
  g.cols = reinterpret_cast<float4*>(take(cols * sizeof(float4)));
  g.etas = reinterpret_cast<float*>(take(cols * sizeof(float)));
  g.max_units = plane_units(np);
  g.lanes = lanes;
  return g;
}

template <bool P2>
int interp_by_kind(const InterpArgs& a, const Levels& lev, const int4* plan, int chunks, int sms, const GatherLists& g,
                   cudaStream_t stream) {
  SWENSE_CUDA_TRY(cudaMemsetAsync(g.slots, 0, PLANE_SLOTS * sizeof(PlaneSlot), stream));
  k_gather_register<P2><<<unsigned((chunks + 255) / 256), 256, 0, stream>>>(a, plan, chunks, g);
  SWENSE_CUDA_TRY(cudaGetLastError());
  k_gather_lists<<<1, 1024, 0, stream>>>(a, lev, plan, chunks, g);
  SWENSE_CUDA_TRY(cudaGetLastError());
  k_plane_collapse<P2><<<unsigned(sms * 4), BOX_THREADS, 0, stream>>>(a, lev, plan, g);
  SWENSE_CUDA_TRY(cudaGetLastError());
  SWENSE_CUDA_TRY(cudaFuncSetAttribute((const void*)k_interp_tiles<P2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(BOX_SMEM)));
  k_interp_tiles<P2><<<unsigned(sms * 3), BOX_THREADS, BOX_SMEM, stream>>>(a, lev, plan, g);
  SWENSE_CUDA_TRY(cudaGetLastError());
  k_interp_planes<P2><<<unsigned(sms * 5), BOX_THREADS, 0, stream>>>(a, lev, plan, g);
  SWENSE_CUDA_TRY(cudaGetLastError());
  k_interp_global<P2><<<unsigned((a.np + GLOBAL_PTS - 1) / GLOBAL_PTS), BOX_THREADS, 0, stream>>>(
      a, lev, plan, &g.n->n_global, g.chunk_slot, 1);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(6);
  if (g.lanes) {
    k_interp_lanes<P2><<<unsigned(sms * 4), BOX_THREADS, 0, stream>>>(a, lev, plan, g.l_lanes, &g.n->n_lanes, &g.n->lane_ticket);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);
  }
  return SWENSE_OK;
}

// plan_in: a plan made earlier by swense_interp_plan for these points and this grid geometry
// (NULL: make one in the workspace first).
int interp_impl(const swense_grid* g, double t, const float* pts, const int32_t* perm, int64_t np,
                float* eta, float* u, float* v, float* w, float* p, int32_t p_mode, double rho,
                double grav, int64_t* n_out_of_range, cudaStream_t stream,
                const int4* plan_in = nullptr) {
  InterpArgs a;
  Levels lev;
  int st = prepare_interp(g, t, pts, np, p_mode, rho, grav, &a, &lev);
  if (st) return st;
  // workspace: [0, 256) counters, one int4 box plan per 1024-point chunk (unless given), and for many
  // points the lists and planes of the gather by kinds, which is passed over where they cannot be had
  const int64_t blocks = (np + BOX_PTS - 1) / BOX_PTS;
  const size_t b_plan = 256 + (plan_in ? 0 : up256(size_t(blocks) * sizeof(int4)));
  // sparse point sets (fewer points than a quarter of a time level's nodes): a chunk's stencils rarely
  // fit a tile
  const bool sparse = double(np) < 0.25 * double(a.Nxr) * double(a.Nyr) * double(a.nz);
  bool kinds = sparse && a.Nyr > 1 && np >= LAYER_POINTS && blocks < (int64_t(1) << 31) / (BOX_PTS / GLOBAL_PTS);
  void* ws = nullptr;
  st = kinds ? workspace_optional(b_plan + lists_bytes(np, blocks), stream, &ws) : SWENSE_OK;
  if (st || !kinds) {
    kinds = false;
    st = workspace(b_plan, stream, &ws);
  }
  if (st) return st;
  unsigned long long* d_count = nullptr;
  if (n_out_of_range) {
    d_count = static_cast<unsigned long long*>(ws);
    SWENSE_CUDA_TRY(cudaMemsetAsync(d_count, 0, sizeof(unsigned long long), stream));
  }
  if (np > 0) {
    a.o_eta = eta;
    a.o_u = u;
    a.o_v = v;
    a.o_w = w;
    a.o_p = p;
    a.n_oor = d_count;
    a.perm = perm;
    if (blocks >= (int64_t(1) << 31)) return fail(SWENSE_ERR_SIZE, "too many points for one call");
    // Fewer chunks than SMs: planning and staging would be two launches of a few blocks each, bound by
    // latency (18 + 25 us for 50,000 points of a 2-D wave); the gather without tiles fills the GPU from
    // a few thousand points on (50,000 points: 7 us). Above that, the tiles' reuse wins on meshes.
    int dev = 0, sms = 0;
    SWENSE_CUDA_TRY(cudaGetDevice(&dev));
    SWENSE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const bool small = blocks < sms;
    // Chunks marked ROWS_BIT by lanes: on grids whose four levels of all time levels do not stay in L2 (on others
    // what a layer or row of tiles reads is still there for the next, and quads are faster), from 2^19 points on
    // (400,000 binned points on the four-fold padded grid: 355 us either way), and below 2^21, where it is one
    // more launch for every set, for binned points only (a mesh of a million points would lose 5 of 120 us).
    bool lanes = sparse && (kinds || perm) && np >= (int64_t(1) << 19) && a.Nyr > 1;
    if (lanes) {
      int l2 = 0;
      SWENSE_CUDA_TRY(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev));
      lanes = double(a.Nxr) * a.Nyr * 64 * a.n_tl > 0.75 * double(l2);
    }
    const int4* plan = small ? nullptr : plan_in;
    if (!plan && !small) {
      int4* pw = reinterpret_cast<int4*>(static_cast<char*>(ws) + 256);
      if (a.p2) k_interp_plan<true><<<unsigned(plan_blocks(np)), BOX_THREADS, 0, stream>>>(a, lev, pw);
      else k_interp_plan<false><<<unsigned(plan_blocks(np)), BOX_THREADS, 0, stream>>>(a, lev, pw);
      SWENSE_CUDA_TRY(cudaGetLastError());
      count_launches(1);
      plan = pw;
    }
    if (kinds) {
      const GatherLists g = lists_in(static_cast<char*>(ws) + b_plan, np, blocks, ws, lanes);
      st = a.p2 ? interp_by_kind<true>(a, lev, plan, int(blocks), sms, g, stream)
                : interp_by_kind<false>(a, lev, plan, int(blocks), sms, g, stream);
      if (st) return st;
    }
    // Sparse sets send the chunks without a tile to k_interp_global, where L1 is not reduced by the
    // tile; dense ones (meshes at their grid's resolution) gather the rare such chunks inside
    // k_interp_box and skip the second launch.
    const bool split = small || sparse;
    if (!kinds) {
      const void* kbox = a.p2 ? (split ? (const void*)k_interp_box<true, true> : (const void*)k_interp_box<true, false>)
                              : (split ? (const void*)k_interp_box<false, true> : (const void*)k_interp_box<false, false>);
      SWENSE_CUDA_TRY(cudaFuncSetAttribute(kbox, cudaFuncAttributeMaxDynamicSharedMemorySize, int(BOX_SMEM)));
      if (split) {
        if (!small) {
          if (a.p2) k_interp_box<true, true><<<unsigned(blocks), BOX_THREADS, BOX_SMEM, stream>>>(a, lev, plan);
          else k_interp_box<false, true><<<unsigned(blocks), BOX_THREADS, BOX_SMEM, stream>>>(a, lev, plan);
          count_launches(1);
        }
        // two rounds a block from 2^20 points on: a mesh's blocks with nothing to do are half as many (1.1 to 2 M
        // mesh points on grids of 1024 x 512 to 2048 x 1024: 2 to 7 % less, 85.4 -> 79.4 us of 2 M, the like or up
        // to 2 % more with three time levels; points in no order 0.7 % more); not for binned points, which lose by
        // it (1.1 M on 1024 x 512: 414 against 526 us); fewer points would leave too few blocks
        const int rounds = !perm && np >= (int64_t(1) << 20) ? 2 : 1;
        const unsigned gctas = unsigned((np + rounds * GLOBAL_PTS - 1) / (rounds * GLOBAL_PTS));
        const auto kglobal = a.p2 ? (lanes ? k_interp_global<true, true> : k_interp_global<true>)
                                  : (lanes ? k_interp_global<false, true> : k_interp_global<false>);
        kglobal<<<gctas, BOX_THREADS, 0, stream>>>(a, lev, plan, nullptr, nullptr, rounds);
        count_launches(1);
        if (lanes) {
          const unsigned lctas = unsigned(blocks * LANE_PARTS);
          if (a.p2) k_interp_lanes<true><<<lctas, BOX_THREADS, 0, stream>>>(a, lev, plan, nullptr, nullptr, nullptr);
          else k_interp_lanes<false><<<lctas, BOX_THREADS, 0, stream>>>(a, lev, plan, nullptr, nullptr, nullptr);
          count_launches(1);
        }
      } else {
        if (a.p2) k_interp_box<true, false><<<unsigned(blocks), BOX_THREADS, BOX_SMEM, stream>>>(a, lev, plan);
        else k_interp_box<false, false><<<unsigned(blocks), BOX_THREADS, BOX_SMEM, stream>>>(a, lev, plan);
        count_launches(1);
      }
      SWENSE_CUDA_TRY(cudaGetLastError());
    }
  }
  if (n_out_of_range) {
    unsigned long long h = 0;
    SWENSE_CUDA_TRY(cudaMemcpyAsync(&h, d_count, sizeof(h), cudaMemcpyDeviceToHost, stream));
    SWENSE_CUDA_TRY(cudaStreamSynchronize(stream));
    *n_out_of_range = int64_t(h);
  }
  return SWENSE_OK;
}

}  // namespace
}  // namespace swense

extern "C" int64_t swense_interp_plan_bytes(int64_t np) {
  return np <= 0 ? 0 : ((np + BOX_PTS - 1) / BOX_PTS) * int64_t(sizeof(int4));
}

extern "C" int swense_interp_plan(const swense_grid* g, const float* pts, int64_t np, void* plan,
                                  void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  InterpArgs a;
  Levels lev;
  const double t0 = g && g->t_levels ? g->t_levels[0] : 0.0;
  int st = prepare_interp(g, t0, pts, np, SWENSE_P_DYN, 1.0, 1.0, &a, &lev);
  if (st) return st;
  if (np == 0) return SWENSE_OK;
  if (!plan || (reinterpret_cast<uintptr_t>(plan) & 15)) return fail(SWENSE_ERR_ARG, "plan must be non-NULL and 16-byte aligned");
  const int64_t blocks = (np + BOX_PTS - 1) / BOX_PTS;
  if (blocks >= (int64_t(1) << 31)) return fail(SWENSE_ERR_SIZE, "too many points for one call");
  if (a.p2) k_interp_plan<true><<<unsigned(plan_blocks(np)), BOX_THREADS, 0, stream>>>(a, lev, static_cast<int4*>(plan));
  else k_interp_plan<false><<<unsigned(plan_blocks(np)), BOX_THREADS, 0, stream>>>(a, lev, static_cast<int4*>(plan));
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

extern "C" int swense_interp_with_plan(const swense_grid* g, double t, const float* pts, int64_t np,
                                       const void* plan, float* eta, float* u, float* v, float* w,
                                       float* p, int32_t p_mode, double rho, double grav,
                                       int64_t* n_out_of_range, void* stream) {
  if (np > 0 && (!plan || (reinterpret_cast<uintptr_t>(plan) & 15)))
    return fail(SWENSE_ERR_ARG, "plan must be non-NULL and 16-byte aligned");
  return interp_impl(g, t, pts, nullptr, np, eta, u, v, w, p, p_mode, rho, grav, n_out_of_range,
                     static_cast<cudaStream_t>(stream), static_cast<const int4*>(plan));
}

extern "C" int swense_interp(const swense_grid* g, double t, const float* pts, int64_t np,
                             float* eta, float* u, float* v, float* w, float* p, int32_t p_mode,
                             double rho, double grav, int64_t* n_out_of_range, void* stream) {
  return interp_impl(g, t, pts, nullptr, np, eta, u, v, w, p, p_mode, rho, grav, n_out_of_range,
                     static_cast<cudaStream_t>(stream));
}

extern "C" int swense_interp_permuted(const swense_grid* g, double t, const float* pts_sorted,
                                      const int32_t* perm, int64_t np, float* eta, float* u,
                                      float* v, float* w, float* p, int32_t p_mode, double rho,
                                      double grav, int64_t* n_out_of_range, void* stream) {
  if (np > 0 && !perm) return fail(SWENSE_ERR_ARG, "NULL perm");
  return interp_impl(g, t, pts_sorted, perm, np, eta, u, v, w, p, p_mode, rho, grav,
                     n_out_of_range, static_cast<cudaStream_t>(stream));
}

namespace swense {
namespace {

// Per device: the batch tables in device memory (instances' arguments and level tables, chunk
// offsets) and their host copy. Rewritten (synchronously, so never during a stream capture)
// only when a batch's tables differ from the last ones; a captured batch therefore replays the
// tables of the uncaptured call that preceded it.
struct BatchTables {
  void* dev = nullptr;
  size_t cap = 0;
  std::vector<double> key;          // the inputs the tables were built from
  int64_t nchunks = 0;
};

// Everything the batch tables depend on, field by field (no struct padding).
std::vector<double> batch_key(const GatherItem* items, int n, int32_t p_mode, double rho, double grav) {
  std::vector<double> k{double(n), double(p_mode), rho, grav};
  auto ptr = [&](const void* q) { k.push_back(double(reinterpret_cast<uintptr_t>(q))); };
  for (int i = 0; i < n; ++i) {
    const GatherItem& it = items[i];
    const swense_grid& g = it.grid;
    ptr(g.nodes); ptr(g.eta); ptr(it.pts); ptr(it.perm);
    ptr(it.eta); ptr(it.u); ptr(it.v); ptr(it.w); ptr(it.p);
    k.insert(k.end(), {double(it.np), it.t, double(g.nx_r), double(g.ny_r), double(g.nz), double(g.n_tl),
                       g.Lx, g.Ly, double(g.scheme)});
    for (int l = 0; l < g.nz && g.z_levels; ++l) k.push_back(double(g.z_levels[l]));
    for (int l = 0; l < g.n_tl && g.t_levels; ++l) k.push_back(g.t_levels[l]);
  }
  return k;
}
std::mutex g_batch_mutex;
BatchTables g_batch[64];

int batch_tables(const GatherItem* items, int n, int32_t p_mode, double rho, double grav, cudaStream_t stream,
                 const BatchInst** d_inst, const int64_t** d_chunk0, int64_t* nchunks) {
  int dev = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SWENSE_ERR_UNSUPPORTED, "device index too large");
  std::vector<double> key = batch_key(items, n, p_mode, rho, grav);
  std::lock_guard<std::mutex> lock(g_batch_mutex);
  BatchTables& T = g_batch[dev];
  if (T.dev && T.key == key) {                      // the same batch as last time: tables in place
    *d_inst = static_cast<const BatchInst*>(T.dev);
    *d_chunk0 = reinterpret_cast<const int64_t*>(static_cast<const char*>(T.dev) + size_t(n) * sizeof(BatchInst));
    *nchunks = T.nchunks;
    return SWENSE_OK;
  }
  std::vector<unsigned char> h(size_t(n) * sizeof(BatchInst) + size_t(n + 1) * sizeof(int64_t));
  BatchInst* bi = reinterpret_cast<BatchInst*>(h.data());
  int64_t* c0 = reinterpret_cast<int64_t*>(h.data() + size_t(n) * sizeof(BatchInst));
  c0[0] = 0;
  for (int k = 0; k < n; ++k) {
    const GatherItem& it = items[k];
    InterpArgs a;
    Levels lev;
    int st = prepare_interp(&it.grid, it.t, it.pts, it.np, p_mode, rho, grav, &a, &lev);
    if (st) return st;
    if (!a.p2) return fail(SWENSE_ERR_UNSUPPORTED, "batched gathers take power-of-two node counts");
    a.o_eta = it.eta;
    a.o_u = it.u;
    a.o_v = it.v;
    a.o_w = it.w;
    a.o_p = it.p;
    a.perm = it.perm;
    a.n_oor = nullptr;
    std::memcpy(&bi[k].a, &a, sizeof(InterpArgs));
    std::memcpy(&bi[k].L, &lev, sizeof(Levels));
    c0[k + 1] = c0[k] + (it.np + BOX_PTS - 1) / BOX_PTS;
  }
  {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    SWENSE_CUDA_TRY(cudaStreamIsCapturing(stream, &cap));
    if (cap != cudaStreamCaptureStatusNone)
      return fail(SWENSE_ERR_ARG, "a captured swense_batch_run must follow an uncaptured call with the "
                                  "same instances (its tables are uploaded outside the capture)");
    SWENSE_CUDA_TRY(cudaStreamSynchronize(stream));
    if (h.size() > T.cap) {
      if (T.dev) SWENSE_CUDA_TRY(cudaFree(T.dev));
      T.dev = nullptr;
      T.cap = 0;
      cudaError_t e = cudaMalloc(&T.dev, h.size());
      if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(SWENSE_ERR_OOM, "cudaMalloc of the batch tables failed");
      }
      T.cap = h.size();
    }
    SWENSE_CUDA_TRY(cudaMemcpy(T.dev, h.data(), h.size(), cudaMemcpyHostToDevice));
    T.key.swap(key);
    T.nchunks = c0[n];
  }
  *d_inst = static_cast<const BatchInst*>(T.dev);
  *d_chunk0 = reinterpret_cast<const int64_t*>(static_cast<const char*>(T.dev) + size_t(n) * sizeof(BatchInst));
  *nchunks = T.nchunks;
  return SWENSE_OK;
}

}  // namespace

int interp_batch_bytes(const GatherItem* items, int n, size_t* bytes) {
  int64_t chunks = 0;
  for (int k = 0; k < n; ++k) chunks += (items[k].np + BOX_PTS - 1) / BOX_PTS;
  *bytes = 256 + size_t(chunks) * sizeof(int4);
  return SWENSE_OK;
}

int interp_batch(const GatherItem* items, int n, int32_t p_mode, double rho, double grav, void* ws,
                 cudaStream_t stream) {
  if (n <= 0) return SWENSE_OK;
  const BatchInst* d_inst = nullptr;
  const int64_t* d_chunk0 = nullptr;
  int64_t nchunks = 0;
  int st = batch_tables(items, n, p_mode, rho, grav, stream, &d_inst, &d_chunk0, &nchunks);
  if (st) return st;
  if (nchunks == 0) return SWENSE_OK;
  if (nchunks >= (int64_t(1) << 31) / (BOX_PTS / GLOBAL_PTS)) return fail(SWENSE_ERR_SIZE, "too many point chunks in one batch");
  unsigned* counter = static_cast<unsigned*>(ws);
  int4* plan = reinterpret_cast<int4*>(static_cast<char*>(ws) + 256);
  const size_t plan_smem = size_t(PLAN_WARPS) * (sizeof(InterpArgs) + sizeof(LevelTables));
  SWENSE_CUDA_TRY(cudaFuncSetAttribute((const void*)k_interp_plan_batch,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, int(plan_smem)));
  k_interp_plan_batch<<<unsigned((nchunks + PLAN_WARPS - 1) / PLAN_WARPS), BOX_THREADS, plan_smem, stream>>>(
      d_inst, d_chunk0, n, plan);
  SWENSE_CUDA_TRY(cudaGetLastError());
  SWENSE_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(unsigned), stream));
  SWENSE_CUDA_TRY(cudaFuncSetAttribute((const void*)k_interp_box_batch,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, int(BATCH_SMEM)));
  int dev = 0, sms = 0, per_sm = 0;
  SWENSE_CUDA_TRY(cudaGetDevice(&dev));
  SWENSE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SWENSE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_interp_box_batch, BOX_THREADS,
                                                                BATCH_SMEM));
  const int64_t ctas = std::min<int64_t>(nchunks, int64_t(std::max(1, sms * std::max(1, per_sm))));
  k_interp_box_batch<<<unsigned(ctas), BOX_THREADS, BATCH_SMEM, stream>>>(d_inst, d_chunk0, n, plan, counter);
  SWENSE_CUDA_TRY(cudaGetLastError());
  k_interp_global_batch<<<unsigned(nchunks * (BOX_PTS / GLOBAL_PTS)), BOX_THREADS, 0, stream>>>(d_inst, d_chunk0, n, plan);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(3);
  return SWENSE_OK;
}

}  // namespace swense
