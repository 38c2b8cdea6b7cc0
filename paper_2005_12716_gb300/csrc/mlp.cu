// Learned correction of the interpolated fields (not in the paper; an addition to its
// interpolation step): one multilayer perceptron shared by the four fields u, v, w, dphi/dt,
//   input  x = [stencil_f / s_f (64 time-blended 4x4x4 node values, x fastest, then y, then z),
//              dx, dy, dz (offsets of the point in the stencil's middle cell)],
//              s_f = max |stencil_f| + 1e-30,
//   layers 67 -> 64 -> 64 -> 4, GELU (tanh form) on the hidden layers, output y[f] used,
//   correction  f = lagrange_f + s_f y[f], pressure from the corrected fields (Bernoulli).
//
// Tensor cores: BF16 mma.sync (m16n8k16) with FP32 accumulation (the fused gather in interp.cu runs the
// same network on tcgen05); one warp owns 16 rows, and a layer's accumulator fragments become the next layer's A fragments in registers. Inference
// splits inputs and activations into BF16 hi + lo (two MMAs per step) so the result tracks an
// FP64 evaluation of the same BF16 weights to ~1e-5; training uses plain BF16 operands.
// Weight gradients (sums over the batch) are formed on the CUDA cores in FP32 by the block that made
// the rows' activations, reduced over the blocks in a fixed order, then Adam.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "internal.cuh"
#include "mlp.cuh"

namespace swense {
namespace {

using namespace mlpnet;

// ------------------------------------------------------------------------------ pack
__global__ void k_mlp_pack(const float* __restrict__ P, Packed* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < NH * KIN) {
    const int n = i / KIN, k = i % KIN;
    out->w1[n][k] = __float2bfloat16_rn(k < NIN ? P[OFF_W1 + n * NIN + k] : 0.f);
  }
  if (i < NH * NH) {
    const int n = i / NH, k = i % NH;
    out->w2[n][k] = __float2bfloat16_rn(P[OFF_W2 + n * NH + k]);
    out->w2t[n][k] = __float2bfloat16_rn(P[OFF_W2 + k * NH + n]);
  }
  if (i < NO * NH) {
    const int n = i / NH, k = i % NH;
    out->w3[n][k] = __float2bfloat16_rn(n < NOUT ? P[OFF_W3 + n * NH + k] : 0.f);
  }
  if (i < NH * 16) {
    const int n = i / 16, k = i % 16;
    out->w3t[n][k] = __float2bfloat16_rn(k < NOUT ? P[OFF_W3 + k * NH + n] : 0.f);
  }
  if (i < NH) {
    out->b1[i] = P[OFF_B1 + i];
    out->b2[i] = P[OFF_B2 + i];
  }
  if (i < NO) out->b3[i] = i < NOUT ? P[OFF_B3 + i] : 0.f;
}

// A fragments of 16 rows of x (FP32, leading dimension XLD; rows past the end read as 0).
__device__ __forceinline__ void load_x(const float* __restrict__ x, int64_t row0, int64_t rows, unsigned (&ahi)[4][4],
                                       unsigned (&alo)[4][4], unsigned (&off)[2], int lane) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int h = 0; h < 2; ++h) {                    // a0, a2: row g; a1, a3: row g + 8
    const int64_t r = row0 + g + 8 * h;
    const float* xr = r < rows ? x + r * XLD : nullptr;
    auto at = [&](int col) { return xr ? __ldg(&xr[col]) : 0.f; };
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int col = 16 * kk + 2 * t + 8 * q;
        bf2_split(at(col), at(col + 1), ahi[kk][h + 2 * q], alo[kk][h + 2 * q]);
      }
    off[h] = offsets_a(at(64), at(65), at(66), t);
  }
}

// Inference: y[row] = network(x[row])[row % 4] (rows ordered point-major, fields u, v, w, phit).
__global__ void __launch_bounds__(128) k_mlp_forward(const Packed* __restrict__ P, const float* __restrict__ x,
                                                     int64_t rows, float* __restrict__ y) {
  __shared__ __align__(16) Packed s;               // copied and read (ldmatrix) in 16-byte rows
  {
    const uint4* src = reinterpret_cast<const uint4*>(P);
    uint4* dst = reinterpret_cast<uint4*>(&s);
    for (int i = threadIdx.x; i < int(sizeof(Packed) / 16); i += blockDim.x)
      dst[i] = i < NH * KIN / 8 && i % (KIN / 8) == 8 ? repeat_offsets(src[i]) : src[i];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  for (int64_t row0 = (int64_t(blockIdx.x) * 4 + warp) * 16; row0 < rows;
       row0 += int64_t(gridDim.x) * 64) {
    unsigned xh[4][4], xl[4][4], xo[2];
    load_x(x, row0, rows, xh, xl, xo, lane);
    float o[4];
    infer(o, xh, xl, xo, s, KIN, NH, lane);
    // row r uses output column r % 4: c0/c1 hold columns 2t, 2t+1 of row g, c2/c3 of row g+8
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t r = row0 + g + 8 * h;
      const int f = (g + 8 * h) & 3;               // row0 is a multiple of 16
      const float yv = (f & 1) ? o[2 * h + 1] : o[2 * h];   // a select, not a local array
      if (r < rows && (f >> 1) == t) y[r] = yv * s.out_scale;
    }
  }
}

// ------------------------------------------------------------------------------ training
// One block takes TROWS rows of the batch at a time: its warps 0..3 run forward and backward on 16 rows
// each (tensor cores) and leave the rows' activations and gradients in shared memory, from which its
// eight other warps add the rows' contribution to every weight gradient, a 4 x 8 tile of one matrix a
// thread (three 16-byte shared loads per 32 products); separate warps, so that neither part's registers
// burden the other (twelve warps in all: three per scheduler leave 168 registers a thread). The sums stay in registers over the block's rows and
// go to the block's own row of `part`. With the activations written out to memory and one thread per
// parameter summing 256 rows, the gradients took 47 us of a 62 us step (batch 8192); this kernel does
// both passes in 21 us (a latency chain of three layers forward and back on one wave of blocks).
constexpr int TROWS = 64, TFB = 128, TTHR = TFB + 256, XS = 72, HS = NH + 4;
struct TrainSmem {
  Packed p;
  float x[TROWS][XS];              // columns >= NIN zero
  float h1[TROWS][HS], h2[TROWS][HS], dz1[TROWS][HS], dz2[TROWS][HS];
  float dy[TROWS][4];
  float loss[4];
};
struct TrainArgs {
  const Packed* P;
  const float* x;          // [N][XLD] features
  const int32_t* field;    // [N]
  const float* target;     // [N]
  const int32_t* batch;    // [B] row indices into x
  int B;
  float* part;             // [gridDim.x][NPARAM] per-block gradient sums
  float* loss_part;        // [gridDim.x] per-block sums of squared residuals / B
  float tscale;            // targets are multiplied by this on reading
};

__global__ void __launch_bounds__(TTHR, 1) k_mlp_train(TrainArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  TrainSmem& s = *reinterpret_cast<TrainSmem*>(smraw);
  const int tid = threadIdx.x;
  {
    const int4* src = reinterpret_cast<const int4*>(a.P);
    int4* dst = reinterpret_cast<int4*>(&s.p);
    for (int i = tid; i < int(sizeof(Packed) / 16); i += TTHR) dst[i] = src[i];
  }
  const int lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const float invB = 1.f / float(a.B);
  const int step = int(gridDim.x) * TROWS;
  // both halves of the block pass the same barriers, three per tile of rows, from their own loops
  auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(TTHR) : "memory"); };
  __syncthreads();                                 // the weights are in place
  if (warp < 4) {
    float lsum = 0.f;
    for (int r0 = blockIdx.x * TROWS; r0 < a.B; r0 += step) {
      sync();                                      // the tile's x rows are in place
      const int w0 = 16 * warp;
      unsigned xh[5][4];
#pragma unroll
      for (int kk = 0; kk < 5; ++kk)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = w0 + g + 8 * (q & 1), col = 16 * kk + 2 * t + (q >= 2 ? 8 : 0);
          xh[kk][q] = col < XS ? bf2(s.x[r][col], s.x[r][col + 1]) : 0u;
        }
      float z1[8][4];
      layer<5, 8>(z1, xh, &s.p.w1[0][0], KIN, s.p.b1, lane);
      unsigned h1[4][4];
      to_a<8>(z1, h1);
      float z2[8][4];
      layer<4, 8>(z2, h1, &s.p.w2[0][0], NH, s.p.b2, lane);
      unsigned h2[4][4];
      to_a<8>(z2, h2);
      float o[1][4];
      layer<4, 1>(o, h2, &s.p.w3[0][0], NH, s.p.b3, lane);
      // dY: only the row's own output column carries 2 (y - target) / B
      float dyf[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t rr = int64_t(r0) + w0 + g + 8 * h;
        const bool ok = rr < a.B;
        const int src = ok ? a.batch[rr] : 0;
        const int f = ok ? a.field[src] : -1;
        const float tg = ok ? a.target[src] * a.tscale : 0.f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int col = 2 * t + c;
          float d = 0.f;
          if (col == f) {
            const float res = o[0][2 * h + c] - tg;
            lsum = fmaf(res, res, lsum);
            d = 2.f * res * invB;
          }
          dyf[2 * h + c] = d;
        }
      }
      // dH2 = dY W3  (K = 8 padded to 16)
      unsigned ady[4] = {bf2(dyf[0], dyf[1]), bf2(dyf[2], dyf[3]), 0u, 0u};
      float dz2[8][4];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        dz2[nt][0] = dz2[nt][1] = dz2[nt][2] = dz2[nt][3] = 0.f;
        const __nv_bfloat16* wr = &s.p.w3t[8 * nt + g][2 * t];
        mma16816(dz2[nt], ady, ld_u32(wr), ld_u32(wr + 8));
      }
      // dZ2 = dH2 * gelu'(Z2); dH1 = dZ2 W2
#pragma unroll
      for (int nt = 0; nt < 8; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) dz2[nt][q] *= gelu_grad(z2[nt][q]);
      unsigned adz2[4][4];
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        adz2[kk][0] = bf2(dz2[2 * kk][0], dz2[2 * kk][1]);
        adz2[kk][1] = bf2(dz2[2 * kk][2], dz2[2 * kk][3]);
        adz2[kk][2] = bf2(dz2[2 * kk + 1][0], dz2[2 * kk + 1][1]);
        adz2[kk][3] = bf2(dz2[2 * kk + 1][2], dz2[2 * kk + 1][3]);
      }
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        float dh1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const __nv_bfloat16* wr = &s.p.w2t[8 * nt + g][16 * kk + 2 * t];
          mma16816(dh1, adz2[kk], ld_u32(wr), ld_u32(wr + 8));
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = w0 + g + 8 * h, col = 8 * nt + 2 * t;
          const float e0 = z1[nt][2 * h], e1 = z1[nt][2 * h + 1];
          *reinterpret_cast<float2*>(&s.h1[r][col]) = make_float2(gelu(e0), gelu(e1));
          *reinterpret_cast<float2*>(&s.h2[r][col]) = make_float2(gelu(z2[nt][2 * h]), gelu(z2[nt][2 * h + 1]));
          *reinterpret_cast<float2*>(&s.dz2[r][col]) = make_float2(dz2[nt][2 * h], dz2[nt][2 * h + 1]);
          *reinterpret_cast<float2*>(&s.dz1[r][col]) =
              make_float2(dh1[2 * h] * gelu_grad(e0), dh1[2 * h + 1] * gelu_grad(e1));
        }
      }
      if (t < 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<float2*>(&s.dy[w0 + g + 8 * h][2 * t]) = make_float2(dyf[2 * h], dyf[2 * h + 1]);
      }
      sync();                                      // activations and gradients are in place
      sync();                                      // and have been read
    }
    // per-block loss in a fixed order (no atomics: training is reproducible bit for bit)
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) s.loss[warp] = lsum;
    sync();
    if (tid == 0) a.loss_part[blockIdx.x] = ((s.loss[0] + s.loss[1]) + (s.loss[2] + s.loss[3])) * invB;
    return;
  }
  // this thread's tile of the gradients: rows of L (dz1, dz2 or dy) times rows of R (x, h1 or h2)
  const int v = tid - TFB;
  const bool first = v < 128;                      // dW1, columns 0..63, or dW2: 16 x 8 tiles of 4 x 8
  const int ig = (v & 127) >> 3, kg = v & 7;
  const float* Lp = first ? &s.dz1[0][4 * ig] : &s.dz2[0][4 * ig];
  const float* Rp = first ? &s.x[0][8 * kg] : &s.h1[0][8 * kg];
  const int ldr = first ? XS : HS;
  // four more sums: dW1's columns 64..66 (threads 0..47) and dW3's columns (threads 48..111)
  const bool extra = v < 112, w1x = v < 48;
  const float* Lx = w1x ? &s.dz1[0][4 * (v / 3)] : &s.dy[0][0];
  const float* Rx = w1x ? &s.x[0][64 + v % 3] : &s.h2[0][(v - 48) & 63];
  const int ldlx = w1x ? HS : 4, ldrx = w1x ? XS : HS;
  const float* bp = v < NH ? &s.dz1[0][v] : (v < 2 * NH ? &s.dz2[0][v - NH] : &s.dy[0][v & 3]);
  const int ldb = v < 2 * NH ? HS : 4;
  float acc[4][8], accx[4] = {0.f, 0.f, 0.f, 0.f}, bacc = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[i][k] = 0.f;
  for (int r0 = blockIdx.x * TROWS; r0 < a.B; r0 += step) {
#pragma unroll 4
    for (int i = v; i < TROWS * XS; i += TTHR - TFB) {
      const int r = i / XS, c = i % XS;
      s.x[r][c] = r0 + r < a.B && c < NIN ? __ldg(&a.x[int64_t(__ldg(&a.batch[r0 + r])) * XLD + c]) : 0.f;
    }
    sync();
    sync();
    // rows past the batch carry dy = 0, so dz1 and dz2 are zero and they add nothing
#pragma unroll 4
    for (int r = 0; r < TROWS; ++r) {
      const float4 l = *reinterpret_cast<const float4*>(Lp + r * HS);
      const float4 x0 = *reinterpret_cast<const float4*>(Rp + r * ldr);
      const float4 x1 = *reinterpret_cast<const float4*>(Rp + r * ldr + 4);
      const float lv[4] = {l.x, l.y, l.z, l.w}, xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[i][k] = fmaf(lv[i], xv[k], acc[i][k]);
    }
    if (extra) {
#pragma unroll 8
      for (int r = 0; r < TROWS; ++r) {
        const float4 l = *reinterpret_cast<const float4*>(Lx + r * ldlx);
        const float xv = Rx[r * ldrx];
        accx[0] = fmaf(l.x, xv, accx[0]);
        accx[1] = fmaf(l.y, xv, accx[1]);
        accx[2] = fmaf(l.z, xv, accx[2]);
        accx[3] = fmaf(l.w, xv, accx[3]);
      }
    }
    if (v < 2 * NH + NOUT) {
#pragma unroll 8
      for (int r = 0; r < TROWS; ++r) bacc += bp[r * ldb];
    }
    sync();
  }
  float* part = a.part + size_t(blockIdx.x) * NPARAM;
  const int off = first ? OFF_W1 : OFF_W2, ld = first ? NIN : NH;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 8; ++k) part[off + (4 * ig + i) * ld + 8 * kg + k] = acc[i][k];
  if (extra) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      part[w1x ? OFF_W1 + (4 * (v / 3) + i) * NIN + 64 + v % 3 : OFF_W3 + i * NH + v - 48] = accx[i];
  }
  if (v < 2 * NH + NOUT)
    part[v < NH ? OFF_B1 + v : (v < 2 * NH ? OFF_B2 + v - NH : OFF_B3 + v - 2 * NH)] = bacc;
  sync();                                          // pairs with the loss's barrier
}

// grad = sum over the blocks' parts in a fixed order (eight interleaved runs, then the runs), loss
// likewise; with params given, one Adam step and the refreshed BF16 copies of the parameter (the
// padding of the packed layout never changes).
struct UpdateArgs {
  const float* part;
  int nparts;
  float* grad;                     // NULL: not wanted
  const float* loss_part;
  float* loss;                     // NULL: not wanted
  float *P, *m, *v;                // NULL: gradient only
  Packed* out;
  float lr, b1, b2, eps, bc1, bc2;
};
constexpr int UPD_RUNS = 8;
__global__ void __launch_bounds__(32 * UPD_RUNS) k_mlp_update(UpdateArgs a) {
  __shared__ float run[UPD_RUNS][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float acc = 0.f;
  if (p < NPARAM) {
#pragma unroll 8
    for (int q = w; q < a.nparts; q += UPD_RUNS) acc += a.part[size_t(q) * NPARAM + p];
  }
  run[w][lane] = acc;
  if (blockIdx.x == 0 && w == 1 && a.loss) {
    float l = 0.f;
    for (int q = lane; q < a.nparts; q += 32) l += a.loss_part[q];
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) *a.loss = l;
  }
  __syncthreads();
  if (w != 0 || p >= NPARAM) return;
  float gr = 0.f;
#pragma unroll
  for (int q = 0; q < UPD_RUNS; ++q) gr += run[q][lane];
  if (a.grad) a.grad[p] = gr;
  if (!a.P) return;
  const float mm = fmaf(a.b1, a.m[p], (1.f - a.b1) * gr);
  const float vv = fmaf(a.b2, a.v[p], (1.f - a.b2) * gr * gr);
  a.m[p] = mm;
  a.v[p] = vv;
  const float np = a.P[p] - a.lr * (mm / a.bc1) / (sqrtf(vv / a.bc2) + a.eps);
  a.P[p] = np;
  Packed& o = *a.out;
  const __nv_bfloat16 b = __float2bfloat16_rn(np);
  if (p < OFF_B1) {
    o.w1[p / NIN][p % NIN] = b;
  } else if (p < OFF_W2) {
    o.b1[p - OFF_B1] = np;
  } else if (p < OFF_B2) {
    const int i = (p - OFF_W2) / NH, k = (p - OFF_W2) % NH;
    o.w2[i][k] = b;
    o.w2t[k][i] = b;
  } else if (p < OFF_W3) {
    o.b2[p - OFF_B2] = np;
  } else if (p < OFF_B3) {
    const int i = (p - OFF_W3) / NH, k = (p - OFF_W3) % NH;
    o.w3[i][k] = b;
    o.w3t[k][i] = b;
  } else {
    o.b3[p - OFF_B3] = np;
  }
}

// Mini-batch row indices of training step `step` (0-based): SplitMix64 (Steele, Lea and Flood,
// "Fast splittable pseudorandom number generators", 2014) of the counter seed + step 2^32 + i,
// reduced modulo n; the same (seed, step) always draws the same batch.
__global__ void k_mlp_batch(uint64_t seed, int64_t step, int64_t n, int B, int32_t* __restrict__ idx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B) return;
  uint64_t z = seed + (uint64_t(step) << 32) + uint64_t(i) + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  idx[i] = int32_t(z % uint64_t(n));
}

// Sum of squares of the n targets (FP64), for the RMS output scale.
__global__ void k_mlp_sumsq(const float* __restrict__ t, int64_t n, double* __restrict__ out) {
  double acc = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    acc += double(t[i]) * double(t[i]);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

// Training targets of the learned correction: row 4 i + f (point i, field f = u, v, w, phi_t)
// gets (exact_f - lagrange_f) / s_f and field id f.
__global__ void k_mlp_targets(const float* __restrict__ eu, const float* __restrict__ ev,
                              const float* __restrict__ ew, const float* __restrict__ et,
                              const float* __restrict__ lag, const float* __restrict__ sc, int64_t np,
                              float* __restrict__ target, int32_t* __restrict__ field) {
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= 4 * np) return;
  const int64_t i = r >> 2;
  const int f = int(r & 3);
  const float ex = f == 0 ? eu[i] : f == 1 ? ev[i] : f == 2 ? ew[i] : et[i];
  target[r] = (ex - lag[r]) / sc[r];
  field[r] = f;
}

}  // namespace
}  // namespace swense

using namespace swense;

extern "C" int swense_mlp_pack(const float* params, float out_scale, void* packed, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (!params || !packed) return fail(SWENSE_ERR_ARG, "NULL params or packed buffer");
  if (reinterpret_cast<uintptr_t>(packed) & 15) return fail(SWENSE_ERR_ARG, "packed must be 16-byte aligned");
  if (!std::isfinite(out_scale) || !(out_scale > 0)) return fail(SWENSE_ERR_ARG, "out_scale must be finite and > 0");
  k_mlp_pack<<<(NH * KIN + 255) / 256, 256, 0, stream>>>(params, static_cast<Packed*>(packed));
  SWENSE_CUDA_TRY(cudaGetLastError());
  SWENSE_CUDA_TRY(cudaMemcpyAsync(&static_cast<Packed*>(packed)->out_scale, &out_scale, sizeof(float),
                                  cudaMemcpyHostToDevice, stream));
  SWENSE_CUDA_TRY(cudaStreamSynchronize(stream));
  count_launches(1);
  return SWENSE_OK;
}

extern "C" int swense_mlp_forward(const void* packed, const float* x, int64_t rows, float* y,
                                  void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (rows < 0) return fail(SWENSE_ERR_ARG, "rows must be >= 0");
  if (rows == 0) return SWENSE_OK;
  if (!packed || !x || !y) return fail(SWENSE_ERR_ARG, "NULL argument");
  if (reinterpret_cast<uintptr_t>(packed) & 15) return fail(SWENSE_ERR_ARG, "packed must be 16-byte aligned");
  const int64_t tiles = (rows + 63) / 64;
  const unsigned blocks = unsigned(std::min<int64_t>(tiles, 152 * 16));
  k_mlp_forward<<<blocks, 128, 0, stream>>>(static_cast<const Packed*>(packed), x, rows, y);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

namespace {

// Workspace layout of one training step for batch B (after `base` bytes the caller keeps).
struct StepWs {
  float *part, *loss_part;
  int32_t* idx;
  unsigned blocks;
};
size_t al256(size_t b) { return (b + 255) & ~size_t(255); }
unsigned step_blocks(int B) { return unsigned(std::min<int64_t>((int64_t(B) + TROWS - 1) / TROWS, 152)); }
size_t step_ws_bytes(int B) {
  const unsigned blocks = step_blocks(B);
  return al256(size_t(blocks) * NPARAM * sizeof(float)) + al256(blocks * sizeof(float)) + al256(size_t(B) * sizeof(int32_t));
}
StepWs step_ws(void* ws, int B) {
  StepWs w{};
  w.blocks = step_blocks(B);
  char* c = static_cast<char*>(ws);
  w.part = reinterpret_cast<float*>(c);
  c += al256(size_t(w.blocks) * NPARAM * sizeof(float));
  w.loss_part = reinterpret_cast<float*>(c);
  c += al256(w.blocks * sizeof(float));
  w.idx = reinterpret_cast<int32_t*>(c);
  return w;
}

// Forward + backward of batch rows `batch`, in a fixed order, then `u`: the gradient and loss into its
// buffers, and the Adam step where it names parameters.
int train_into(const StepWs& w, const void* packed, const float* x, const int32_t* field, const float* target,
               float tscale, const int32_t* batch, int B, UpdateArgs u, cudaStream_t stream) {
  const TrainArgs a{static_cast<const Packed*>(packed), x, field, target, batch, B, w.part, w.loss_part, tscale};
  SWENSE_CUDA_TRY(cudaFuncSetAttribute((const void*)k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(sizeof(TrainSmem))));
  k_mlp_train<<<w.blocks, TTHR, sizeof(TrainSmem), stream>>>(a);
  SWENSE_CUDA_TRY(cudaGetLastError());
  u.part = w.part;
  u.nparts = int(w.blocks);
  u.loss_part = w.loss_part;
  k_mlp_update<<<(NPARAM + 31) / 32, 32 * UPD_RUNS, 0, stream>>>(u);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(2);
  return SWENSE_OK;
}

// Adam step (1-based `step`) of params and their packed copy.
UpdateArgs adam_args(float* params, float* adam_m, float* adam_v, void* packed, int64_t step, float lr, float beta1,
                     float beta2, float eps, float* loss) {
  UpdateArgs u{};
  u.loss = loss;
  u.P = params;
  u.m = adam_m;
  u.v = adam_v;
  u.out = static_cast<Packed*>(packed);
  u.lr = lr;
  u.b1 = beta1;
  u.b2 = beta2;
  u.eps = eps;
  u.bc1 = float(1.0 - std::pow(double(beta1), double(step)));
  u.bc2 = float(1.0 - std::pow(double(beta2), double(step)));
  return u;
}

}  // namespace

extern "C" int swense_mlp_train_step(float* params, float* adam_m, float* adam_v, void* packed,
                                     int64_t step, const float* x, const int32_t* field,
                                     const float* target, const int32_t* batch, int32_t B, float lr,
                                     float beta1, float beta2, float eps, float* loss, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (!params || !adam_m || !adam_v || !packed || !x || !field || !target || !batch)
    return fail(SWENSE_ERR_ARG, "NULL argument");
  if (B < 1 || B > (1 << 24)) return fail(SWENSE_ERR_ARG, "batch size must be in [1, 2^24]");
  if (step < 1) return fail(SWENSE_ERR_ARG, "step is 1-based");
  if (!(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0))
    return fail(SWENSE_ERR_ARG, "bad Adam hyper-parameters");
  void* ws = nullptr;
  int st = workspace(step_ws_bytes(B), stream, &ws);
  if (st) return st;
  return train_into(step_ws(ws, B), packed, x, field, target, 1.f, batch, B,
                    adam_args(params, adam_m, adam_v, packed, step, lr, beta1, beta2, eps, loss), stream);
}

extern "C" int swense_mlp_grad(const void* packed, const float* x, const int32_t* field,
                               const float* target, const int32_t* batch, int32_t B, float* grad,
                               float* loss, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (!packed || !x || !field || !target || !batch || !grad) return fail(SWENSE_ERR_ARG, "NULL argument");
  if (B < 1 || B > (1 << 24)) return fail(SWENSE_ERR_ARG, "batch size must be in [1, 2^24]");
  void* ws = nullptr;
  int st = workspace(step_ws_bytes(B), stream, &ws);
  if (st) return st;
  UpdateArgs u{};
  u.grad = grad;
  u.loss = loss;
  return train_into(step_ws(ws, B), packed, x, field, target, 1.f, batch, B, u, stream);
}

extern "C" int swense_mlp_targets(const float* exact_u, const float* exact_v, const float* exact_w,
                                  const float* exact_phit, const float* lagrange, const float* scale,
                                  int64_t np, float* target, int32_t* field, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (np < 0) return fail(SWENSE_ERR_ARG, "np must be >= 0");
  if (np == 0) return SWENSE_OK;
  if (!exact_u || !exact_v || !exact_w || !exact_phit || !lagrange || !scale || !target || !field)
    return fail(SWENSE_ERR_ARG, "NULL argument");
  k_mlp_targets<<<unsigned((4 * np + 255) / 256), 256, 0, stream>>>(exact_u, exact_v, exact_w, exact_phit,
                                                                   lagrange, scale, np, target, field);
  SWENSE_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return SWENSE_OK;
}

extern "C" int swense_mlp_train(swense_mlp* mlp, const float* x, const int32_t* field, const float* target,
                                int64_t n_rows, int32_t steps, int32_t B, float lr, int64_t schedule_steps,
                                float beta1, float beta2, float eps, float* losses, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (!mlp || !mlp->params || !mlp->adam_m || !mlp->adam_v || !mlp->packed || !x || !field || !target)
    return fail(SWENSE_ERR_ARG, "NULL argument");
  if (n_rows < 1 || n_rows > (int64_t(1) << 31)) return fail(SWENSE_ERR_ARG, "n_rows must be in [1, 2^31]");
  if (steps < 0 || B < 1 || B > (1 << 24)) return fail(SWENSE_ERR_ARG, "steps >= 0, batch in [1, 2^24]");
  if (!(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0) || mlp->step < 0)
    return fail(SWENSE_ERR_ARG, "bad Adam hyper-parameters or step");
  if (reinterpret_cast<uintptr_t>(mlp->packed) & 15) return fail(SWENSE_ERR_ARG, "packed must be 16-byte aligned");
  void* ws = nullptr;
  int st = workspace(step_ws_bytes(B) + 256, stream, &ws);
  if (st) return st;
  const StepWs w = step_ws(ws, B);
  if (!(mlp->out_scale > 0)) {
    // the output scale: RMS of the raw targets (the network then trains on O(1) values)
    double* acc = reinterpret_cast<double*>(static_cast<char*>(ws) + step_ws_bytes(B));
    SWENSE_CUDA_TRY(cudaMemsetAsync(acc, 0, sizeof(double), stream));
    k_mlp_sumsq<<<unsigned(std::min<int64_t>((n_rows + 255) / 256, 152 * 8)), 256, 0, stream>>>(target, n_rows, acc);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);
    double ss = 0.0;
    SWENSE_CUDA_TRY(cudaMemcpyAsync(&ss, acc, sizeof(double), cudaMemcpyDeviceToHost, stream));
    SWENSE_CUDA_TRY(cudaStreamSynchronize(stream));
    const double rms = std::sqrt(ss / double(n_rows));
    mlp->out_scale = rms > 0 ? float(rms) : 1.f;
    st = swense_mlp_pack(mlp->params, mlp->out_scale, mlp->packed, stream_);
    if (st) return st;
  }
  const float tscale = 1.f / mlp->out_scale;
  for (int32_t i = 0; i < steps; ++i) {
    const int64_t s = mlp->step;                 // steps already taken
    k_mlp_batch<<<(B + 255) / 256, 256, 0, stream>>>(mlp->seed, s, n_rows, B, w.idx);
    SWENSE_CUDA_TRY(cudaGetLastError());
    count_launches(1);
    double lr_s = lr;
    if (schedule_steps > 0)
      lr_s = lr * 0.5 * (1.0 + std::cos(3.14159265358979323846 * double(std::min(s, schedule_steps)) /
                                        double(schedule_steps)));
    st = train_into(w, mlp->packed, x, field, target, tscale, w.idx, B,
                    adam_args(mlp->params, mlp->adam_m, mlp->adam_v, mlp->packed, s + 1, float(std::max(lr_s, 1e-30)),
                              beta1, beta2, eps, losses ? losses + i : nullptr), stream);
    if (st) return st;
    mlp->step = s + 1;
  }
  return SWENSE_OK;
}

// Checkpoint, little-endian: "SWMLP002", int64 step, uint64 seed, int64 nparam, float64
// out_scale, then params, Adam m, Adam v as float32.
extern "C" int swense_mlp_save(const swense_mlp* mlp, const char* path, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (!mlp || !path || !mlp->params || !mlp->adam_m || !mlp->adam_v) return fail(SWENSE_ERR_ARG, "NULL argument");
  std::vector<float> buf(3 * size_t(NPARAM));
  const float* src[3] = {mlp->params, mlp->adam_m, mlp->adam_v};
  for (int q = 0; q < 3; ++q)
    SWENSE_CUDA_TRY(cudaMemcpyAsync(buf.data() + size_t(q) * NPARAM, src[q], NPARAM * sizeof(float),
                                    cudaMemcpyDeviceToHost, stream));
  SWENSE_CUDA_TRY(cudaStreamSynchronize(stream));
  FILE* f = std::fopen(path, "wb");
  if (!f) return fail(SWENSE_ERR_ARG, std::string("cannot open ") + path + " for writing");
  const int64_t step = mlp->step, np = NPARAM;
  const uint64_t seed = mlp->seed;
  const double os = mlp->out_scale;
  bool ok = std::fwrite("SWMLP002", 1, 8, f) == 8 && std::fwrite(&step, 8, 1, f) == 1 &&
            std::fwrite(&seed, 8, 1, f) == 1 && std::fwrite(&np, 8, 1, f) == 1 && std::fwrite(&os, 8, 1, f) == 1 &&
            std::fwrite(buf.data(), sizeof(float), buf.size(), f) == buf.size();
  ok = (std::fclose(f) == 0) && ok;
  if (!ok) return fail(SWENSE_ERR_ARG, std::string("writing ") + path + " failed");
  return SWENSE_OK;
}

extern "C" int swense_mlp_load(swense_mlp* mlp, const char* path, void* stream_) {
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (!mlp || !path || !mlp->params || !mlp->adam_m || !mlp->adam_v || !mlp->packed)
    return fail(SWENSE_ERR_ARG, "NULL argument");
  FILE* f = std::fopen(path, "rb");
  if (!f) return fail(SWENSE_ERR_ARG, std::string("cannot open ") + path);
  char magic[8];
  int64_t step = 0, np = 0;
  uint64_t seed = 0;
  double os = 0.0;
  std::vector<float> buf(3 * size_t(NPARAM));
  bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "SWMLP002", 8) == 0 &&
            std::fread(&step, 8, 1, f) == 1 && std::fread(&seed, 8, 1, f) == 1 && std::fread(&np, 8, 1, f) == 1 &&
            np == NPARAM && std::fread(&os, 8, 1, f) == 1 &&
            std::fread(buf.data(), sizeof(float), buf.size(), f) == buf.size();
  std::fclose(f);
  if (!ok || step < 0 || !(os > 0) || !std::isfinite(os))
    return fail(SWENSE_ERR_ARG, std::string(path) + " is not a swense MLP checkpoint (SWMLP002)");
  float* dst[3] = {mlp->params, mlp->adam_m, mlp->adam_v};
  for (int q = 0; q < 3; ++q)
    SWENSE_CUDA_TRY(cudaMemcpyAsync(dst[q], buf.data() + size_t(q) * NPARAM, NPARAM * sizeof(float),
                                    cudaMemcpyHostToDevice, stream));
  mlp->step = step;
  mlp->seed = seed;
  mlp->out_scale = float(os);
  return swense_mlp_pack(mlp->params, mlp->out_scale, mlp->packed, stream_);   // synchronises
}
