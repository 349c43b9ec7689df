// Row kernels of the network: everything that happens at one grid row (b, x, y)
// of N points z and all channels, in one pass over the activations.
//
//   out[o][z] = epi( sum_c A[o][c] in[c][z] + bias[o] + sum_k Iy[k][o] T[k][z] )
//   Yz[k][o]  = sum_z T[k][z] out[o][z]
//   y[q][z]   = sum_o Q[q][o] out[o][z] + qb[q]
//
// A is the 1 x 1 layer (the lift P, a hidden W_l, or in the backward pass a
// transposed one), Iy the row's spectral coefficients after the inverse
// transforms along x and y (fno_spec.cuh), T the real table of the truncated
// z-DFT (rows k < m: cos(2 pi k z / N), rows m + k: -sin), epi the identity, the
// GELU or the product with gelu'(u).  The z-transform of the next spectral layer
// (Yz) and the projection (y, in training with the mean-squared error and its
// gradient) are taken from the row while it is in shared memory.
//
// A hidden layer reads v once and writes u (training only) and v' once; the
// former chain of kernels (DFT planes, pointwise, inverse DFT planes) moved the
// activations seven times and was bound by scalar shared-memory loads.  Each
// thread holds an 8 x 4 tile of (o, z): per input channel two broadcast and one
// row 16-byte shared-memory loads for 32 multiply-adds, so the FP32 pipe and
// not shared memory bounds it.  Row stride N + 4 (rounded up to 4): the tiles'
// 16-byte accesses and the dot products along z are free of bank conflicts.
// A hidden layer of the 64^3 network (32 channels, 12 modes): 82 us for one
// sample, 291 us for four (445 MB of HBM traffic; FP32 pipe 33 % busy, issue
// 53 %, the rest is the wait for a tile's loads); the kernels it replaces took
// 239 us and 850 us.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace fhrow {

constexpr int kRowThreads = 256;

// q = n / d by multiplication, exact for n < 2^16 and d < 2^16
struct UDiv {
  unsigned d, mul;
};
inline UDiv make_udiv(unsigned d) { return {d, d > 1 ? (unsigned)((0x100000000ull + d - 1) / d) : 0u}; }
__device__ __forceinline__ unsigned udiv(unsigned n, UDiv u) { return u.d > 1 ? __umulhi(n, u.mul) : n; }

struct RowArgs {
  int N, N3, N2;       // points per row, per sample; rows per sample
  int N4, NS;          // N rounded up to 4, row stride in shared memory
  int W, WP, Cin;      // output channels (WP: rounded up to 8), input channels
  int m2, m2p;         // 2 m spectral rows (0: none), rounded up to 4
  int nrows, rpb;      // rows in all, rows per block
  int vec;             // rows and pointers allow 16-byte accesses
  int kc;              // rows of the activation tile, max(Cin, W)
  UDiv dNq, dCin, dTask, dOg, dCg, dKg, dQt, dQg;
  const float* in;     // [b][Cin][N3]
  const void* A;       // [W][Cin], or [Cin][W] when a_trans
  int a_bf16, a_trans;
  const float* bias;   // [W] or null
  const float* Iy;     // [row][m2][W] or null
  const float* T;      // [m2][N]
  const float* u_in;   // gelu' argument [b][W][N3] (EPI 2)
  float* u_out;        // pre-activation (EPI 1, 3) or null
  float* out;          // [b][W][N3] or null
  float* Yz;           // [row][m2][W] or null
  // projection
  const float* Q;      // [cout][W] or null
  const float* qb;
  int cout, QP;
  float* y;            // [b][cout][N3] (EPI 1)
  const float* target; // [b][cout][N3] (EPI 3)
  float* gy;           // 2 (y - target) inv_count (EPI 3)
  double* part;        // one block sum of (y - target)^2 per block (EPI 3)
  float inv_count;
};

__host__ inline size_t row_smem_floats(const RowArgs& a) {
  size_t n = 0;
  if (a.m2) n += (size_t)a.m2p * a.NS;
  n += (size_t)a.Cin * a.WP;
  if (a.Q) n += (size_t)a.W * a.QP;
  n += (size_t)a.rpb * a.kc * a.NS;
  if (a.Iy) n += (size_t)a.rpb * a.m2 * a.WP;
  return n;
}

__device__ __forceinline__ float row_gelu(float u) { return 0.5f * u * (1.f + erff(u * 0.70710678118654752f)); }
__device__ __forceinline__ float row_dgelu(float u) {
  return 0.5f * (1.f + erff(u * 0.70710678118654752f)) + u * 0.39894228040143268f * expf(-0.5f * u * u);
}

// four consecutive values p[0..3] of a row, n of them inside it
__device__ __forceinline__ float4 load4(const float* p, int n, int vec) {
  if (vec) return *reinterpret_cast<const float4*>(p);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (n > 0) v.x = p[0];
  if (n > 1) v.y = p[1];
  if (n > 2) v.z = p[2];
  if (n > 3) v.w = p[3];
  return v;
}
__device__ __forceinline__ void store4(float* p, float4 v, int n, int vec) {
  if (vec) {
    *reinterpret_cast<float4*>(p) = v;
    return;
  }
  if (n > 0) p[0] = v.x;
  if (n > 1) p[1] = v.y;
  if (n > 2) p[2] = v.z;
  if (n > 3) p[3] = v.w;
}

// acc[8][4] += a[8] x b[4]
__device__ __forceinline__ void outer84(float (&acc)[8][4], const float4 a0, const float4 a1, const float4 b) {
  const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    acc[i][0] = fmaf(a[i], b.x, acc[i][0]);
    acc[i][1] = fmaf(a[i], b.y, acc[i][1]);
    acc[i][2] = fmaf(a[i], b.z, acc[i][2]);
    acc[i][3] = fmaf(a[i], b.w, acc[i][3]);
  }
}

// e^2 to the float pair (hi, lo) (TwoSum / TwoProduct: an FP64 multiply-add per element
// is a large part of the last layer's time)
__device__ __forceinline__ void add_square(float e, float& hi, float& lo) {
  const float pr = e * e, er = fmaf(e, e, -pr);
  const float hs = hi + pr, bp = hs - hi;
  lo += ((hi - (hs - bp)) + (pr - bp)) + er;
  hi = hs;
}
// the pair of at most 32 squares holds their sum: no square has left FP32's range (the
// sum would be infinite or NaN), and those whose rounding errors have (below 2^-102) are
// less than 2^-37 of it
__device__ __forceinline__ bool pair_holds(float hi) { return hi >= 0x1p-60f && hi < 0x1p126f; }

// EPI 0: the identity, 1: the GELU (with the projection y where Q is given), 2: the
// product with gelu'(u), 3: the GELU with the projection, the squared errors and their
// gradient (training's last layer)
template <int EPI>
__global__ void __launch_bounds__(kRowThreads, 2) k_rows(const RowArgs a) {
  extern __shared__ __align__(16) float smf[];
  const int tid = threadIdx.x;
  float* sT = smf;                                   // [m2p][NS]
  float* sW = sT + (a.m2 ? a.m2p * a.NS : 0);        // [Cin][WP]
  float* sQ = sW + a.Cin * a.WP;                     // [W][QP]
  float* sV = sQ + (a.Q ? a.W * a.QP : 0);           // [rpb][kc][NS]
  float* sI = sV + a.rpb * a.kc * a.NS;              // [rpb][m2][WP]
  const int nz4 = a.N4 >> 2;
  if (a.m2)
    for (int i = tid; i < a.m2p * a.NS; i += kRowThreads) {
      const int k = i / a.NS, z = i - k * a.NS;
      sT[i] = (k < a.m2 && z < a.N) ? a.T[k * a.N + z] : 0.f;
    }
  for (int i = tid; i < a.Cin * a.WP; i += kRowThreads) {
    const int c = i / a.WP, o = i - c * a.WP;
    const int j = a.a_trans ? c * a.W + o : o * a.Cin + c;
    float v = 0.f;
    if (o < a.W)
      v = a.a_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(a.A)[j]) : reinterpret_cast<const float*>(a.A)[j];
    sW[i] = v;
  }
  if (a.Q)
    for (int i = tid; i < a.W * a.QP; i += kRowThreads) {
      const int c = i / a.QP, q = i - c * a.QP;
      sQ[i] = q < a.cout ? a.Q[q * a.W + c] : 0.f;
    }
  constexpr bool PROJ = EPI == 1 || EPI == 3, LOSS = EPI == 3;
  double esum = 0.0;   // this thread's squared errors
  const int ntiles = (a.nrows + a.rpb - 1) / a.rpb;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int row0 = tile * a.rpb;
    const int nr = min(a.rpb, a.nrows - row0);
    __syncthreads();   // the last tile's reads are done
    // the rows' input channels and spectral coefficients
    for (int i = tid; i < nr * a.Cin * nz4; i += kRowThreads) {
      const int rc = udiv(i, a.dNq), z = (i - rc * nz4) * 4;
      const int r = udiv(rc, a.dCin), c = rc - r * a.Cin;
      const int row = row0 + r, b = row / a.N2;
      const float* p = a.in + ((size_t)b * a.Cin + c) * a.N3 + (size_t)(row - b * a.N2) * a.N + z;
      *reinterpret_cast<float4*>(sV + (r * a.kc + c) * a.NS + z) = load4(p, a.N - z, a.vec);
    }
    if (a.Iy)
      for (int i = tid; i < nr * a.m2 * a.WP; i += kRowThreads) {
        const int rk = i / a.WP, o = i - rk * a.WP;
        sI[i] = o < a.W ? a.Iy[((size_t)row0 * a.m2 + rk) * a.W + o] : 0.f;
      }
    __syncthreads();
    // task: row r, channels 8 og .. 8 og + 7, points 4 zg .. 4 zg + 3
    const int r = udiv(tid, a.dTask);
    const int rem = tid - r * a.dTask.d;
    const int zg = udiv(rem, a.dOg), og = rem - zg * a.dOg.d;
    const bool on = r < nr;
    const int row = row0 + r, b = row / a.N2;
    const int z = 4 * zg, zn = a.N - z;
    float acc[8][4];
    if (on) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float bi = (a.bias && 8 * og + i < a.W) ? a.bias[8 * og + i] : 0.f;
        acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = bi;
      }
      const float* w = sW + 8 * og;
      const float* v = sV + r * a.kc * a.NS + z;
#pragma unroll 4
      for (int c = 0; c < a.Cin; ++c, w += a.WP, v += a.NS)
        outer84(acc, *reinterpret_cast<const float4*>(w), *reinterpret_cast<const float4*>(w + 4),
                *reinterpret_cast<const float4*>(v));
      if (a.Iy) {
        const float* s = sI + r * a.m2 * a.WP + 8 * og;
        const float* t = sT + z;
#pragma unroll 4
        for (int k = 0; k < a.m2; ++k, s += a.WP, t += a.NS)
          outer84(acc, *reinterpret_cast<const float4*>(s), *reinterpret_cast<const float4*>(s + 4),
                  *reinterpret_cast<const float4*>(t));
      }
      const size_t base = (size_t)b * a.W * a.N3 + (size_t)(row - b * a.N2) * a.N + z;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int o = 8 * og + i;
        if (o >= a.W) break;
        const size_t p = base + (size_t)o * a.N3;
        if (EPI == 1 || EPI == 3) {
          if (a.u_out) store4(a.u_out + p, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]), zn, a.vec);
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = row_gelu(acc[i][j]);
        } else if (EPI == 2) {
          const float4 u = load4(a.u_in + p, zn, a.vec);
          acc[i][0] *= row_dgelu(u.x);
          acc[i][1] *= row_dgelu(u.y);
          acc[i][2] *= row_dgelu(u.z);
          acc[i][3] *= row_dgelu(u.w);
        }
        if (a.out) store4(a.out + p, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]), zn, a.vec);
      }
    }
    if (!a.Yz && !a.Q) continue;
    __syncthreads();   // every thread has read its input rows
    if (on) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (8 * og + i < a.W)
          *reinterpret_cast<float4*>(sV + (r * a.kc + 8 * og + i) * a.NS + z) =
              make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    }
    __syncthreads();
    if (a.Yz) {
      // task: row, channels cg + j (WP / 4), spectral rows kg + j (m2p / 4)
      const int ncg = a.dCg.d, nkg = a.m2p >> 2;
      for (int t = tid; t < nr * ncg * nkg; t += kRowThreads) {
        const int rk = udiv(t, a.dCg), cg = t - rk * ncg;
        const int rr = udiv(rk, a.dKg), kg = rk - rr * nkg;
        float s[4][4] = {};
        const int cb = min(cg, a.W - 1);   // channels beyond W read a row below it (their sums are not stored)
        const float* v = sV + (rr * a.kc + cb) * a.NS;
        const float* tt = sT + kg * a.NS;
        const int ts = nkg * a.NS;
        int vo[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) vo[j] = cg + j * ncg < a.W ? j * ncg * a.NS : 0;
#pragma unroll 1   // unrolled twice, every instance but EPI 2 spills (64^3, width 16, two samples: 530 against 522 us)
        for (int q = 0; q < a.N4; q += 4) {
          float4 x[4], y[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            x[j] = *reinterpret_cast<const float4*>(v + vo[j] + q);
            y[j] = *reinterpret_cast<const float4*>(tt + j * ts + q);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              s[i][j] = fmaf(x[j].x, y[i].x, fmaf(x[j].y, y[i].y, fmaf(x[j].z, y[i].z, fmaf(x[j].w, y[i].w, s[i][j]))));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = kg + i * nkg;
          if (k >= a.m2) continue;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int c = cg + j * ncg;
            if (c < a.W) a.Yz[((size_t)(row0 + rr) * a.m2 + k) * a.W + c] = s[i][j];
          }
        }
      }
    }
    if (PROJ && a.Q) {
      const int nqg = a.QP >> 3;
      for (int t = tid; t < nr * nqg * nz4; t += kRowThreads) {
        const int rr = udiv(t, a.dQt), rm = t - rr * a.dQt.d;
        const int zq = udiv(rm, a.dQg), qg = rm - zq * nqg;
        const int row2 = row0 + rr, b2 = row2 / a.N2, z2 = 4 * zq, zn2 = a.N - z2;
        float s[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float bi = 8 * qg + i < a.cout ? a.qb[8 * qg + i] : 0.f;
          s[i][0] = s[i][1] = s[i][2] = s[i][3] = bi;
        }
        const float* w = sQ + 8 * qg;
        const float* v = sV + rr * a.kc * a.NS + z2;
#pragma unroll 4
        for (int c = 0; c < a.W; ++c, w += a.QP, v += a.NS)
          outer84(s, *reinterpret_cast<const float4*>(w), *reinterpret_cast<const float4*>(w + 4),
                  *reinterpret_cast<const float4*>(v));
        const size_t base = (size_t)b2 * a.cout * a.N3 + (size_t)(row2 - b2 * a.N2) * a.N + z2;
        float ehi = 0.f, elo = 0.f;   // the task's squared errors as a float pair
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int q = 8 * qg + i;
          if (q >= a.cout) break;
          const size_t p = base + (size_t)q * a.N3;
          if (!LOSS) {
            store4(a.y + p, make_float4(s[i][0], s[i][1], s[i][2], s[i][3]), zn2, a.vec);
            continue;
          }
          const float4 tv = load4(a.target + p, zn2, a.vec);
          const float tq[4] = {tv.x, tv.y, tv.z, tv.w};
          float g[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float e = s[i][j] - tq[j];
            g[j] = 2.f * e * a.inv_count;
            s[i][j] = e;
            if (j < zn2) add_square(e, ehi, elo);
          }
          store4(a.gy + p, make_float4(g[0], g[1], g[2], g[3]), zn2, a.vec);
        }
        if (!LOSS) continue;
        if (pair_holds(ehi)) {
          esum += (double)ehi + (double)elo;
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (8 * qg + i < a.cout && j < zn2) esum += (double)s[i][j] * s[i][j];
        }
      }
    }
  }
  if (LOSS) {
    __shared__ double red[kRowThreads / 32];
    double v = esum;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < kRowThreads / 32; ++w) s += red[w];
      a.part[blockIdx.x] = s;
    }
  }
}

// gA[o][c] += sum_{b,p} g[b][o][p] x[b][c][p], gbias[o] += sum g[b][o][p].
// A block takes chunks of 128 voxels, each warp 16 of them with the whole
// 32 x 32 tile of (o, c) in registers (8 x 4 per lane, rows and columns dealt
// round-robin so that the 16-byte reads of four voxels are conflict-free): 12
// shared-memory reads for 128 multiply-adds.  The warps' tiles are summed once
// at the end and added to the gradient (blockIdx.y: the 32 x 32 tile).  Where there are
// at most eight rows (TO) or columns (TC) the tile has eight: the multiply-adds of
// channels that are not there made a training step of a network of one channel a fifth
// longer than a sum per weight did (64^3, 36 outputs, four samples: 0.98 against 0.84 ms; 0.80 so).
constexpr int kWgVox = 128, kWgStride = kWgVox + 4, kWgThreads = 256;
template <int TO, int TC>
__global__ void __launch_bounds__(kWgThreads, 2) k_weight_grad(int total, int N3, int Cin, int Cout, int vec,
                                                               const float* __restrict__ g, const float* __restrict__ x,
                                                               float* __restrict__ gA, float* __restrict__ gbias) {
  __shared__ __align__(16) float gs[TO * kWgStride];
  __shared__ __align__(16) float xs[TC * kWgStride];
  const int ntc = (Cin + TC - 1) / TC;
  const int o0 = (blockIdx.y / ntc) * TO, c0 = (blockIdx.y % ntc) * TC;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int og = lane & 3, cg = lane >> 2;
  float acc[TO / 4][TC / 8] = {};
  float bsum = 0.f;   // thread t: row t / 8, eighth t % 8
  // the next chunk's values wait in registers while the current one is multiplied:
  // warp w loads rows w + 8 i (lane: four voxels)
  float4 ng[TO / 8], nx[TC / 8];
  auto fetch = [&](int t0) {
    int b = 0, p = 0;
    const int t = t0 + 4 * lane;
    if (t < total) {
      b = t / N3;
      p = t - b * N3;
    }
    // row `ch` of [b][C][N3] at this lane's four voxels, zero beyond the last channel or voxel
    auto row = [&](const float* s, int C, int ch) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (vec) {   // N3 a multiple of 4: the four voxels lie in one sample
        if (t < total && ch < C) v = *reinterpret_cast<const float4*>(s + ((size_t)b * C + ch) * N3 + p);
      } else {
        float e[4] = {0.f, 0.f, 0.f, 0.f};
        for (int j = 0; j < 4; ++j)
          if (t + j < total && ch < C) {
            const int bj = (t + j) / N3, pj = t + j - bj * N3;
            e[j] = s[((size_t)bj * C + ch) * N3 + pj];
          }
        v = make_float4(e[0], e[1], e[2], e[3]);
      }
      return v;
    };
#pragma unroll
    for (int i = 0; i < TO / 8; ++i) ng[i] = row(g, Cout, o0 + warp + 8 * i);
#pragma unroll
    for (int i = 0; i < TC / 8; ++i) nx[i] = row(x, Cin, c0 + warp + 8 * i);
  };
  fetch(blockIdx.x * kWgVox);
  for (int t0 = blockIdx.x * kWgVox; t0 < total; t0 += gridDim.x * kWgVox) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TO / 8; ++i) *reinterpret_cast<float4*>(gs + (warp + 8 * i) * kWgStride + 4 * lane) = ng[i];
#pragma unroll
    for (int i = 0; i < TC / 8; ++i) *reinterpret_cast<float4*>(xs + (warp + 8 * i) * kWgStride + 4 * lane) = nx[i];
    __syncthreads();
    if (t0 + (int)gridDim.x * kWgVox < total) fetch(t0 + gridDim.x * kWgVox);
#pragma unroll
    for (int q = 0; q < kWgVox / 8; q += 4) {
      const int p = warp * (kWgVox / 8) + q;
      float4 b[TC / 8];
#pragma unroll
      for (int j = 0; j < TC / 8; ++j) b[j] = *reinterpret_cast<const float4*>(xs + (cg + 8 * j) * kWgStride + p);
#pragma unroll
      for (int i = 0; i < TO / 4; ++i) {
        const float4 a = *reinterpret_cast<const float4*>(gs + (og + 4 * i) * kWgStride + p);
#pragma unroll
        for (int j = 0; j < TC / 8; ++j)
          acc[i][j] = fmaf(a.x, b[j].x, fmaf(a.y, b[j].y, fmaf(a.z, b[j].z, fmaf(a.w, b[j].w, acc[i][j]))));
      }
    }
    if (c0 == 0 && (tid >> 3) < TO) {
      const float* p = gs + (tid >> 3) * kWgStride + (tid & 7) * (kWgVox / 8);
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < kWgVox / 8; q += 4) {
        const float4 v = *reinterpret_cast<const float4*>(p + q);
        s += (v.x + v.y) + (v.z + v.w);
      }
      bsum += s;
    }
  }
  // sum of the warps' tiles, one after the other in the staging buffer
  __syncthreads();
  float* buf = gs;
  for (int w = 0; w < kWgThreads / 32; ++w) {
    if (warp == w) {
#pragma unroll
      for (int i = 0; i < TO / 4; ++i)
#pragma unroll
        for (int j = 0; j < TC / 8; ++j) {
          const int e = (og + 4 * i) * (TC + 1) + cg + 8 * j;
          buf[e] = (w ? buf[e] : 0.f) + acc[i][j];
        }
    }
    __syncthreads();
  }
  for (int i = tid; i < TO * TC; i += kWgThreads) {
    const int o = i / TC, c = i % TC;
    if (o0 + o < Cout && c0 + c < Cin) atomicAdd(&gA[(o0 + o) * Cin + c0 + c], buf[o * (TC + 1) + c]);
  }
  if (c0 == 0) {
    for (int o = 4; o > 0; o >>= 1) bsum += __shfl_down_sync(0xffffffffu, bsum, o, 8);
    if ((tid & 7) == 0 && (tid >> 3) < TO && o0 + (tid >> 3) < Cout) atomicAdd(&gbias[o0 + (tid >> 3)], bsum);
  }
}

}  // namespace fhrow
