// Spectral kernels of the network: truncated DFTs along y and x and the mixing
// of the channels per mode.  The z transforms are part of the row kernels
// (fno_rows.cuh).  Spectral data is channels-last, so that a warp's accesses are
// contiguous over the channels:
//   Yz [b][x][y][2m][W]      real rows k < m and imaginary rows m + k
//   Yy [b][x][a][kz][W]      complex; a = 0 .. 2m-1 stands for ky = a or a - 2m
//   vh [b][ax][ay][kz][W]    complex
// A transform of length N to or from the frequencies |k| <= m folds its real
// axis: with E = Y[p] + Y[N-p] and O = Y[p] - Y[N-p],
//   X[+-k] = sum_p E cos(2 pi k p / N) -+ i sum_p O sin(2 pi k p / N),
// so both signs of k and both halves of the axis share their products (a quarter
// of the multiplications of the direct sum); the inverse folds the frequencies
// the same way.  A thread keeps four magnitudes |k| (or four points p) in
// registers: two 8-byte loads of the data and four broadcast table entries for
// 16 multiply-adds.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fno_rows.cuh"

namespace fhspec {

using fhrow::UDiv;
using fhrow::udiv;

constexpr int kSpecThreads = 256;

// divisors of the index arithmetic (a runtime division costs more than the
// multiply-adds of an element): channels, folded axis, magnitudes in fours,
// points in fours, m + 1, 2m, and W W / 4 or W W elements of a mixing matrix
struct SpecDiv {
  UDiv W, np, ngrp, npg, m1, m2, mm1, WW, WV;
};

// channels-last sums of one column: E, O [p][W] for p = 0 .. N/2, magnitudes k0 .. k0 + 3
// (those above m are computed and dropped); put(a, value) receives index a of +k and -k
template <typename Put>
__device__ __forceinline__ void fold_dft(const float2* E, const float2* O, const float2* tw, int N, int m, int W, int k0,
                                         Put put) {
  float2 P[4] = {}, Q[4] = {};
  int t[4] = {0, 0, 0, 0};
  const int np = N / 2 + 1;
  for (int p = 0; p < np; ++p) {
    const float2 e = E[p * W], o = O[p * W];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 w = tw[t[j]];   // (cos, -sin)
      P[j].x = fmaf(e.x, w.x, P[j].x);
      P[j].y = fmaf(e.y, w.x, P[j].y);
      Q[j].x = fmaf(o.x, w.y, Q[j].x);   // -sum O sin
      Q[j].y = fmaf(o.y, w.y, Q[j].y);
      t[j] += k0 + j;
      if (t[j] >= N) t[j] -= N;
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int k = k0 + j;
    if (k > m) break;
    // X[+k] = P - i sum O sin = P + i Q,  X[-k] = P - i Q
    if (k < m) put(k, make_float2(P[j].x - Q[j].y, P[j].y + Q[j].x));
    if (k > 0) put(2 * m - k, make_float2(P[j].x + Q[j].y, P[j].y - Q[j].x));
  }
}

// the inverse: C [a][W] with the frequencies folded in place (fold_modes); points
// p0 .. p0 + 3 and their mirrors; put(point, value)
template <typename Put>
__device__ __forceinline__ void fold_idft(const float2* C, const float2* tw, int N, int m, int W, int p0, Put put) {
  float2 P[4], Q[4] = {};
  int t[4];
  const float2 c0 = C[0];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    P[j] = c0;
    t[j] = p0 + j;
    if (t[j] >= N) t[j] -= N;
  }
  int step[4] = {t[0], t[1], t[2], t[3]};
  for (int k = 1; k <= m; ++k) {
    float2 s = C[k * W], d;
    if (k < m) d = C[(2 * m - k) * W];
    else d = make_float2(-s.x, -s.y);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 w = tw[t[j]];   // (cos, -sin)
      P[j].x = fmaf(s.x, w.x, P[j].x);
      P[j].y = fmaf(s.y, w.x, P[j].y);
      Q[j].x = fmaf(d.x, w.y, Q[j].x);   // -sum D sin
      Q[j].y = fmaf(d.y, w.y, Q[j].y);
      t[j] += step[j];
      if (t[j] >= N) t[j] -= N;
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int p = p0 + j;
    if (p > N / 2) break;
    // out[p] = P + i sum D sin = P - i Q,  out[N - p] = P + i Q
    put(p, make_float2(P[j].x + Q[j].y, P[j].y - Q[j].x));
    if (p > 0 && 2 * p != N) put(N - p, make_float2(P[j].x - Q[j].y, P[j].y + Q[j].x));
  }
}

// frequencies +k and -k (0 < k < m) replaced by their sum (at k) and difference (at 2m - k)
__device__ __forceinline__ void fold_pair(float2& a, float2& b) {
  const float2 s = make_float2(a.x + b.x, a.y + b.y), d = make_float2(a.x - b.x, a.y - b.y);
  a = s;
  b = d;
}

// DFT along y: block (b, x, group of KB kz), Yz -> Yy
__global__ void __launch_bounds__(kSpecThreads) k_dft_y(int N, int m, int W, int KB, SpecDiv dv, const float* __restrict__ Yz,
                                                        float2* __restrict__ Yy, const float2* __restrict__ twg) {
  extern __shared__ __align__(16) float2 sc[];
  const int np = N / 2 + 1, m2 = 2 * m;
  float2* tw = sc;                 // N
  float2* E = tw + N;              // [kb][np][W]
  float2* O = E + KB * np * W;
  const int ng = (m + KB - 1) / KB;
  const int bx = blockIdx.x / ng;
  const int kz0 = (blockIdx.x % ng) * KB;
  const int kb = min(KB, m - kz0);
  for (int i = threadIdx.x; i < N; i += kSpecThreads) tw[i] = twg[i];
  const float* src = Yz + (size_t)bx * N * m2 * W + (size_t)kz0 * W;
  for (int i = threadIdx.x; i < kb * np * W; i += kSpecThreads) {
    const int q = udiv(i, dv.W), c = i - q * W, k = udiv(q, dv.np), p = q - k * np;
    const float* r = src + (p * m2 + k) * W + c;
    float2 a = make_float2(r[0], r[m * W]), b = make_float2(0.f, 0.f);
    if (p > 0 && 2 * p != N) {
      const float* s = src + ((N - p) * m2 + k) * W + c;
      b = make_float2(s[0], s[m * W]);
      fold_pair(a, b);
    }
    E[i] = a;
    O[i] = b;
  }
  __syncthreads();
  const int ngrp = m / 4 + 1;   // magnitudes 0 .. m in fours
  for (int i = threadIdx.x; i < kb * ngrp * W; i += kSpecThreads) {
    const int q = udiv(i, dv.W), c = i - q * W, k = udiv(q, dv.ngrp), gk = q - k * ngrp;
    float2* dst = Yy + ((size_t)bx * m2 * m + kz0 + k) * W + c;
    fold_dft(E + k * np * W + c, O + k * np * W + c, tw, N, m, W, 4 * gk, [&](int a, float2 v) { dst[a * m * W] = v; });
  }
}

// inverse DFT along y: block (b, x, group of KB kz), Yy -> Yz rows scaled by
// scale (times 2 for kz > 0 when wz)
__global__ void __launch_bounds__(kSpecThreads) k_idft_y(int N, int m, int W, int KB, SpecDiv dv,
                                                         const float2* __restrict__ Yy, float* __restrict__ Yz,
                                                         const float2* __restrict__ twg, float scale, int wz) {
  extern __shared__ __align__(16) float2 sc[];
  const int np = N / 2 + 1, m2 = 2 * m;
  float2* tw = sc;                 // N
  float2* C = tw + N;              // [kb][a][W]
  const int ng = (m + KB - 1) / KB;
  const int bx = blockIdx.x / ng;
  const int kz0 = (blockIdx.x % ng) * KB;
  const int kb = min(KB, m - kz0);
  for (int i = threadIdx.x; i < N; i += kSpecThreads) tw[i] = twg[i];
  const float2* src = Yy + ((size_t)bx * m2 * m + kz0) * W;
  for (int i = threadIdx.x; i < kb * (m + 1) * W; i += kSpecThreads) {
    const int q = udiv(i, dv.W), c = i - q * W, k = udiv(q, dv.m1), a = q - k * (m + 1);
    const float s = scale * ((wz && kz0 + k > 0) ? 2.f : 1.f);
    float2 v = src[(a * m + k) * W + c];
    v.x *= s;
    v.y *= s;
    if (a > 0 && a < m) {
      float2 w = src[((m2 - a) * m + k) * W + c];
      w.x *= s;
      w.y *= s;
      fold_pair(v, w);
      C[(k * m2 + m2 - a) * W + c] = w;
    }
    C[(k * m2 + a) * W + c] = v;
  }
  __syncthreads();
  const int npg = (np + 3) / 4;
  float* dst0 = Yz + (size_t)bx * N * m2 * W + (size_t)kz0 * W;
  for (int i = threadIdx.x; i < kb * npg * W; i += kSpecThreads) {
    const int q = udiv(i, dv.W), c = i - q * W, k = udiv(q, dv.npg), g = q - k * npg;
    float* dst = dst0 + k * W + c;
    fold_idft(C + k * m2 * W + c, tw, N, m, W, 4 * g, [&](int p, float2 v) {
      dst[p * m2 * W] = v.x;
      dst[(p * m2 + m) * W] = v.y;
    });
  }
}

// DFT along x, channel mixing and inverse DFT along x, in place on Yy: block
// (ay, kz) owns these columns of every sample.  Samples go through in chunks of
// BC; the block's 2m matrices R [o][i] (BF16 pairs) are staged RS at a time.
//   forward  (BACK = false): x = DFT, stored to vh; c[o] = sum_i R[o][i] x[i]
//   backward (BACK = true):  g = scale w(kz) DFT; gin[i] = sum_o conj(R[o][i]) g[o];
//                            gR[o][i] += sum_b g[b][o] conj(vh[b][i])
// Fusing the three steps leaves one read and one write of the columns and one
// read of R: bound by R's 4 W^2 bytes per mode (28 MB a layer at W = 32, m = 12).
// 64^3, one sample: 22 us where the separate x transforms and the mixing took 95;
// four samples forward and backward: 50 and 87 us (243 and 241).
template <bool BACK>
__global__ void __launch_bounds__(kSpecThreads) k_mix_x(int N, int m, int W, int B, int BC, int RS, SpecDiv dv,
                                                        const __nv_bfloat162* __restrict__ R, float2* __restrict__ Yy,
                                                        float2* __restrict__ vh, float2* __restrict__ gR,
                                                        const float2* __restrict__ twg, float scale) {
  extern __shared__ __align__(16) float2 sc[];
  const int np = N / 2 + 1, m2 = 2 * m, NM = m2 * m2 * m;
  float2* tw = sc;                          // N
  float2* EO = tw + N;                      // [bc][2][np][W]: folded columns, later the mixed coefficients [bc][ax][W]
  float2* xs = EO + BC * 2 * np * W;        // [bc][ax][W]
  float2* xv = xs + BC * m2 * W;            // BACK: vh [bc][ax][W]
  __nv_bfloat162* Rs = reinterpret_cast<__nv_bfloat162*>(xv + (BACK ? BC * m2 * W : 0));   // [rs][o][W + 1]
  const int ay = blockIdx.x / m, kz = blockIdx.x - ay * m;
  const int tid = threadIdx.x;
  const int mode_ax = m2 * m, mode0 = ay * m + kz;   // mode of ax: mode0 + ax mode_ax
  const int WW = W * W;
  for (int i = tid; i < N; i += kSpecThreads) tw[i] = twg[i];
  for (int b0 = 0; b0 < B; b0 += BC) {
    const int bc = min(BC, B - b0);
    float2* col0 = Yy + ((size_t)b0 * N * mode_ax + mode0) * W;   // sample b0, x = 0
    const int xstep = mode_ax * W;
    __syncthreads();
    for (int i = tid; i < bc * np * W; i += kSpecThreads) {
      const int q = udiv(i, dv.W), c = i - q * W, b = udiv(q, dv.np), p = q - b * np;
      const float2* col = col0 + (size_t)b * N * xstep + c;
      float2 e = col[p * xstep], o = make_float2(0.f, 0.f);
      if (p > 0 && 2 * p != N) {
        o = col[(N - p) * xstep];
        fold_pair(e, o);
      }
      EO[(b * 2 * np + p) * W + c] = e;
      EO[((b * 2 + 1) * np + p) * W + c] = o;
    }
    if (BACK)
      for (int i = tid; i < bc * m2 * W; i += kSpecThreads) {
        const int q = udiv(i, dv.W), c = i - q * W, b = udiv(q, dv.m2), ax = q - b * m2;
        xv[i] = vh[((size_t)(b0 + b) * NM + mode0 + ax * mode_ax) * W + c];
      }
    __syncthreads();
    const int ngrp = m / 4 + 1;
    for (int i = tid; i < bc * ngrp * W; i += kSpecThreads) {
      const int q = udiv(i, dv.W), c = i - q * W, b = udiv(q, dv.ngrp), gk = q - b * ngrp;
      const float2* E = EO + b * 2 * np * W + c;
      const float s = (BACK && kz > 0) ? 2.f * scale : scale;
      float2* vhb = vh + ((size_t)(b0 + b) * NM + mode0) * W + c;
      fold_dft(E, E + np * W, tw, N, m, W, 4 * gk, [&](int a, float2 v) {
        if (BACK) {
          v.x *= s;
          v.y *= s;
        } else {
          vhb[(size_t)a * mode_ax * W] = v;
        }
        xs[(b * m2 + a) * W + c] = v;
      });
    }
    float2* cs = EO;   // the columns are done with
    for (int a0 = 0; a0 < m2; a0 += RS) {
      const int na = min(RS, m2 - a0);
      __syncthreads();
      if ((W & 3) == 0) {   // 16-byte reads, four entries of one row each
        const int wv = W >> 2, per = WW >> 2;
        for (int i = tid; i < na * per; i += kSpecThreads) {
          const int a = udiv(i, dv.WV), rem = i - a * per, o = udiv(4 * rem, dv.W), ii = 4 * (rem - o * wv);
          const uint4 v = *reinterpret_cast<const uint4*>(R + (size_t)(mode0 + (a0 + a) * mode_ax) * WW + 4 * rem);
          unsigned* d = reinterpret_cast<unsigned*>(Rs + (a * W + o) * (W + 1) + ii);
          d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
        }
      } else {
        for (int i = tid; i < na * WW; i += kSpecThreads) {
          const int a = udiv(i, dv.WW), rem = i - a * WW, o = udiv(rem, dv.W), ii = rem - o * W;
          Rs[(a * W + o) * (W + 1) + ii] = R[(size_t)(mode0 + (a0 + a) * mode_ax) * WW + rem];
        }
      }
      __syncthreads();
      // task (ax, output channel), the chunk's samples two at a time on the same matrix entries
      for (int i = tid; i < na * W; i += kSpecThreads) {
        const int a = udiv(i, dv.W), o = i - a * W;
        const __nv_bfloat162* r = Rs + a * W * (W + 1) + (BACK ? o : o * (W + 1));
        const int rstep = BACK ? W + 1 : 1;
        for (int b = 0; b < bc; b += 2) {
          const float2* x = xs + (b * m2 + a0 + a) * W;
          const float2* x2 = x + (b + 1 < bc ? m2 * W : 0);
          float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll 4
          for (int j = 0; j < W; ++j) {
            const float2 rv = __bfloat1622float2(r[j * rstep]);
            const float ry = BACK ? -rv.y : rv.y;
            const float2 v = x[j], w = x2[j];
            s0.x = fmaf(rv.x, v.x, fmaf(-ry, v.y, s0.x));
            s0.y = fmaf(rv.x, v.y, fmaf(ry, v.x, s0.y));
            s1.x = fmaf(rv.x, w.x, fmaf(-ry, w.y, s1.x));
            s1.y = fmaf(rv.x, w.y, fmaf(ry, w.x, s1.y));
          }
          cs[(b * m2 + a0 + a) * W + o] = s0;
          if (b + 1 < bc) cs[((b + 1) * m2 + a0 + a) * W + o] = s1;
        }
      }
      if (BACK) {
        // an entry's read, sum and write wait for memory: two entries of a row in one
        // 16-byte access and four accesses in flight a thread (one 8-byte access at a
        // time: 140 us a layer of 64^3, four samples; 87 us so)
        constexpr int U = 4;
        auto outer = [&](int a, int o, int ii, int b) {   // g conj(x)
          const float2 gg = xs[(b * m2 + a0 + a) * W + o], xx = xv[(b * m2 + a0 + a) * W + ii];
          return make_float2(gg.x * xx.x + gg.y * xx.y, gg.y * xx.x - gg.x * xx.y);
        };
        if ((W & 1) == 0) {
          const int n2 = (na * WW) >> 1;
          for (int i0 = tid; i0 < n2; i0 += U * kSpecThreads) {
            float4 acc[U];
            float4* t[U];
            int a[U], o[U], ii[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int i = min(i0 + u * kSpecThreads, n2 - 1);
              a[u] = udiv(2 * i, dv.WW);
              const int rem = 2 * i - a[u] * WW;
              o[u] = udiv(rem, dv.W);
              ii[u] = rem - o[u] * W;
              t[u] = reinterpret_cast<float4*>(gR + (size_t)(mode0 + (a0 + a[u]) * mode_ax) * WW + rem);
              acc[u] = i0 + u * kSpecThreads < n2 ? *t[u] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              float2 s0 = make_float2(0.f, 0.f), s1 = s0;
              for (int b = 0; b < bc; ++b) {
                const float2 p = outer(a[u], o[u], ii[u], b), q = outer(a[u], o[u], ii[u] + 1, b);
                s0.x += p.x;
                s0.y += p.y;
                s1.x += q.x;
                s1.y += q.y;
              }
              if (i0 + u * kSpecThreads < n2)
                *t[u] = make_float4(acc[u].x + s0.x, acc[u].y + s0.y, acc[u].z + s1.x, acc[u].w + s1.y);
            }
          }
        } else {
          for (int i = tid; i < na * WW; i += kSpecThreads) {
            const int a = udiv(i, dv.WW), rem = i - a * WW, o = udiv(rem, dv.W), ii = rem - o * W;
            float2* t = gR + (size_t)(mode0 + (a0 + a) * mode_ax) * WW + rem;
            const float2 acc = *t;
            float2 sum = make_float2(0.f, 0.f);
            for (int b = 0; b < bc; ++b) {
              const float2 p = outer(a, o, ii, b);
              sum.x += p.x;
              sum.y += p.y;
            }
            *t = make_float2(acc.x + sum.x, acc.y + sum.y);
          }
        }
      }
    }
    __syncthreads();
    for (int i = tid; i < bc * (m - 1) * W; i += kSpecThreads) {
      const int q = udiv(i, dv.W), c = i - q * W, b = udiv(q, dv.mm1), k = 1 + q - b * (m - 1);
      fold_pair(cs[(b * m2 + k) * W + c], cs[(b * m2 + m2 - k) * W + c]);
    }
    __syncthreads();
    const int npg = (np + 3) / 4;
    for (int i = tid; i < bc * npg * W; i += kSpecThreads) {
      const int q = udiv(i, dv.W), c = i - q * W, b = udiv(q, dv.npg), g = q - b * npg;
      float2* col = col0 + (size_t)b * N * xstep + c;
      fold_idft(cs + b * m2 * W + c, tw, N, m, W, 4 * g, [&](int p, float2 v) { col[p * xstep] = v; });
    }
  }
}

}  // namespace fhspec
