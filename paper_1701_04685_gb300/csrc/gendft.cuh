// Small DFTs of 4 to 16, 18, 20, 24 and 32 points in registers, X_k = sum_t v_t w^{kt},
// w = exp(DIR 2 pi i / R), for the two-step passes of any length R1 R2.
// Lengths with coprime factors take the prime-factor map (no twiddles between
// the factors), 9 and 16 the Cooley-Tukey split, 7, 11 and 13 the real-pair sums
//   X_{k}, X_{R-k} = v_0 + sum_t cos(2 pi k t / R) (v_t + v_{R-t})
//                    +- DIR i sum_t sin(2 pi k t / R) (v_t - v_{R-t}),
// a quarter of the multiplications of the direct sum.
#pragma once

#include "gensplit.hpp"
#include "warprow.cuh"

namespace fh {

// cos and sin of 2 pi k / R, k = 1 .. (R - 1) / 2 (indices are compile-time
// constants after unrolling, so the tables become immediates)
template <int R>
__device__ __forceinline__ double odd_cos(int k) {
  if (R == 7) {
    const double c[3] = {0.6234898018587335305, -0.2225209339563144043, -0.9009688679024191262};
    return c[(k - 1) % 3];
  }
  if (R == 11) {
    const double c[5] = {0.8412535328311811688, 0.4154150130018864255, -0.1423148382732851405, -0.6548607339452850641,
                         -0.9594929736144973898};
    return c[(k - 1) % 5];
  }
  const double c[6] = {0.8854560256532098959, 0.5680647467311558024, 0.1205366802553230534, -0.3546048870425356259,
                       -0.7485107481711010987, -0.9709418174260520272};
  return c[(k - 1) % 6];
}
template <int R>
__device__ __forceinline__ double odd_sin(int k) {
  if (R == 7) {
    const double s[3] = {0.7818314824680298087, 0.9749279121818236070, 0.4338837391175581205};
    return s[(k - 1) % 3];
  }
  if (R == 11) {
    const double s[5] = {0.5406408174555975822, 0.9096319953545183715, 0.9898214418809327323, 0.7557495743542582838,
                         0.2817325568414296977};
    return s[(k - 1) % 5];
  }
  const double s[6] = {0.4647231720437685456, 0.8229838658936563945, 0.9927088740980539928, 0.9350162426854148234,
                       0.6631226582407952024, 0.2393156642875577671};
  return s[(k - 1) % 6];
}

template <int R, int DIR, typename T>
__device__ __forceinline__ void dft_odd(cplx<T>* v) {
  constexpr int H = (R - 1) / 2;
  cplx<T> p[H], d[H], x0 = v[0];
  const cplx<T> a = v[0];
#pragma unroll
  for (int t = 0; t < H; ++t) {
    p[t] = cadd(v[t + 1], v[R - 1 - t]);
    d[t] = csub(v[t + 1], v[R - 1 - t]);
    x0 = cadd(x0, p[t]);
  }
  v[0] = x0;
#pragma unroll
  for (int k = 1; k <= H; ++k) {
    cplx<T> m = a, q;
    q.x = q.y = T(0);
#pragma unroll
    for (int t = 1; t <= H; ++t) {
      const int e = (k * t) % R;
      const int f = e <= H ? e : R - e;
      const T c = (T)odd_cos<R>(f);
      const T s = e <= H ? (T)odd_sin<R>(f) : (T)-odd_sin<R>(f);
      m.x = fma(c, p[t - 1].x, m.x);
      m.y = fma(c, p[t - 1].y, m.y);
      q.x = fma(s, d[t - 1].x, q.x);
      q.y = fma(s, d[t - 1].y, q.y);
    }
    const cplx<T> r = mul_i<DIR>(q);
    v[k] = cadd(m, r);
    v[R - k] = csub(m, r);
  }
}

// 9 = 3 x 3: n = 3 n1 + n2, k = k1 + 3 k2
template <int DIR, typename T>
__device__ __forceinline__ void dft9(cplx<T>* v) {
  auto root = [](int e) {   // exp(DIR 2 pi i e / 9), e = 1, 2, 4
    cplx<T> w;
    w.x = e == 1 ? T(0.7660444431189780352) : e == 2 ? T(0.1736481776669303488) : T(-0.9396926207859083841);
    w.y = e == 1 ? T(0.6427876096865393263) : e == 2 ? T(0.9848077530122080594) : T(0.3420201433256687330);
    if (DIR < 0) w.y = -w.y;
    return w;
  };
  cplx<T> y[3][3];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    y[n2][0] = v[n2];
    y[n2][1] = v[3 + n2];
    y[n2][2] = v[6 + n2];
    dft3<DIR, T>(y[n2]);
  }
#pragma unroll
  for (int n2 = 1; n2 < 3; ++n2)
#pragma unroll
    for (int k1 = 1; k1 < 3; ++k1) y[n2][k1] = cmul(y[n2][k1], root(n2 * k1));
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cplx<T> b[3] = {y[0][k1], y[1][k1], y[2][k1]};
    dft3<DIR, T>(b);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = b[k2];
  }
}

template <int R, int DIR, typename T>
__device__ __forceinline__ void dft_n(cplx<T>* v);

// 32 = 4 x 8: n = 8 n1 + n2, k = k1 + 4 k2
template <int DIR, typename T>
__device__ __forceinline__ void dft32(cplx<T>* v) {
  auto root = [](int e) {   // exp(DIR 2 pi i e / 32), 0 <= e <= 21
    const double c[9] = {1.0, 0.9807852804032304491, 0.9238795325112867561, 0.8314696123025452371, 0.7071067811865475244,
                         0.5555702330196022247, 0.3826834323650897717, 0.1950903220161282678, 0.0};
    cplx<T> w;
    const int q = e & 7, s = e >> 3;   // e = 8 s + q: quarter turns
    const T a = (T)c[q], b = (T)c[8 - q];
    w.x = s == 0 ? a : s == 1 ? -b : -a;
    w.y = s == 0 ? b : s == 1 ? a : -b;
    if (DIR < 0) w.y = -w.y;
    return w;
  };
  cplx<T> y[8][4];
#pragma unroll
  for (int n2 = 0; n2 < 8; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) y[n2][n1] = v[8 * n1 + n2];
    dft4<DIR, T>(y[n2]);
  }
#pragma unroll
  for (int n2 = 1; n2 < 8; ++n2)
#pragma unroll
    for (int k1 = 1; k1 < 4; ++k1) y[n2][k1] = cmul(y[n2][k1], root(n2 * k1));
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    cplx<T> a[8];
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2) a[n2] = y[n2][k1];
    dft8<DIR, T>(a);
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) v[k1 + 4 * k2] = a[k2];
  }
}

// R = RA RB, coprime: v[(RB n1 + RA n2) mod R] -> X[k] = Z[k mod RA][k mod RB]
template <int RA, int RB, int DIR, typename T>
__device__ __forceinline__ void dft_pfa(cplx<T>* v) {
  constexpr int R = RA * RB;
  cplx<T> z[RA][RB];
#pragma unroll
  for (int n2 = 0; n2 < RB; ++n2) {
    cplx<T> a[RA];
#pragma unroll
    for (int n1 = 0; n1 < RA; ++n1) a[n1] = v[(RB * n1 + RA * n2) % R];
    dft_n<RA, DIR, T>(a);
#pragma unroll
    for (int k1 = 0; k1 < RA; ++k1) z[k1][n2] = a[k1];
  }
#pragma unroll
  for (int k1 = 0; k1 < RA; ++k1) dft_n<RB, DIR, T>(z[k1]);
#pragma unroll
  for (int k = 0; k < R; ++k) v[k] = z[k % RA][k % RB];
}

template <int R, int DIR, typename T>
__device__ __forceinline__ void dft_n(cplx<T>* v) {
  if constexpr (R == 2) dft2<DIR, T>(v);
  else if constexpr (R == 3) dft3<DIR, T>(v);
  else if constexpr (R == 4) dft4<DIR, T>(v);
  else if constexpr (R == 5) dft5<DIR, T>(v);
  else if constexpr (R == 6) dft_pfa<2, 3, DIR, T>(v);
  else if constexpr (R == 8) dft8<DIR, T>(v);
  else if constexpr (R == 9) dft9<DIR, T>(v);
  else if constexpr (R == 10) dft_pfa<2, 5, DIR, T>(v);
  else if constexpr (R == 12) dft_pfa<4, 3, DIR, T>(v);
  else if constexpr (R == 14) dft_pfa<2, 7, DIR, T>(v);
  else if constexpr (R == 15) dft_pfa<3, 5, DIR, T>(v);
  else if constexpr (R == 16) dft16<DIR, T>(v);
  else if constexpr (R == 18) dft_pfa<2, 9, DIR, T>(v);
  else if constexpr (R == 20) dft_pfa<4, 5, DIR, T>(v);
  else if constexpr (R == 24) dft_pfa<3, 8, DIR, T>(v);
  else if constexpr (R == 32) dft32<DIR, T>(v);
  else dft_odd<R, DIR, T>(v);
}

// f(integral_constant R) for a run-time radix, up to RM (the branch is uniform in a block)
template <int R> struct RadixC { static constexpr int value = R; };
template <int RM, typename F>
__device__ __forceinline__ void with_radix(int r, F f) {
  if constexpr (RM > 16) {
    switch (r) {
      case 18: f(RadixC<18>{}); return;
      case 20: f(RadixC<20>{}); return;
      case 24: f(RadixC<24>{}); return;
      case 32: f(RadixC<32>{}); return;
      default: break;
    }
  }
  switch (r) {
    case 4: f(RadixC<4>{}); break;
    case 5: f(RadixC<5>{}); break;
    case 6: f(RadixC<6>{}); break;
    case 7: f(RadixC<7>{}); break;
    case 8: f(RadixC<8>{}); break;
    case 9: f(RadixC<9>{}); break;
    case 10: f(RadixC<10>{}); break;
    case 11: f(RadixC<11>{}); break;
    case 12: f(RadixC<12>{}); break;
    case 13: f(RadixC<13>{}); break;
    case 14: f(RadixC<14>{}); break;
    case 15: f(RadixC<15>{}); break;
    default: f(RadixC<16>{}); break;
  }
}

}  // namespace fh
