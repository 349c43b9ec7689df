// Shared-memory line transforms of the cluster kernel.
//
// warp_two_step (FP32, grids that are no powers of two): lines of N = R1 R2 points
// (gen_split) or of at most 16, by single warps without block barriers.  A CTA holds a
// few lines (96^2 on 16 CTAs: nine of 96 points), and a block-wide stage then lasts
// about 3000 cycles, most of it index arithmetic, twiddle look-up and barrier latency
// with few lanes at work: 6000 cycles for each of an iteration's four transforms, two
// thirds of it.  Here floor(32 / R2) lines share a warp, lane = (line, j2) and then
// (line, k1): 3000 cycles (96^2 18.1 -> 12.4 us an iteration, 60^2 14.9 -> 10.2, 100^2
// 16.5 -> 12.5).  FP64 keeps the block-wide stages: an FP64 instruction takes its
// quarter of the SM 64 cycles, and one warp's two steps use one quarter only (96^2
// 48.7 against 53.6 us).
//
// fft_lines_big, for the other lengths of the general variant: the Stockham stages of
// fft.cuh with every radix from 2 to 16 (gendft.cuh), so that most lengths need two
// stages and none below 4096 more than four (96 = 8 x 12, 192 = 12 x 16, 768 = 8 x 8 x
// 12, where the schedule of 8, 4, 2, 3, ... has three to five), plus the direct stage
// for larger primes.  A called stage costs about 700 cycles more than an inlined one, so
// that clusterplan.cpp sends the lengths that gain less to the staged variant.
//
// A stage deals its butterflies line by line across the lanes: with the odd line
// strides of the cluster layout every access is free of bank conflicts and a warp's
// twiddles are broadcasts (butterfly by butterfly along a line, stages of stride 12
// conflict four ways).  The function is not inlined: its 15 register DFTs appear
// once per direction, the kernel keeps 16 warps per CTA in FP32, and shared memory
// is addressed by byte offsets so that the accesses stay shared-memory instructions.
#pragma once

#include "bigsplit.hpp"
#include "gendft.cuh"

namespace fh {

// f(RadixC<R>) for a run-time R from 2 to 16
template <typename F>
__device__ __forceinline__ void with_small_radix(int r, F f) {
  if (r == 2) f(RadixC<2>{});
  else if (r == 3) f(RadixC<3>{});
  else with_radix<16>(r, f);
}

// In-place transform of nlines lines (entry i of line q at q ls + i + (i >> sh)) at
// byte offset `a` of the dynamic shared memory, by the warps of threads 0 .. nthr - 1
// (tid in that range); ends with a team barrier.  One body for both directions (the
// inverse is the forward transform of the values with their parts exchanged) and both
// layouts: the register DFTs are compiled once per kernel.
template <typename T>
__device__ __noinline__ void warp_two_step(unsigned a, int nlines, int ls, int sh, bool inverse, LineSplit K, unsigned two,
                                           int tid, int nthr) {
  extern __shared__ __align__(128) unsigned char sm[];
  using C = cplx<T>;
  C* buf = reinterpret_cast<C*>(sm + a);
  const C* tw = reinterpret_cast<const C*>(sm + two);
  auto get = [&](const C* ln, int i) {
    const C z = ln[i + (i >> sh)];
    C r;
    r.x = inverse ? z.y : z.x;
    r.y = inverse ? z.x : z.y;
    return r;
  };
  auto put = [&](C* ln, int i, C z) {
    C r;
    r.x = inverse ? z.y : z.x;
    r.y = inverse ? z.x : z.y;
    ln[i + (i >> sh)] = r;
  };
  // rows of 8 or 16 entries are turned by k1 entries between the steps, so that they do
  // not start on the same banks
  auto turn = [&](int i) { return i >= K.R2 ? i - K.R2 : i; };
  const int lane = tid & 31, nw = nthr >> 5;
  const bool whole = K.R1 == 1;   // a line per lane: the second step alone
  if (!whole) {
    const int lpw = (int)__umulhi(32u, K.m2);
    const int sa = (int)__umulhi((unsigned)lane, K.m2), j2 = lane - sa * K.R2;
    with_radix<16>(K.R1, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
#pragma unroll 1
      for (int l0 = (tid >> 5) * lpw; l0 < nlines; l0 += nw * lpw) {
        const bool on = sa < lpw && l0 + sa < nlines;
        C* ln = buf + (on ? l0 + sa : 0) * ls;
        C v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = get(ln, j2 + K.R2 * j);
        dft_n<R, -1, T>(v);
#pragma unroll
        for (int k = 1; k < R; ++k) v[k] = cmul(v[k], tw[j2 * k]);
        __syncwarp();
        if (on && (K.R2 & 7) == 0) {
#pragma unroll
          for (int k = 0; k < R; ++k) put(ln, k * K.R2 + turn(j2 + k), v[k]);
        } else if (on) {
#pragma unroll
          for (int k = 0; k < R; ++k) put(ln, k * K.R2 + j2, v[k]);
        }
      }
    });
    __syncwarp();
  }
  const int lpw = whole ? 32 : (int)__umulhi(32u, K.m2);
  const int sb = whole ? lane : (int)__umulhi((unsigned)lane, K.m1), k1 = whole ? 0 : lane - sb * K.R1;
  with_small_radix(K.R2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
#pragma unroll 1
    for (int l0 = (tid >> 5) * lpw; l0 < nlines; l0 += nw * lpw) {
      const bool on = sb < lpw && l0 + sb < nlines;
      C* ln = buf + (on ? l0 + sb : 0) * ls;
      C v[R];
#pragma unroll
      for (int j = 0; j < R; ++j) v[j] = get(ln, k1 * K.R2 + (R % 8 == 0 && !whole ? turn(k1 + j) : j));
      dft_n<R, -1, T>(v);
      __syncwarp();
      if (on) {
#pragma unroll
        for (int j = 0; j < R; ++j) put(ln, k1 + K.R1 * j, v[j]);
      }
    }
  });
  team_sync(nthr);
}

template <int R, int DIR, typename T, int PADSH>
__device__ __forceinline__ void big_stage(const cplx<T>* in, cplx<T>* out, int nlines, int ls, int L, int Ns,
                                          const cplx<T>* tw, int tid, int nthr) {
  const int nb = L / R, stride = nb / Ns, total = nlines * nb;
  const bool by_line = (ls & 1) != 0;
  const FDiv fq = make_fdiv(by_line ? nlines : nb), fns = make_fdiv(Ns);
  for (int idx = tid; idx < total; idx += nthr) {
    const int q = fdiv(idx, fq), rem = idx - q * fq.d;
    const int line = by_line ? rem : q, j = by_line ? q : rem;
    const cplx<T>* li = in + line * ls;
    cplx<T>* lo = out + line * ls;
    const int jq = fdiv(j, fns), k = j - jq * Ns;
    cplx<T> v[R];
#pragma unroll
    for (int t = 0; t < R; ++t) v[t] = li[padi<PADSH>(j + t * nb)];
    if (k != 0) {
#pragma unroll
      for (int t = 1; t < R; ++t) {
        cplx<T> w = tw[t * k * stride];
        if (DIR > 0) w.y = -w.y;
        v[t] = cmul(v[t], w);
      }
    }
    dft_n<R, DIR, T>(v);
    const int base = jq * Ns * R + k;
#pragma unroll
    for (int t = 0; t < R; ++t) lo[padi<PADSH>(base + t * Ns)] = v[t];
  }
}

// Transforms nlines lines (stride ls elements) at byte offset `a` of the dynamic
// shared memory, ping-pong with offset `b`; returns the offset that holds the
// result.  Every thread 0 .. nthr - 1 of the team calls it; ends with a team barrier.
template <int DIR, typename T, int PADSH>
__device__ __noinline__ unsigned fft_lines_big(unsigned a, unsigned b, int nlines, int ls, const DevPlan* plan, unsigned two,
                                               int tid, int nthr) {
  extern __shared__ __align__(128) unsigned char sm[];
  const cplx<T>* tw = reinterpret_cast<const cplx<T>*>(sm + two);
  const int L = plan->L;
  int Ns = 1;
  for (int s = 0; s < plan->np; ++s) {
    const cplx<T>* in = reinterpret_cast<const cplx<T>*>(sm + a);
    cplx<T>* out = reinterpret_cast<cplx<T>*>(sm + b);
    const int r = plan->r[s];
    switch (r) {
#define FH_BIG_STAGE(R) \
  case R: big_stage<R, DIR, T, PADSH>(in, out, nlines, ls, L, Ns, tw, tid, nthr); break;
      FH_BIG_STAGE(2) FH_BIG_STAGE(3) FH_BIG_STAGE(4) FH_BIG_STAGE(5) FH_BIG_STAGE(6) FH_BIG_STAGE(7) FH_BIG_STAGE(8)
      FH_BIG_STAGE(9) FH_BIG_STAGE(10) FH_BIG_STAGE(11) FH_BIG_STAGE(12) FH_BIG_STAGE(13) FH_BIG_STAGE(14)
      FH_BIG_STAGE(15) FH_BIG_STAGE(16)
#undef FH_BIG_STAGE
      default:   // reached in FP64 only (cluster_choice); without it ptxas spills more of the FP32 kernel
        stockham_stage_prime<DIR, T, PADSH>(in, out, nlines, ls, L, Ns, r, tw, tid, nthr);
        break;
    }
    team_sync(nthr);
    const unsigned t = a;
    a = b;
    b = t;
    Ns *= r;
  }
  return a;
}

}  // namespace fh
