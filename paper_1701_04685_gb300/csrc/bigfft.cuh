// Shared-memory line transform of the cluster kernel for axes that are no powers
// of two: the Stockham stages of fft.cuh with every radix from 2 to 16 (gendft.cuh),
// so that most lengths need two stages and none below 4096 more than four (96 = 8 x
// 12, 192 = 12 x 16, 768 = 8 x 8 x 12, where the schedule of 8, 4, 2, 3, ... has
// three to five), plus the direct stage for larger primes.
//
// A stage deals its butterflies line by line across the lanes: with the odd line
// strides of the cluster layout every access is free of bank conflicts and a warp's
// twiddles are broadcasts (butterfly by butterfly along a line, stages of stride 12
// conflict four ways).  The function is not inlined: its 15 register DFTs appear
// once per direction, the kernel keeps 16 warps per CTA in FP32, and shared memory
// is addressed by byte offsets so that the accesses stay shared-memory instructions.
#pragma once

#include "gendft.cuh"

namespace fh {

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
      default: stockham_stage_prime<DIR, T, PADSH>(in, out, nlines, ls, L, Ns, r, tw, tid, nthr); break;
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
