// Two-step passes for axes of any length N = R1 R2 with radices 4 to 16 (and 18,
// 20, 24, 32 in FP32): 100 = 10 x 10, 96 = 8 x 12, 84 = 7 x 12, 512 = 16 x 32, ...,
// 2-D and 3-D grids, FP32 and FP64, phase-wise or point-by-point stiffness.
//
// The same two steps as line_pass_2s and row_pass_2s (colpass2.cuh,
// rowpass2.cuh, whose compile-time lengths 32, 64 and 128 stay there), with the
// radices chosen at run time by a switch that is uniform over the grid:
//   X[k1 + R1 k2] = sum_j2 w_R2^{j2 k2} w_N^{j2 k1} sum_j1 w_R1^{j1 k1} x[j2 + R2 j1].
// Each value passes through shared memory once per transform (columns) or three
// times (rows), where the general block passes run three or more Stockham stages
// with all index arithmetic, twiddle reads from global memory and a barrier each.
// Index divisions are one multiplication per R points.  100^3 x 6 loads in FP32:
// 0.55 ms an iteration against 2.6 ms (a solve of 20 iterations 12.4 against 53.5 ms).
//
// Line layout: row k1 at offset (R2 | 1) k1, so that its stride is odd.  Column
// tiles: CT = 8 columns a block in FP32 3-D as far as shared memory goes (N <= 512),
// else 4 (gen_columns; FP64: shared memory; 2-D: a 512^2 grid with 3 loads has only
// 771 columns).  Row lines: stride R2 mod 16, so that consecutive entries of
// consecutive lines follow one another.
// 512^2 x 3 loads FP32 with point-by-point stiffness: 63 us an iteration against
// 132 us (block row pass 79, block line pass 53).  Four columns at 640 points (2 x 640 x
// 640 x 6 loads, axis-1 pass): 85 us against 303 us for the block line pass.
#pragma once

#include "genpass.hpp"
#include "gendft.cuh"
#include "smem.hpp"

namespace fh {

template <typename T, int NV> __host__ __device__ constexpr int gen_threads() { return sizeof(T) == 4 && NV == 6 ? 384 : 256; }
template <typename T> __host__ __device__ constexpr int gen_rmax() { return sizeof(T) == 4 ? 32 : 16; }

// q = n / d for n < 2^16, d < 2^16
struct MulDiv {
  unsigned d, mul;
};
inline MulDiv make_muldiv(int d) { return {(unsigned)d, d > 1 ? (unsigned)((0x100000000ull + d - 1) / d) : 0u}; }
__device__ __forceinline__ int qdiv(int n, MulDiv m) { return m.d > 1 ? (int)__umulhi((unsigned)n, m.mul) : n; }

struct GenShape {
  int N, R1, R2;
  int RS;     // stride of row k1 inside a line, R2 | 1
  int LS;     // line stride
  MulDiv dR1, dR2, dN, dH;
};

template <int DIR, typename C>
__device__ __forceinline__ C twiddle(const C* tw, int t) {
  C w = tw[t];
  if (DIR > 0) w.y = -w.y;
  return w;
}

// MODE 0 forward, 1 inverse, 2 forward + Green step + inverse (axis 0), as line_pass_2s
template <typename T, int NV, int MODE, int CT>
__global__ void __launch_bounds__(gen_threads<T, NV>(), 2)
    line_pass_gen(GridInfo g, GenShape K, const cplx<T>* __restrict__ twg, cplx<T>* __restrict__ S,
                  const T* __restrict__ Gt, const LoadState* st, long long stride, long long ncols, int nload) {
  using C = cplx<T>;
  constexpr int NTRI = NV * (NV + 1) / 2, RM = gen_rmax<T>();
  constexpr int DIR = MODE == 1 ? 1 : -1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);   // tw[t] = exp(-2 pi i t / N)
  C* tile = tw + K.N;                        // [NV * CT][LS]
  __shared__ long long colbase[CT];
  const int load = blockIdx.x % nload;
  const long long q0 = (long long)(blockIdx.x / nload) * CT;
  if (st[load].done) return;
  const int nthr = blockDim.x;
  for (int i = threadIdx.x; i < K.N; i += nthr) tw[i] = twg[i];
  if (threadIdx.x < CT) {
    const long long q = q0 + threadIdx.x;
    const long long outer = q / stride;
    colbase[threadIdx.x] = outer * K.N * stride + (q - outer * stride);
  }
  __syncthreads();
  C* Sl = S + (size_t)load * NV * g.nhalf;
  const long long sl0 = (long long)load * NV * g.nhalf, nS = (long long)nload * NV * g.nhalf;
  const int nT = NV * CT * K.LS;
  (void)sl0; (void)nS; (void)nT;

  // stage A: column w, entry j2, component c: points j2 + R2 j1 from global memory
  with_radix<RM>(K.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int a = threadIdx.x; a < NV * CT * K.R2; a += nthr) {
      const int w = a % CT, t = a / CT, c = qdiv(t, K.dR2), j2 = t - c * K.R2;
      const long long o = (long long)c * g.nhalf + colbase[w] + (long long)j2 * stride, step = (long long)K.R2 * stride;
      const bool ok = q0 + w < ncols && FH_IN(CK_C2_S, sl0 + o + (R - 1) * step, nS);
      C v[R];
#pragma unroll
      for (int j = 0; j < R; ++j) {
        v[j].x = v[j].y = T(0);
        if (ok) v[j] = Sl[o + j * step];
      }
      dft_n<R, DIR, T>(v);
      if (!FH_IN(CK_C2_TILE, (c * CT + w) * K.LS + (R - 1) * K.RS + j2, nT)) continue;
      C* line = tile + (c * CT + w) * K.LS + j2;
      line[0] = v[0];
#pragma unroll
      for (int k = 1; k < R; ++k) line[k * K.RS] = cmul(v[k], twiddle<DIR>(tw, j2 * k));
    }
  });
  __syncthreads();

  // stage B: row k1; MODE 0 and 1: frequencies k1 + R1 k2 to global memory, MODE 2: in place
  with_radix<RM>(K.R2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for (int b = threadIdx.x; b < NV * CT * K.R1; b += nthr) {
      const int w = b % CT, t = b / CT, c = qdiv(t, K.dR1), k1 = t - c * K.R1;
      if (!FH_IN(CK_C2_TILE, (c * CT + w) * K.LS + k1 * K.RS + R - 1, nT)) continue;
      C* line = tile + (c * CT + w) * K.LS + k1 * K.RS;
      C v[R];
#pragma unroll
      for (int j = 0; j < R; ++j) v[j] = line[j];
      dft_n<R, DIR, T>(v);
      if constexpr (MODE != 2) {
        const long long o = (long long)c * g.nhalf + colbase[w] + (long long)k1 * stride, step = (long long)K.R1 * stride;
        if (q0 + w < ncols && FH_IN(CK_C2_S, sl0 + o + (R - 1) * step, nS)) {
#pragma unroll
          for (int j = 0; j < R; ++j) Sl[o + j * step] = v[j];
        }
      } else {
#pragma unroll
        for (int j = 0; j < R; ++j) line[j] = v[j];
      }
    }
  });
  if constexpr (MODE == 2) {
    __syncthreads();
    // Green step at frequency (n along this axis, column q): f = n * stride + q
    for (int idx = threadIdx.x; idx < K.N * CT; idx += nthr) {
      const int w = idx % CT, n = idx / CT;
      const long long q = q0 + w;
      if (q >= ncols) continue;
      const long long f = (long long)n * stride + q;
      const int k2 = qdiv(n, K.dR1);
      const int off = (n - k2 * K.R1) * K.RS + k2;
      if (!FH_IN(CK_C2_G, f, g.nhalf) || !FH_IN(CK_C2_TILE, ((NV - 1) * CT + w) * K.LS + off, nT)) continue;
      C tv[NV];
#pragma unroll
      for (int c = 0; c < NV; ++c) tv[c] = tile[(c * CT + w) * K.LS + off];
      T gm[NTRI];
#pragma unroll
      for (int t = 0; t < NTRI; ++t) gm[t] = Gt[(size_t)t * g.nhalf + f];
#pragma unroll
      for (int a = 0; a < NV; ++a) {
        T re = T(0), im = T(0);
#pragma unroll
        for (int b = 0; b < NV; ++b) {
          const int lo = a < b ? a : b, hi = a < b ? b : a;
          const T gv = gm[lo * NV - (lo * (lo - 1)) / 2 + (hi - lo)];
          re = fma(-gv, tv[b].x, re);
          im = fma(-gv, tv[b].y, im);
        }
        C e;
        e.x = (f == 0) ? T(0) : re;
        e.y = (f == 0) ? T(0) : im;
        tile[(a * CT + w) * K.LS + off] = e;
      }
    }
    __syncthreads();
    // inverse, stage B: row k1, sum over k2, then the twiddles w_N^{+j2 k1}
    with_radix<RM>(K.R2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int b = threadIdx.x; b < NV * CT * K.R1; b += nthr) {
        const int w = b % CT, t = b / CT, c = qdiv(t, K.dR1), k1 = t - c * K.R1;
        if (!FH_IN(CK_C2_TILE, (c * CT + w) * K.LS + k1 * K.RS + R - 1, nT)) continue;
        C* line = tile + (c * CT + w) * K.LS + k1 * K.RS;
        C v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = line[j];
        dft_n<R, 1, T>(v);
        line[0] = v[0];
#pragma unroll
        for (int j = 1; j < R; ++j) line[j] = cmul(v[j], twiddle<1>(tw, j * k1));
      }
    });
    __syncthreads();
    // inverse, stage A: entry j2, sum over k1, points j2 + R2 j1 to global memory
    with_radix<RM>(K.R1, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int a = threadIdx.x; a < NV * CT * K.R2; a += nthr) {
        const int w = a % CT, t = a / CT, c = qdiv(t, K.dR2), j2 = t - c * K.R2;
        if (!FH_IN(CK_C2_TILE, (c * CT + w) * K.LS + (R - 1) * K.RS + j2, nT)) continue;
        const C* line = tile + (c * CT + w) * K.LS + j2;
        C v[R];
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = line[k * K.RS];
        dft_n<R, 1, T>(v);
        const long long o = (long long)c * g.nhalf + colbase[w] + (long long)j2 * stride, step = (long long)K.R2 * stride;
        if (q0 + w < ncols && FH_IN(CK_C2_S, sl0 + o + (R - 1) * step, nS)) {
#pragma unroll
          for (int j = 0; j < R; ++j) Sl[o + j * step] = v[j];
        }
      }
    });
  }
}

// The row pass (row_pass_2s): a block owns RB rows of one load, their RB n_v real
// lines taken in pairs as complex lines (real line f = n_v r + c is component c of
// row r); one task per thread and stage, so that a stage's results wait in registers
// for the barrier before they are written.  Cfld (not null): the stiffness point by
// point, upper triangle [tri][m], instead of the phase table.
template <typename T, int NV, bool FIRST, bool KINV>
__global__ void __launch_bounds__(gen_threads<T, NV>(), 2)
    row_pass_gen(GridInfo g, GenShape K, int RB, const cplx<T>* __restrict__ twg, T* __restrict__ E, cplx<T>* __restrict__ S,
                 const uint8_t* __restrict__ phase, const T* __restrict__ dC, Control* ctl, LoadState* st,
                 double* __restrict__ partials, double* __restrict__ hist, int blocks_per_load, T* __restrict__ Wout,
                 const T* __restrict__ Yaux, const T* __restrict__ Cfld) {
  static_assert(!(FIRST && KINV), "the inverse-only pass follows a transform");
  using C = cplx<T>;
  constexpr int RM = gen_rmax<T>();
  const int L = K.N, H = g.H, NT = blockDim.x, tid = threadIdx.x;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + L;                           // [ceil(RB NV / 2)][LS]
  __shared__ __align__(16) T dcs[16 * NV * NV];
  __shared__ __align__(16) T dcp[NV == 6 ? 16 * 12 : 1];   // the 12 nonzeros of decoupled phase matrices
  __shared__ double red[32];
  if (!FIRST && !KINV && ctl->all_done) return;   // replays after the last iteration
  const bool decoupled = NV == 6 && ctl->decoupled != 0;
  const bool no_fwd = !FIRST && !KINV && ctl->no_forward != 0;
  const int load = blockIdx.x / blocks_per_load;
  const int qb = blockIdx.x - load * blocks_per_load;
  const long long row0 = (long long)qb * RB;
  const int nrow = (int)min((long long)RB, g.nrows - row0);
  const int nreal = nrow * NV, npair = (nreal + 1) >> 1;
  const bool skip = st[load].done != 0;
  if ((FIRST || KINV) && skip) return;
  ResAcc<T> acc_d, acc_n;
  const size_t cstrS = (size_t)g.nrows * H, cstrE = (size_t)g.m;
  const long long nS = (long long)ctl->nload * NV * g.nhalf, nE = (long long)ctl->nload * NV * g.m;
  const int nB = ((RB * NV + 1) >> 1) * K.LS;
  (void)nS; (void)nE; (void)nB;
  if (!skip) {
    for (int i = tid; i < L; i += NT) tw[i] = twg[i];
    if (!KINV && !Cfld) {   // tau / 2, as in row_pass_2s
      if (decoupled) {
        for (int i = tid; i < 16 * 12; i += NT) dcp[i % (NV == 6 ? 192 : 1)] = T(0.5) * decoupled_entry(dC + (i / 12) * NV * NV, i % 12);
      } else {
        for (int i = tid; i < 16 * NV * NV; i += NT) dcs[i] = T(0.5) * dC[i];
      }
    }
    __syncthreads();
    T e0[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) e0[c] = (T)ctl->eps0[load][c];
    const T scale = (T)g.inv_m;
    const bool incremental = ctl->form == 1;
    C* Sl = S + (size_t)load * NV * cstrS;
    T* El = E + (size_t)load * NV * cstrE;
    // stage A and B tasks of this thread
    const int la = qdiv(tid, K.dR2), j2 = tid - la * K.R2;
    const int lb = qdiv(tid, K.dR1), k1 = tid - lb * K.R1;
    const bool onA = la < npair, onB = lb < npair;
    C* lineA = buf + la * K.LS;
    C* lineB = buf + lb * K.LS;
    // half spectrum of real line f of this block (row row0 + f / NV, component f % NV)
    auto spec = [&](int f) -> long long {
      const int r = f / NV;
      return (long long)(f - r * NV) * (long long)cstrS + (row0 + r) * H;
    };

    // one stage with its barrier: values to registers, then to the other layout
    auto stageB = [&](auto dir) {   // row k1 -> points or frequencies k1 + R1 k2 in natural order
      constexpr int DIR = decltype(dir)::value;
      with_radix<RM>(K.R2, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        C v[R];
        if (onB && FH_IN(CK_ROW_SMEM, lb * K.LS + k1 * K.RS + R - 1, nB)) {
#pragma unroll
          for (int j = 0; j < R; ++j) v[j] = lineB[k1 * K.RS + j];
          dft_n<R, DIR, T>(v);
        }
        __syncthreads();
        if (onB && FH_IN(CK_ROW_SMEM, lb * K.LS + k1 + K.R1 * (R - 1), nB)) {
#pragma unroll
          for (int j = 0; j < R; ++j) lineB[k1 + K.R1 * j] = v[j];
        }
      });
      __syncthreads();
    };

    if (!FIRST) {
      // inverse, stage A: Z[j2 + R2 j1] = A + i B from the half spectra (conjugate mirror for k > L / 2)
      with_radix<RM>(K.R1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        if (onA && FH_IN(CK_ROW_S, (long long)load * NV * (long long)cstrS + spec(2 * la) + H - 1, nS) &&
            FH_IN(CK_ROW_SMEM, la * K.LS + (R - 1) * K.RS + j2, nB)) {
          const C* SA = Sl + spec(2 * la);
          const bool two = NV == 6 || 2 * la + 1 < nreal;   // an odd number of real lines: the last pair has one
          const C* SB = two ? Sl + spec(2 * la + 1) : SA;
          const T tb = two ? T(1) : T(0);
          C v[R];
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const int k = j2 + K.R2 * j;
            const bool lo = 2 * k <= L;
            const int kk = lo ? k : L - k;
            const T s = lo ? T(1) : T(-1);
            const C A = SA[kk];
            C B = SB[kk];
            if (NV != 6) { B.x *= tb; B.y *= tb; }
            v[j].x = A.x - s * B.y;
            v[j].y = s * A.y + B.x;
          }
          dft_n<R, 1, T>(v);
          lineA[j2] = v[0];
#pragma unroll
          for (int k = 1; k < R; ++k) lineA[k * K.RS + j2] = cmul(v[k], twiddle<1>(tw, j2 * k));
        }
      });
      __syncthreads();
      stageB(RadixC<1>{});
    }

    // pointwise: E update, residual sums, tau into the lines
    for (int idx = tid; idx < nrow * L; idx += NT) {
      const int r = qdiv(idx, K.dN), x = idx - r * L;
      const size_t pt = (size_t)(row0 + r) * L + x;
      if (!(FH_IN(CK_ROW_E, (long long)load * NV * (long long)cstrE + (NV - 1) * (long long)cstrE + (long long)pt, nE) &&
            FH_IN(CK_ROW_PHASE, (long long)pt, g.m) && FH_IN(CK_ROW_SMEM, ((r * NV + NV - 1) >> 1) * K.LS + x, nB)))
        continue;
      const int f0 = r * NV;
      T* ln = reinterpret_cast<T*>(buf + x);   // real line f at ln[(f >> 1) 2 LS + (f & 1)]
      auto at = [&](int c) -> T& { return ln[(size_t)((f0 + c) >> 1) * 2 * K.LS + ((f0 + c) & 1)]; };
      T ev[NV];
#pragma unroll
      for (int c = 0; c < NV; ++c) ev[c] = El[c * cstrE + pt];
      if constexpr (KINV) {
        const T* Yl = Yaux ? Yaux + (size_t)load * NV * cstrE : El;
        T* Wl = Wout + (size_t)load * NV * cstrE;
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          const T wv = ev[c] - at(c) * scale;
          Wl[c * cstrE + pt] = wv;
          acc_d.add_prod(wv, Yaux ? Yl[c * cstrE + pt] : ev[c]);
          acc_n.add_sq(wv);
        }
        continue;
      }
      T en[NV];
      if (FIRST) {
#pragma unroll
        for (int c = 0; c < NV; ++c) en[c] = ev[c];
      } else {
        T rd = T(0), rn = T(0);
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          en[c] = at(c) * scale;
          if (incremental) en[c] += ev[c];
          const T dd = en[c] - ev[c], nn = en[c] + e0[c];
          rd = fma(dd, dd, rd);
          rn = fma(nn, nn, rn);
          El[c * cstrE + pt] = en[c];
        }
        acc_d.add(rd);
        acc_n.add(rn);
      }
      if (no_fwd) continue;
      T xv[NV], tau[NV];
#pragma unroll
      for (int b = 0; b < NV; ++b) xv[b] = en[b] + e0[b];
      if (Cfld) {
#pragma unroll
        for (int a = 0; a < NV; ++a) tau[a] = T(0);
#pragma unroll
        for (int a = 0; a < NV; ++a)
#pragma unroll
          for (int b = a; b < NV; ++b) {
            const T cab = Cfld[(size_t)(a * NV - (a * (a - 1)) / 2 + (b - a)) * g.m + pt];
            tau[a] = fma(cab, xv[b], tau[a]);
            if (b != a) tau[b] = fma(cab, xv[a], tau[b]);
          }
#pragma unroll
        for (int a = 0; a < NV; ++a) tau[a] *= T(0.5);
      } else {
        int ph = phase[pt];
        if (!FH_IN(CK_ROW_PHASE, ph, 16)) ph = 0;
        if (NV == 6 && decoupled) {
          if constexpr (NV == 6) stress6_decoupled<T>(dcp + ph * 12, xv, tau);
        } else {
          const T* dc = dcs + ph * NV * NV;
#pragma unroll
          for (int a = 0; a < NV; ++a) {
            T t = T(0);
#pragma unroll
            for (int b = 0; b < NV; ++b) t = fma(dc[a * NV + b], xv[b], t);
            tau[a] = t;
          }
        }
      }
#pragma unroll
      for (int c = 0; c < NV; ++c) at(c) = tau[c];
    }
    if (NV != 6 && !KINV && (nreal & 1))   // the imaginary part of the last pair
      for (int x = tid; x < L; x += NT) buf[(npair - 1) * K.LS + x].y = T(0);

    if (!KINV && !no_fwd) {
      __syncthreads();
      // forward, stage A: points j2 + R2 j1 -> row layout with the twiddles
      with_radix<RM>(K.R1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        C v[R];
        if (onA && FH_IN(CK_ROW_SMEM, la * K.LS + j2 + K.R2 * (R - 1), nB)) {
#pragma unroll
          for (int j = 0; j < R; ++j) v[j] = lineA[j2 + K.R2 * j];
          dft_n<R, -1, T>(v);
#pragma unroll
          for (int k = 1; k < R; ++k) v[k] = cmul(v[k], twiddle<-1>(tw, j2 * k));
        }
        __syncthreads();
        if (onA && FH_IN(CK_ROW_SMEM, la * K.LS + (R - 1) * K.RS + j2, nB)) {
#pragma unroll
          for (int k = 0; k < R; ++k) lineA[k * K.RS + j2] = v[k];
        }
      });
      __syncthreads();
      stageB(RadixC<-1>{});
      // split each line's spectrum into the half spectra of its two real lines
      for (int idx = tid; idx < npair * H; idx += NT) {
        const int line = qdiv(idx, K.dH), k = idx - line * H;
        if (!FH_IN(CK_ROW_S, (long long)load * NV * (long long)cstrS + spec(2 * line) + k, nS)) continue;
        const C* ln = buf + line * K.LS;
        const C zk = ln[k];
        const C zm = ln[k == 0 ? 0 : L - k];
        C A, B;
        A.x = zk.x + zm.x;
        A.y = zk.y - zm.y;
        B.x = zk.y + zm.y;
        B.y = zm.x - zk.x;
        Sl[spec(2 * line) + k] = A;
        if (NV == 6 || 2 * line + 1 < nreal) Sl[spec(2 * line + 1) + k] = B;
      }
    }
  }
  if (FIRST) return;
  const double d2 = block_sum_acc(acc_d, red);
  const double n2 = block_sum_acc(acc_n, red);
  if (tid == 0) {
    partials[2 * (size_t)blockIdx.x] = d2;
    partials[2 * (size_t)blockIdx.x + 1] = n2;
  }
  if (KINV) return;
  __shared__ unsigned int s_ticket;
  if (tid == 0) {
    __threadfence();
    s_ticket = atomicAdd(&ctl->ticket, 1u);
  }
  __syncthreads();
  if (s_ticket != gridDim.x - 1) return;
  __threadfence();
  finish_row_pass(ctl, st, partials, hist, blocks_per_load);
}

inline GenShape gen_shape(int N, bool fp32, int H) {
  GenShape K{};
  K.N = N;
  gen_split(N, fp32, &K.R1, &K.R2);
  K.RS = gen_row_stride(K.R2);
  K.dR1 = make_muldiv(K.R1);
  K.dR2 = make_muldiv(K.R2);
  K.dN = make_muldiv(N);
  K.dH = make_muldiv(H);
  return K;
}
inline GenShape gen_row_shape(int N, bool fp32, int H) {
  GenShape K = gen_shape(N, fp32, H);
  K.LS = gen_line_stride(K.R1, K.R2, K.R2 % 16);
  return K;
}

// rows per block: one task per thread, two blocks' lines in shared memory, and
// (few rows) about two blocks per SM
template <typename T, int NV>
int gen_rb(int L, long long rows_of_all_loads) {
  constexpr bool fp32 = sizeof(T) == 4;
  const GenShape K = gen_row_shape(L, fp32, 1);
  int rb = std::max(1, 2 * (gen_threads<T, NV>() / K.R2) / NV);
  auto lines = [](int r) { return (r * NV + 1) / 2; };
  while (rb > 1 && (lines(rb) * K.R2 > gen_threads<T, NV>() || (size_t)(L + lines(rb) * K.LS) * 2 * sizeof(T) > 96 * 1024)) --rb;
  const long long want = (rows_of_all_loads + 2 * 152 - 1) / (2 * 152);
  return (int)std::max<long long>(1, std::min<long long>(rb, want));
}

template <typename T, int NV, int CT>
cudaError_t gen_col_prepare_ct(int N) {
  const size_t sm = gen_col_bytes(N, sizeof(T) == 4, NV, CT);
  cudaError_t e = allow_smem((const void*)line_pass_gen<T, NV, 2, CT>, sm);
  if constexpr (NV == 6) {   // 2-D grids have axis 0 only
    if (e == cudaSuccess) e = allow_smem((const void*)line_pass_gen<T, NV, 0, CT>, sm);
    if (e == cudaSuccess) e = allow_smem((const void*)line_pass_gen<T, NV, 1, CT>, sm);
  }
  return e;
}
template <typename T, int NV>
cudaError_t gen_col_prepare_t(int N) {
  if constexpr (sizeof(T) == 4 && NV == 6) {
    if (gen_columns(N, true, NV) == 8) return gen_col_prepare_ct<T, NV, 8>(N);
  }
  return gen_col_prepare_ct<T, NV, 4>(N);
}
// shared memory of the row pass with rb rows per block
template <typename T, int NV>
size_t gen_row_bytes(const GenShape& K, int rb) {
  return (size_t)(K.N + (rb * NV + 1) / 2 * K.LS) * 2 * sizeof(T);
}
template <typename T, int NV>
cudaError_t gen_row_prepare_t(const GridInfo& g, int rb) {
  const size_t sm = gen_row_bytes<T, NV>(gen_row_shape(g.L, sizeof(T) == 4, g.H), rb);
  cudaError_t e = allow_smem((const void*)row_pass_gen<T, NV, true, false>, sm);
  if (e == cudaSuccess) e = allow_smem((const void*)row_pass_gen<T, NV, false, true>, sm);
  if (e == cudaSuccess) e = allow_smem((const void*)row_pass_gen<T, NV, false, false>, sm);
  return e;
}

template <typename T, int NV, int CT>
cudaError_t gen_col_ct(int mode, const GridInfo& g, int N, const cplx<T>* tw, cplx<T>* S, const T* G, const LoadState* st,
                      long long stride, int nload, cudaStream_t stream) {
  constexpr int TH = gen_threads<T, NV>();
  GenShape K = gen_shape(N, sizeof(T) == 4, 1);
  K.LS = gen_col_stride(K.R1, K.R2, sizeof(T) == 4, CT);
  const long long ncols = g.nhalf / N, tiles = (ncols + CT - 1) / CT;
  const size_t sm = gen_col_bytes(N, sizeof(T) == 4, NV, CT);
  // a stage's NV CT R2 tasks in equal rounds
  const int tasks = NV * CT * K.R2, rounds = (tasks + TH - 1) / TH;
  const int threads = ((tasks + rounds - 1) / rounds + 31) / 32 * 32;
  auto launch = [&](auto kern) {
    kern<<<(unsigned)(tiles * nload), threads, sm, stream>>>(g, K, tw, S, G, st, stride, ncols, nload);
    return cudaGetLastError();
  };
  if constexpr (NV == 6) {
    if (mode == 0) return launch(line_pass_gen<T, NV, 0, CT>);
    if (mode == 1) return launch(line_pass_gen<T, NV, 1, CT>);
  }
  return launch(line_pass_gen<T, NV, 2, CT>);
}

template <typename T, int NV>
cudaError_t gen_col_t(int mode, const GridInfo& g, int N, const cplx<T>* tw, cplx<T>* S, const T* G, const LoadState* st,
                      long long stride, int nload, cudaStream_t stream) {
  if constexpr (sizeof(T) == 4 && NV == 6) {
    if (gen_columns(N, true, NV) == 8) return gen_col_ct<T, NV, 8>(mode, g, N, tw, S, G, st, stride, nload, stream);
  }
  return gen_col_ct<T, NV, 4>(mode, g, N, tw, S, G, st, stride, nload, stream);
}

template <typename T, int NV>
cudaError_t gen_row_t(bool first, bool kinv, const GridInfo& g, const cplx<T>* tw, T* E, cplx<T>* S, const uint8_t* phase,
                      const T* dC, Control* ctl, LoadState* st, double* partials, double* hist, int nload, int rb, T* Wout,
                      const T* Yaux, const T* Cfld, cudaStream_t stream) {
  const GenShape K = gen_row_shape(g.L, sizeof(T) == 4, g.H);
  const int bpl = (int)((g.nrows + rb - 1) / rb), lines = (rb * NV + 1) / 2;
  const size_t sm = gen_row_bytes<T, NV>(K, rb);
  const int threads = (lines * K.R2 + 31) / 32 * 32;
  auto launch = [&](auto kern) {
    kern<<<(unsigned)(nload * bpl), threads, sm, stream>>>(g, K, rb, tw, E, S, phase, dC, ctl, st, partials, hist, bpl, Wout, Yaux,
                                                           Cfld);
    return cudaGetLastError();
  };
  if (first) return launch(row_pass_gen<T, NV, true, false>);
  if (kinv) return launch(row_pass_gen<T, NV, false, true>);
  return launch(row_pass_gen<T, NV, false, false>);
}

}  // namespace fh
