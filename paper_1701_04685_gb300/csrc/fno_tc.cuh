// Tensor-core (tcgen05) form of the hidden layers' row kernel (fno_rows.cuh) for 32
// channels and rows of N = 16 .. 128 points, a multiple of 16.
//
// A CTA takes four rows (b, x, y) at a time, 128 lines (row r, channel o):
//   D1[(r,o)][z] = sum_c W[o][c] in[r][c][z] + sum_k Iy[r][k][o] T[k][z]
//   out = epi(D1 + bias);   D2[(r,o)][k] = sum_z out[r][o][z] T[k][z]  (the next Yz)
// with M = 128 lines, N points or spectral rows, accumulated in FP32 in tensor memory.
// The 1 x 1 layer of row r is one MMA over K = 32 channels whose A operand is W in the
// 32 rows of r and zero elsewhere (a window into 96 zero rows, W, 96 zero rows), so the
// four rows add up in one accumulator; the zero products cost nothing that is scarce.
// Weights are BF16; every FP32 operand is split into three BF16 terms, x = x0 + x1 + x2
// (to 2^-24 relative): three products with the exact weights, the six leading ones of
// (three terms) x (three terms of T), smallest first.  This keeps the FP32 accuracy of
// the SIMT form.  A lane of tensor memory is a line, so an epilogue thread holds
// consecutive points: its 32-byte stores are whole sectors, and its values go back to
// shared memory as the K-major operand of the second product without a transposition.
//
// Operands: K-major without swizzle, 8 x 8 core matrices of 128 bytes, core matrices
// along K 128 bytes apart, 8-row groups K / 8 * 128 bytes apart.  One thread issues,
// tcgen05.commit signals an mbarrier; waits are bounded: a kernel whose wait gave up
// records an error, frees its tensor memory and returns.
//
// The SIMT form issues 11 000 warp instructions a row, 5 100 of them multiply-adds, at
// 53 % issue; here the products leave the FP32 pipe and what remains is the splitting,
// the GELU and the traffic: 4 900 instructions a row.  64^3, 32 channels, 12 modes, one
// sample: 48 us a layer with two CTAs per SM (70 with one, 82 in the SIMT form), bound by
// the wait for a tile's loads (HBM floor of four samples' 445 MB: 65 us).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "fno_rows.cuh"

namespace fhtc {

constexpr int kTcThreads = 256;
constexpr int kTcW = 32;        // channels
constexpr int kTcRows = 4;      // rows per tile: 128 lines
constexpr int kTcWin = 96 + kTcW + 96;   // rows of the weight window

struct TcArgs {
  int N, N3, N2, m2, Kp, ntiles;
  int ncols;                    // tensor-memory columns (a power of two >= N + Kp)
  const float* in;              // [b][32][N3]
  const __nv_bfloat16* W;       // [32][32]
  int trans;                    // A[o][c] = W[c][o]
  const float* bias;            // [32] or null
  const float* Iy;              // [row][m2][32]
  const float* T;               // [m2][N]
  const float* u_in;
  float* u_out;
  float* out;
  float* Yz;                    // [row][m2][32] or null
  int* err;
};

// byte offsets of the operands in shared memory
struct TcLayout {
  uint32_t win, v, iy, t1, t2, total;
};
__host__ __device__ inline TcLayout tc_layout(int N, int Kp) {
  TcLayout l;
  uint32_t o = 0;
  l.win = o; o += kTcWin * kTcW * 2;
  l.v = o;   o += 128 * N * 6;            // [r][3][N][32], later out as [3][128][N]
  l.iy = o;  o += 128 * Kp * 6;           // [3][128][Kp]
  l.t1 = o;  o += N * Kp * 6;             // [3][N][Kp]
  l.t2 = o;  o += Kp * N * 6;             // [3][Kp][N]
  l.total = o;
  return l;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: K-major, no swizzle, K columns
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, int K) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((128u >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((((uint32_t)K / 8 * 128) >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, M = 128
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (8u << 24);
}
// byte offset of row r, columns k .. k + 7 (k a multiple of 8)
__device__ __forceinline__ uint32_t koff(int r, int k, int K) {
  return (uint32_t)((r >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (r & 7) * 16);
}

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar) : "memory");
}
// bounded wait for the phase; false when it gave up
__device__ __forceinline__ bool wait_phase(uint32_t mbar, uint32_t phase) {
  uint32_t done = 0;
  for (int it = 0; it < (1 << 20) && !done; ++it)
    asm volatile("{\n .reg .pred q;\n mbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n selp.u32 %0, 1, 0, q;\n}\n"
                 : "=r"(done)
                 : "r"(mbar), "r"(phase)
                 : "memory");
  return done != 0;
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, float (&r)[8]) {
  uint32_t v[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) r[i] = __uint_as_float(v[i]);
}
// eight consecutive floats (32-byte aligned), one sector
__device__ __forceinline__ void st8(float* p, const float (&v)[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
               "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void ld8(const float* p, float (&v)[8]) {
  asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p));
}

// eight values as three BF16 terms, 16 bytes each, to p, p + step, p + 2 step
__device__ __forceinline__ void split_store(unsigned char* p, uint32_t step, const float (&x)[8]) {
  uint32_t t[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a = x[2 * i], b = x[2 * i + 1];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
      t[s][i] = *reinterpret_cast<const uint32_t*>(&h);
      if (s < 2) {
        a -= __uint_as_float(t[s][i] << 16);
        b -= __uint_as_float(t[s][i] & 0xffff0000u);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < 3; ++s) *reinterpret_cast<uint4*>(p + s * step) = make_uint4(t[s][0], t[s][1], t[s][2], t[s][3]);
}

template <int EPI>
__global__ void __launch_bounds__(kTcThreads, 2) k_rows_tc(const TcArgs a) {
  extern __shared__ __align__(1024) unsigned char smt[];
  __shared__ __align__(8) uint64_t mbar_s;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = a.N, Kp = a.Kp;
  const TcLayout lay = tc_layout(N, Kp);
  const uint32_t base = smem_addr(smt), mbar = smem_addr(&mbar_s);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(&tmem_slot)), "r"(a.ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    s_abort = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mbar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  // constant operands: the weight window, T as [z][k] and as [k][z]
  for (int i = tid; i < kTcWin * kTcW / 8; i += kTcThreads) {
    const int r = i >> 2, k0 = (i & 3) * 8, o = r - 96;
    __nv_bfloat16 w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      w[j] = o >= 0 && o < kTcW ? (a.trans ? a.W[(k0 + j) * kTcW + o] : a.W[o * kTcW + k0 + j]) : __float2bfloat16_rn(0.f);
    uint4 q;
    memcpy(&q, w, 16);
    *reinterpret_cast<uint4*>(smt + lay.win + koff(r, k0, kTcW)) = q;
  }
  for (int i = tid; i < N * (Kp >> 3); i += kTcThreads) {
    const int z = i % N, k0 = (i / N) * 8;
    float x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = k0 + j < a.m2 ? a.T[(k0 + j) * N + z] : 0.f;
    split_store(smt + lay.t1 + koff(z, k0, Kp), (uint32_t)N * Kp * 2, x);
  }
  for (int i = tid; i < Kp * (N >> 3); i += kTcThreads) {
    const int k = i % Kp, z0 = (i / Kp) * 8;
    float x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = k < a.m2 ? a.T[k * N + z0 + j] : 0.f;
    split_store(smt + lay.t2 + koff(k, z0, N), (uint32_t)N * Kp * 2, x);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_slot, d2 = tmem + (uint32_t)N;
  const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
  const int r = warp & 3, half = warp >> 2, line = 32 * r + lane;   // this thread's line: row r, channel lane
  const float bias = a.bias ? a.bias[lane] : 0.f;
  uint32_t phase = 0;
  for (int tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const int row0 = tile * kTcRows;
    // input rows as B operands [z][c], their spectral coefficients as the A operand [(r,o)][k]
#pragma unroll 4
    for (int i = tid; i < kTcRows * N * (kTcW / 8); i += kTcThreads) {
      const int z = i % N, q = i / N, c0 = (q & 3) * 8, rr = q >> 2;
      const int row = row0 + rr, b = row / a.N2;
      const float* p = a.in + ((size_t)b * kTcW + c0) * a.N3 + (size_t)(row - b * a.N2) * N + z;
      float x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = p[(size_t)j * a.N3];
      split_store(smt + lay.v + (uint32_t)rr * N * kTcW * 6 + koff(z, c0, kTcW), (uint32_t)N * kTcW * 2, x);
    }
#pragma unroll 2
    for (int i = tid; i < 128 * (Kp >> 3); i += kTcThreads) {
      const int ln = i & 127, k0 = (i >> 7) * 8;
      const float* p = a.Iy + ((size_t)(row0 + (ln >> 5)) * a.m2 + k0) * kTcW + (ln & 31);
      float x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = k0 + j < a.m2 ? p[j * kTcW] : 0.f;
      split_store(smt + lay.iy + koff(ln, k0, Kp), 128u * Kp * 2, x);
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (tid == 0) {
      const uint32_t id = idesc_bf16(N);
      uint32_t acc = 0;
      // terms (s of Iy, t of T), smallest products first; 16 columns are 256 bytes
      const int ps[6] = {2, 1, 0, 1, 0, 0}, pt[6] = {0, 1, 2, 0, 1, 0};
      for (int q = 0; q < 6; ++q)
        for (int k = 0; k < Kp / 16; ++k) {
          mma(tmem, sdesc(base + lay.iy + ps[q] * 128 * Kp * 2 + k * 256, Kp), sdesc(base + lay.t1 + pt[q] * N * Kp * 2 + k * 256, Kp),
              id, acc);
          acc = 1;
        }
      for (int s = 2; s >= 0; --s)
        for (int rr = 0; rr < kTcRows; ++rr)
          for (int k = 0; k < 2; ++k)
            mma(tmem, sdesc(base + lay.win + (uint32_t)(12 - 4 * rr) * 512 + k * 256, kTcW),
                sdesc(base + lay.v + (uint32_t)(rr * 3 + s) * N * kTcW * 2 + k * 256, kTcW), id, 1);
      commit(mbar);
    }
    if (!wait_phase(mbar, phase)) s_abort = 1;
    __syncthreads();
    if (s_abort) {
      if (tid == 0) atomicExch(a.err, 1);
      break;
    }
    phase ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    // epilogue: this thread's line, half of its points
    {
      const int row = row0 + r, b = row / a.N2;
      const size_t p0 = ((size_t)b * kTcW + lane) * a.N3 + (size_t)(row - b * a.N2) * N;
      for (int z0 = half * (N / 2); z0 < (half + 1) * (N / 2); z0 += 8) {
        float v[8];
        tmem_ld8(tmem + lane_base + (uint32_t)z0, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += bias;
        if (EPI == 1) {
          if (a.u_out) st8(a.u_out + p0 + z0, v);
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = fhrow::row_gelu(v[j]);
        } else if (EPI == 2) {
          float u[8];
          ld8(a.u_in + p0 + z0, u);
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] *= fhrow::row_dgelu(u[j]);
        }
        if (a.out) st8(a.out + p0 + z0, v);
        if (a.Yz) split_store(smt + lay.v + koff(line, z0, N), 128u * N * 2, v);   // the input operands are done with
      }
    }
    if (a.Yz) {
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      if (tid == 0) {
        const uint32_t id = idesc_bf16(Kp);
        uint32_t acc = 0;
        const int ps[6] = {2, 1, 0, 1, 0, 0}, pt[6] = {0, 1, 2, 0, 1, 0};
        for (int q = 0; q < 6; ++q)
          for (int k = 0; k < N / 16; ++k) {
            mma(d2, sdesc(base + lay.v + ps[q] * 128 * N * 2 + k * 256, N), sdesc(base + lay.t2 + pt[q] * N * Kp * 2 + k * 256, N), id,
                acc);
            acc = 1;
          }
        commit(mbar);
      }
      if (!wait_phase(mbar, phase)) s_abort = 1;
      __syncthreads();
      if (s_abort) {
        if (tid == 0) atomicExch(a.err, 1);
        break;
      }
      phase ^= 1u;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      for (int k0 = half * 8; k0 < a.m2; k0 += 16) {
        float v[8];
        tmem_ld8(d2 + lane_base + (uint32_t)k0, v);
        float* p = a.Yz + ((size_t)(row0 + r) * a.m2 + k0) * kTcW + lane;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (k0 + j < a.m2) p[j * kTcW] = v[j];
      }
    }
    // every warp has read the accumulators before the next tile's products overwrite them
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  }
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(a.ncols) : "memory");
}

}  // namespace fhtc
