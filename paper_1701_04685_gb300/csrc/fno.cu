// Fourier-neural-operator start predictor: forward, backward and Adam kernels.
//
// The network (not part of the paper; it supplies the starting strain of the
// paper's fixed point) maps input channels x on an N^3 grid to the strain
// fluctuation y:
//   v_0 = P x + p;  u_l = W_l v_l + w_l + K_l v_l,  v_{l+1} = gelu(u_l);  y = Q v_L + q,
// with the spectral convolution restricted to kx, ky in {-m..m-1}, kz in {0..m-1}:
//   v^(k) = sum_x v(x) e^{-2 pi i k.x/N},  c = R_l(k) v^(k),
//   (K v)(x) = N^-3 Re sum_k w(kz) c(k) e^{+2 pi i k.x/N},  w(0) = 1, w(kz>0) = 2.
// Only 4 m^3 of the N^3 modes are kept, so each transform is a small dense
// contraction along one axis at a time.  R and W are used in BF16 (stored from
// FP32 master weights), every product is accumulated in FP32.  A layer is four
// launches: DFT along y; DFT along x, channel mixing and inverse DFT along x;
// inverse DFT along y (fno_spec.cuh); and the row kernel (fno_rows.cuh) with
// both z transforms, the 1 x 1 layer and the activation.
//
// Layouts: activations [B][C][N^3] (z fastest); spectral coefficients
// channels-last [B][mode][C], mode = (ax * 2m + ay) * m + kz;
// R [layer][mode][out][in].

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "internal.hpp"
#include "fno_rows.cuh"
#include "fno_spec.cuh"
#include "fno_out.hpp"
#include "fno_tc.cuh"
#include "smem.hpp"

namespace {

constexpr int kT = 256;

struct FnoDims {
  int N, cin, cout, W, m, L;
  int N3;      // N^3
  int NM;      // (2m)^2 m modes
};

__global__ void k_adam(long long n, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    w[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
  }
}

// public order of a parameter vector (real parts of R, then its imaginary parts)
// from the device's (interleaved)
__global__ void k_to_flat(long long n, long long off, long long nR, const float* __restrict__ src, float* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long j = i - off;
    dst[i] = src[j < 0 || j >= 2 * nR ? i : j < nR ? off + 2 * j : off + 2 * (j - nR) + 1];
  }
}

struct FeatParams {
  float logE[16];
  float e0[6];
};

__global__ void k_features(int N3, FeatParams P, const uint8_t* __restrict__ phase, float* __restrict__ x,
                           int with_strain) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N3; i += gridDim.x * blockDim.x) {
    x[i] = P.logE[phase[i] & 15];
    if (with_strain)
      for (int c = 0; c < 6; ++c) x[(size_t)(c + 1) * N3 + i] = P.e0[c];
  }
}

__global__ void k_to_bf16(long long n, const float* __restrict__ src, __nv_bfloat16* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = __float2bfloat16_rn(src[i]);
}

}  // namespace

// ---------------------------------------------------------------- host object
struct fh_fno {
  FnoDims d{};
  int max_batch = 0;
  cudaStream_t stream = nullptr;
  // parameters (FP32 master): P [W][cin], p [W], Wl [L][W][W], wl [L][W], R [L][NM][W][W] complex, Q [cout][W], q [cout]
  long long off_P, off_p, off_W, off_w, off_R, off_Q, off_q, nparam;
  float* prm = nullptr;
  float* grd_mem = nullptr;
  float* grd = nullptr;   // in grd_mem, placed so that the gradient of R is 16-byte aligned for any channel counts
  float* m1 = nullptr;
  float* m2 = nullptr;
  __nv_bfloat16* Wbf = nullptr;   // [L][W][W]
  __nv_bfloat16* Rbf = nullptr;   // [L][NM][W][W][2]
  float2* tw = nullptr;           // e^{-2 pi i t/N}
  float* flat = nullptr;          // parameters or gradients in the public order (first read-out on)
  std::mutex flat_mutex;
  float* zt = nullptr;            // z-DFT table [2m][N]: cos(2 pi k z / N), then -sin
  // activations
  float* v = nullptr;       // [L+1][B][W][N3]
  float* u = nullptr;       // [L][B][W][N3]
  float2* vh = nullptr;     // [L][B][NM][W]
  float* Yz = nullptr;      // [B][N][N][2m][W]
  float2* Yy = nullptr;     // [B][N][2m][m][W]
  float* y = nullptr;       // [B][cout][N3]
  float* gy = nullptr;      // [B][cout][N3]
  float* ga = nullptr;      // [B][W][N3]  gradient wrt an activation
  float* gb = nullptr;      // [B][W][N3]
  double* part = nullptr;
  int nparts = 0;
  int device = 0;
  int sms = 1;
  std::map<std::pair<const void*, size_t>, int> prepared;   // see prepare
  // hidden layers on the tensor cores (fno_tc.cuh) where they apply; tc_err is set by
  // a kernel whose bounded wait gave up
  bool tensor_cores = true;
  int* tc_err = nullptr;
};

namespace {

#define FCK(call)                                                            \
  do {                                                                       \
    cudaError_t e_ = (call);                                                 \
    if (e_ != cudaSuccess) {                                                 \
      fh::set_error(std::string(#call) + ": " + cudaGetErrorString(e_));     \
      return FH_ERR_CUDA;                                                    \
    }                                                                        \
  } while (0)

int grid_for(long long n) { return (int)std::min<long long>((n + kT - 1) / kT, 152 * 16); }

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// row-kernel arguments of `cin` input and W output channels (see fno_rows.cuh)
fhrow::RowArgs row_args(const fh_fno* f, int B, int cin, const float* in, const void* A, bool bf16, bool trans,
                        const float* bias) {
  const FnoDims& d = f->d;
  fhrow::RowArgs a{};
  a.N = d.N; a.N2 = d.N * d.N; a.N3 = d.N3;
  a.N4 = (d.N + 3) & ~3;
  a.NS = a.N4 + 4;
  a.W = d.W; a.WP = (d.W + 7) & ~7; a.Cin = cin;
  a.kc = std::max(cin, d.W);
  a.nrows = B * a.N2;
  a.in = in; a.A = A; a.a_bf16 = bf16; a.a_trans = trans; a.bias = bias;
  a.T = f->zt;
  return a;
}

// A kernel's shared-memory limit, once per kernel and size; *resident (where asked for)
// its resident blocks per SM.
cudaError_t prepare(fh_fno* f, const void* kernel, int threads, size_t sm, int* resident = nullptr) {
  auto it = f->prepared.find({kernel, sm});
  if (it == f->prepared.end()) {
    cudaError_t e = fh::allow_smem(kernel, sm);
    int res = 1;
    if (e == cudaSuccess && resident) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&res, kernel, threads, sm);
    if (e != cudaSuccess) return e;
    it = f->prepared.insert({{kernel, sm}, res}).first;
  }
  if (resident) *resident = it->second;
  return cudaSuccess;
}

template <int EPI>
fh_status launch_rows(fh_fno* f, fhrow::RowArgs& a, int* blocks = nullptr) {
  const int nz4 = a.N4 / 4, per_row = (a.WP / 8) * nz4;
  if (a.Iy || a.Yz) a.m2 = 2 * f->d.m;
  a.m2p = (a.m2 + 3) & ~3;
  a.QP = (a.cout + 7) & ~7;
  // a block's rows: one 8 x 4 tile per thread, as far as shared memory goes
  a.rpb = std::max(1, fhrow::kRowThreads / per_row);
  while (a.rpb > 1 && fhrow::row_smem_floats(a) * 4 > 100 * 1024) a.rpb /= 2;
  a.vec = a.N % 4 == 0 && aligned16(a.in) && aligned16(a.y) && aligned16(a.target) && aligned16(a.out);
  a.dNq = fhrow::make_udiv(nz4);
  a.dCin = fhrow::make_udiv(a.Cin);
  a.dTask = fhrow::make_udiv(per_row);
  a.dOg = fhrow::make_udiv(a.WP / 8);
  a.dCg = fhrow::make_udiv(a.WP / 4);
  a.dKg = fhrow::make_udiv(std::max(1, a.m2p / 4));
  a.dQt = fhrow::make_udiv(std::max(1, (a.QP / 8) * nz4));
  a.dQg = fhrow::make_udiv(std::max(1, a.QP / 8));
  const size_t sm = fhrow::row_smem_floats(a) * 4;
  const int ntiles = (a.nrows + a.rpb - 1) / a.rpb;
  int res = 1;
  FCK(prepare(f, (const void*)fhrow::k_rows<EPI>, fhrow::kRowThreads, sm, &res));
  const int grid = std::min(ntiles, std::max(1, res) * f->sms);
  if (blocks) *blocks = grid;
  fhrow::k_rows<EPI><<<grid, fhrow::kRowThreads, sm, f->stream>>>(a);
  FCK(cudaGetLastError());
  return FH_OK;
}

// The tensor-core form takes the hidden layers (BF16 weights, spectral input, no
// projection) of 32 channels on rows of 16 .. 128 points, a multiple of 16, whose
// operands fit a CTA's shared memory.  Its tile is written for that width, the learned
// start's: four rows of 32 channels are the 128 lines of an MMA.  16 channels would take
// eight rows a tile (and twice the spectral operand), which is not written: their SIMT
// rows halve the time of the former layers, whose 1 x 1 products alone ran on the tensor
// cores (64^3, 12 modes, four samples: forward 2.35 -> 0.96 ms).
bool use_tc(const fh_fno* f, const fhrow::RowArgs& a) {
  const FnoDims& d = f->d;
  const int Kp = (2 * d.m + 15) & ~15;
  return f->tensor_cores && d.W == fhtc::kTcW && a.Cin == fhtc::kTcW && a.a_bf16 && a.Iy && !a.Q && d.N % 16 == 0 &&
         fhtc::tc_layout(d.N, Kp).total + 1024 <= 227 * 1024;
}

// a hidden layer's rows, on the tensor cores where that applies
template <int EPI>
fh_status hidden_rows(fh_fno* f, fhrow::RowArgs& a, int* blocks = nullptr) {
  if (!use_tc(f, a)) return launch_rows<EPI>(f, a, blocks);
  const FnoDims& d = f->d;
  fhtc::TcArgs t{};
  t.N = d.N; t.N3 = d.N3; t.N2 = a.N2; t.m2 = 2 * d.m;
  t.Kp = (t.m2 + 15) & ~15;
  t.ntiles = a.nrows / fhtc::kTcRows;   // N^2 rows a sample, N a multiple of 16
  t.ncols = 32;
  while (t.ncols < d.N + t.Kp) t.ncols *= 2;
  t.in = a.in; t.W = reinterpret_cast<const __nv_bfloat16*>(a.A); t.trans = a.a_trans; t.bias = a.bias;
  t.Iy = a.Iy; t.T = a.T; t.u_in = a.u_in; t.u_out = a.u_out; t.out = a.out; t.Yz = a.Yz; t.err = f->tc_err;
  const size_t sm = fhtc::tc_layout(d.N, t.Kp).total;
  FCK(prepare(f, (const void*)fhtc::k_rows_tc<EPI>, fhtc::kTcThreads, sm));
  // two CTAs share an SM where their shared memory allows (tensor memory has 512 columns)
  const int res = 2 * (sm + 2048) <= 228 * 1024 && 2 * t.ncols <= 512 ? 2 : 1;
  fhtc::k_rows_tc<EPI><<<std::min(t.ntiles, res * f->sms), fhtc::kTcThreads, sm, f->stream>>>(t);
  FCK(cudaGetLastError());
  return FH_OK;
}

// a tensor-core layer whose bounded wait gave up leaves an error word
fh_status tc_status(fh_fno* f) {
  int h = 0;
  FCK(cudaMemcpy(&h, f->tc_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (h != 0) {
    FCK(cudaMemset(f->tc_err, 0, sizeof(int)));
    fh::set_error("a tensor-core layer's wait for its MMAs gave up");
    return FH_ERR_TIMEOUT;
  }
  return FH_OK;
}

// kz per block of the y transforms: enough columns for one task per thread
int y_group(const FnoDims& d, int tasks_per_kz, size_t bytes_per_kz) {
  int kb = std::max(1, std::min(d.m, fhspec::kSpecThreads / std::max(1, tasks_per_kz)));
  while (kb > 1 && kb * bytes_per_kz > 64 * 1024) --kb;
  return kb;
}

fhspec::SpecDiv spec_div(const FnoDims& d) {
  using fhrow::make_udiv;
  const unsigned np = d.N / 2 + 1, W = d.W;
  return {make_udiv(W), make_udiv(np), make_udiv(d.m / 4 + 1), make_udiv((np + 3) / 4), make_udiv(d.m + 1), make_udiv(2 * d.m),
          make_udiv(d.m > 1 ? d.m - 1 : 1), make_udiv(W * W), make_udiv(W * W >= 4 ? W * W / 4 : 1)};
}

fh_status dft_y(fh_fno* f, int B) {
  const FnoDims& d = f->d;
  const size_t per = (size_t)2 * (d.N / 2 + 1) * d.W * sizeof(float2);
  const int kb = y_group(d, (d.m / 4 + 1) * d.W, per);
  const size_t sm = d.N * sizeof(float2) + kb * per;
  FCK(prepare(f, (const void*)fhspec::k_dft_y, fhspec::kSpecThreads, sm));
  fhspec::k_dft_y<<<B * d.N * ((d.m + kb - 1) / kb), fhspec::kSpecThreads, sm, f->stream>>>(
      d.N, d.m, d.W, kb, spec_div(d), f->Yz, f->Yy, f->tw);
  FCK(cudaGetLastError());
  return FH_OK;
}

fh_status idft_y(fh_fno* f, int B, float scale, int wz) {
  const FnoDims& d = f->d;
  const size_t per = (size_t)2 * d.m * d.W * sizeof(float2);
  const int kb = y_group(d, (d.N / 8 + 1) * d.W, per);
  const size_t sm = d.N * sizeof(float2) + kb * per;
  FCK(prepare(f, (const void*)fhspec::k_idft_y, fhspec::kSpecThreads, sm));
  fhspec::k_idft_y<<<B * d.N * ((d.m + kb - 1) / kb), fhspec::kSpecThreads, sm, f->stream>>>(
      d.N, d.m, d.W, kb, spec_div(d), f->Yy, f->Yz, f->tw, scale, wz);
  FCK(cudaGetLastError());
  return FH_OK;
}

// DFT along x, mixing with layer l's matrices, inverse DFT along x (in place on Yy)
template <bool BACK>
fh_status mix_x(fh_fno* f, int B, int l, float scale) {
  const FnoDims& d = f->d;
  const int m2 = 2 * d.m;
  const size_t per_b = ((size_t)2 * (d.N / 2 + 1) + (BACK ? 2 : 1) * m2) * d.W * sizeof(float2);
  const size_t per_r = (size_t)d.W * (d.W + 1) * sizeof(__nv_bfloat162);
  // two blocks per SM: two samples at a time, the matrices in what is left of half the shared memory
  const size_t half = 110 * 1024;
  const int bc = B > 1 && 2 * per_b + per_r <= half ? 2 : 1;
  const size_t base = d.N * sizeof(float2) + bc * per_b;
  const int rs = (int)std::max<size_t>(1, std::min<size_t>(m2, base < half ? (half - base) / per_r : 1));
  const size_t sm = base + rs * per_r;
  FCK(prepare(f, (const void*)fhspec::k_mix_x<BACK>, fhspec::kSpecThreads, sm));
  fhspec::k_mix_x<BACK><<<m2 * d.m, fhspec::kSpecThreads, sm, f->stream>>>(
      d.N, d.m, d.W, B, bc, rs, spec_div(d), reinterpret_cast<const __nv_bfloat162*>(f->Rbf) + (size_t)l * d.NM * d.W * d.W, f->Yy,
      f->vh + (size_t)l * B * d.NM * d.W,
      BACK ? reinterpret_cast<float2*>(f->grd + f->off_R) + (size_t)l * d.NM * d.W * d.W : nullptr, f->tw, scale);
  FCK(cudaGetLastError());
  return FH_OK;
}

// the network's forward; `y` receives the output, or with `target` (training) the
// pre-activations are kept and the output's error gradient goes to gy (block sums
// of the squared error to part, *blocks of them)
fh_status forward_all(fh_fno* f, int B, const float* x, float* y, const float* target, int* blocks) {
  const FnoDims& d = f->d;
  const size_t act = (size_t)B * d.W * d.N3;
  fhrow::RowArgs a = row_args(f, B, d.cin, x, f->prm + f->off_P, false, false, f->prm + f->off_p);
  a.out = f->v;
  a.Yz = f->Yz;
  fh_status rc = launch_rows<0>(f, a);
  for (int l = 0; l < d.L && rc == FH_OK; ++l) {
    if ((rc = dft_y(f, B)) != FH_OK) return rc;
    if ((rc = mix_x<false>(f, B, l, 1.f)) != FH_OK) return rc;
    if ((rc = idft_y(f, B, 1.f / (float)d.N3, 1)) != FH_OK) return rc;
    a = row_args(f, B, d.W, f->v + (size_t)l * act, f->Wbf + (size_t)l * d.W * d.W, true, false,
                 f->prm + f->off_w + (size_t)l * d.W);
    a.Iy = f->Yz;
    if (target) a.u_out = f->u + (size_t)l * act;
    if (l + 1 < d.L || target) a.out = f->v + (size_t)(l + 1) * act;
    if (l + 1 < d.L) {
      a.Yz = f->Yz;
    } else {
      a.Q = f->prm + f->off_Q;
      a.qb = f->prm + f->off_q;
      a.cout = d.cout;
      if (target) {
        a.target = target;
        a.gy = f->gy;
        a.part = f->part;
        a.inv_count = 1.f / (float)((long long)B * d.cout * d.N3);
      } else {
        a.y = y;
      }
    }
    rc = a.target ? launch_rows<3>(f, a, blocks) : hidden_rows<1>(f, a, blocks);
  }
  return rc;
}

fh_status weight_grad(fh_fno* f, int B, int cin, int cout, const float* g, const float* x, long long off_A, long long off_b) {
  const FnoDims& d = f->d;
  const int total = B * d.N3;   // at most 64 * 128^3
  const int to = cout <= 8 ? 8 : 32, tc = cin <= 8 ? 8 : 32;
  const int tiles = ((cout + to - 1) / to) * ((cin + tc - 1) / tc);
  const int chunks = (total + fhrow::kWgVox - 1) / fhrow::kWgVox;
  const int vec = d.N3 % 4 == 0 && aligned16(g) && aligned16(x);
  const dim3 grid(std::min(chunks, 2 * f->sms), tiles);
  auto launch = [&](auto kernel) {
    kernel<<<grid, fhrow::kWgThreads, 0, f->stream>>>(total, d.N3, cin, cout, vec, g, x, f->grd + off_A, f->grd + off_b);
  };
  if (to == 8) launch(tc == 8 ? fhrow::k_weight_grad<8, 8> : fhrow::k_weight_grad<8, 32>);
  else launch(tc == 8 ? fhrow::k_weight_grad<32, 8> : fhrow::k_weight_grad<32, 32>);
  FCK(cudaGetLastError());
  return FH_OK;
}

// the tensor-core rows' share of an SM's shared memory and L1 cache
cudaError_t prefer_shared() {
  for (const void* k : {(const void*)fhtc::k_rows_tc<0>, (const void*)fhtc::k_rows_tc<1>, (const void*)fhtc::k_rows_tc<2>}) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

fh_status refresh_bf16(fh_fno* f) {
  const FnoDims& d = f->d;
  const long long nW = (long long)d.L * d.W * d.W, nR = (long long)d.L * d.NM * d.W * d.W * 2;
  k_to_bf16<<<grid_for(nW), kT, 0, f->stream>>>(nW, f->prm + f->off_W, f->Wbf);
  k_to_bf16<<<grid_for(nR), kT, 0, f->stream>>>(nR, f->prm + f->off_R, f->Rbf);
  FCK(cudaGetLastError());
  return FH_OK;
}

}  // namespace

extern "C" {

fh_status fh_fno_create(int n, int cin, int cout, int width, int modes, int layers, int max_batch, void* stream,
                        fh_fno** out) {
  if (!out) { fh::set_error("null argument"); return FH_ERR_ARG; }
  if (n < 4 || n > 128 || cin < 1 || cin > 64 || cout < 1 || cout > 64 || width < 1 || width > 64 || modes < 1 ||
      2 * modes > n || layers < 1 || layers > 8 || max_batch < 1 || max_batch > 64) {
    fh::set_error("FNO sizes out of range (n<=128, channels<=64, 2*modes<=n, layers<=8, batch<=64)");
    return FH_ERR_ARG;
  }
  // a limit of the interface, not of the kernels (which go further)
  if (width * (width + 2 * max_batch) > 3632) {
    fh::set_error("FNO width/batch too large: width (width + 2 max_batch) must not exceed 3632");
    return FH_ERR_UNSUPPORTED;
  }
  fh_fno* f = new fh_fno();
  FnoDims& d = f->d;
  d.N = n; d.cin = cin; d.cout = cout; d.W = width; d.m = modes; d.L = layers;
  d.N3 = n * n * n;
  d.NM = 4 * modes * modes * modes;
  f->max_batch = max_batch;
  f->stream = reinterpret_cast<cudaStream_t>(stream);
  long long o = 0;
  f->off_P = o; o += (long long)width * cin;
  f->off_p = o; o += width;
  f->off_W = o; o += (long long)layers * width * width;
  f->off_w = o; o += (long long)layers * width;
  f->off_R = o; o += (long long)layers * d.NM * width * width * 2;
  f->off_Q = o; o += (long long)cout * width;
  f->off_q = o; o += cout;
  f->nparam = o;
  auto fail = [&](cudaError_t e) {
    fh::set_error(std::string("FNO allocation: ") + cudaGetErrorString(e));
    fh_fno_destroy(f);
    return FH_ERR_CUDA;
  };
  cudaError_t e;
  const size_t act = (size_t)max_batch * width * d.N3;
  if ((e = cudaMalloc(&f->prm, o * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->grd_mem, (o + 3) * 4)) != cudaSuccess) return fail(e);
  f->grd = f->grd_mem + (4 - f->off_R % 4) % 4;
  if ((e = cudaMalloc(&f->m1, o * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->m2, o * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->Wbf, (size_t)layers * width * width * 2)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->Rbf, (size_t)layers * d.NM * width * width * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->tw, (size_t)n * 8)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->zt, (size_t)2 * modes * n * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->v, (layers + 1) * act * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->u, layers * act * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->vh, (size_t)layers * max_batch * width * d.NM * 8)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->Yz, (size_t)max_batch * width * n * n * 2 * modes * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->Yy, (size_t)max_batch * width * n * 2 * modes * modes * 8)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->y, (size_t)max_batch * cout * d.N3 * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->gy, (size_t)max_batch * cout * d.N3 * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->ga, act * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->gb, act * 4)) != cudaSuccess) return fail(e);
  if ((e = cudaGetDevice(&f->device)) != cudaSuccess) return fail(e);
  if ((e = cudaDeviceGetAttribute(&f->sms, cudaDevAttrMultiProcessorCount, f->device)) != cudaSuccess) return fail(e);
  if ((e = prefer_shared()) != cudaSuccess) return fail(e);
  f->nparts = 8 * f->sms;   // at least the resident blocks of a row kernel
  if ((e = cudaMalloc(&f->part, f->nparts * sizeof(double))) != cudaSuccess) return fail(e);
  if ((e = cudaMalloc(&f->tc_err, sizeof(int))) != cudaSuccess) return fail(e);
  if ((e = cudaMemset(f->tc_err, 0, sizeof(int))) != cudaSuccess) return fail(e);
  cudaMemset(f->prm, 0, o * 4);
  cudaMemset(f->grd, 0, o * 4);
  cudaMemset(f->m1, 0, o * 4);
  cudaMemset(f->m2, 0, o * 4);
  std::vector<float2> tw(n);
  for (int t = 0; t < n; ++t) {
    const long double a = 2.0L * 3.141592653589793238462643383279502884L * t / n;
    tw[t] = make_float2((float)cosl(a), (float)(-sinl(a)));
  }
  if ((e = cudaMemcpy(f->tw, tw.data(), n * 8, cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
  std::vector<float> zt((size_t)2 * modes * n);
  for (int k = 0; k < modes; ++k)
    for (int z = 0; z < n; ++z) {
      zt[(size_t)k * n + z] = tw[(k * z) % n].x;
      zt[(size_t)(modes + k) * n + z] = tw[(k * z) % n].y;
    }
  if ((e = cudaMemcpy(f->zt, zt.data(), zt.size() * 4, cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
  *out = f;
  return FH_OK;
}

void fh_fno_destroy(fh_fno* f) {
  if (!f) return;
  void* ptrs[] = {f->prm, f->grd_mem, f->m1, f->m2, f->Wbf, f->Rbf, f->tw, f->zt, f->v, f->u, f->vh,
                  f->Yz, f->Yy, f->y, f->gy, f->ga, f->gb, f->part, f->flat, f->tc_err};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete f;
}

fh_status fh_fno_param_count(const fh_fno* f, long long* count) {
  if (!f || !count) { fh::set_error("null argument"); return FH_ERR_ARG; }
  *count = f->nparam;
  return FH_OK;
}

}  // extern "C"

namespace {
// The public parameter vector stores R as all real parts then all imaginary
// parts; the device keeps each complex weight interleaved.
void flat_to_device(const fh_fno* f, const float* flat, std::vector<float>& dev) {
  dev.assign(flat, flat + f->nparam);
  const long long nR = (f->off_Q - f->off_R) / 2;
  for (long long i = 0; i < nR; ++i) {
    dev[f->off_R + 2 * i] = flat[f->off_R + i];
    dev[f->off_R + 2 * i + 1] = flat[f->off_R + nR + i];
  }
}
// A parameter-shaped device vector in the public order: the complex weights are
// taken apart on the device (an HBM pass, 0.1 ms for 57 M parameters) and the copy
// goes straight to the caller's buffer, where a host loop over a second copy took
// five times as long as the copy itself.  Where the device has no room for the second
// vector the host takes them apart.
fh_status copy_out(const fh_fno* fc, const float* src, float* flat) {
  fh_fno* f = const_cast<fh_fno*>(fc);
  std::lock_guard<std::mutex> lock(f->flat_mutex);   // read-outs from several threads share the buffer
  if (!f->flat && cudaMalloc(&f->flat, f->nparam * 4) != cudaSuccess) {
    cudaGetLastError();
    f->flat = nullptr;
    FCK(cudaMemcpyAsync(flat, src, f->nparam * 4, cudaMemcpyDeviceToHost, f->stream));
    FCK(cudaStreamSynchronize(f->stream));
    const long long nR = (f->off_Q - f->off_R) / 2;
    const std::vector<float> R(flat + f->off_R, flat + f->off_Q);
    for (long long i = 0; i < nR; ++i) {
      flat[f->off_R + i] = R[2 * i];
      flat[f->off_R + nR + i] = R[2 * i + 1];
    }
    return FH_OK;
  }
  k_to_flat<<<grid_for(f->nparam), kT, 0, f->stream>>>(f->nparam, f->off_R, (f->off_Q - f->off_R) / 2, src, f->flat);
  FCK(cudaGetLastError());
  FCK(cudaMemcpyAsync(flat, f->flat, f->nparam * 4, cudaMemcpyDeviceToHost, f->stream));
  FCK(cudaStreamSynchronize(f->stream));
  return FH_OK;
}
}  // namespace

extern "C" {

fh_status fh_fno_set_params(fh_fno* f, const float* flat) {
  if (!f || !flat) { fh::set_error("null argument"); return FH_ERR_ARG; }
  std::vector<float> dev;
  flat_to_device(f, flat, dev);
  FCK(cudaMemcpyAsync(f->prm, dev.data(), f->nparam * 4, cudaMemcpyHostToDevice, f->stream));
  fh_status rc = refresh_bf16(f);
  if (rc != FH_OK) return rc;
  FCK(cudaStreamSynchronize(f->stream));
  return FH_OK;
}

fh_status fh_fno_get_params(const fh_fno* f, float* flat) {
  if (!f || !flat) { fh::set_error("null argument"); return FH_ERR_ARG; }
  return copy_out(f, f->prm, flat);
}

fh_status fh_fno_get_grads(const fh_fno* f, float* flat) {
  if (!f || !flat) { fh::set_error("null argument"); return FH_ERR_ARG; }
  return copy_out(f, f->grd, flat);
}

// input channels of one sample: [log10 E(x) / 2, eps0 (n_v constant channels)]
fh_status fh_fno_make_input(const fh_fno* f, const uint8_t* phase, int nphase, const double* phase_logE,
                            const double* eps0, float* x) {
  if (!f || !phase || !phase_logE || !eps0 || !x) { fh::set_error("null argument"); return FH_ERR_ARG; }
  if (nphase < 1 || nphase > 16) { fh::set_error("nphase must be 1..16"); return FH_ERR_ARG; }
  if (f->d.cin != 7 && f->d.cin != 1) {
    fh::set_error("make_input builds 1 channel (log10 E) or 7 (log10 E, 6 strains)");
    return FH_ERR_ARG;
  }
  FeatParams P{};
  for (int q = 0; q < nphase; ++q) P.logE[q] = (float)(0.5 * phase_logE[q]);
  for (int c = 0; c < 6; ++c) P.e0[c] = (float)eps0[c];
  k_features<<<grid_for(f->d.N3), kT, 0, f->stream>>>(f->d.N3, P, phase, x, f->d.cin == 7);
  FCK(cudaGetLastError());
  FCK(cudaStreamSynchronize(f->stream));
  return FH_OK;
}

fh_status fh_fno_zero_grad(fh_fno* f) {
  if (!f) { fh::set_error("null argument"); return FH_ERR_ARG; }
  FCK(cudaMemsetAsync(f->grd, 0, f->nparam * 4, f->stream));
  return FH_OK;
}

fh_status fh_fno_forward(fh_fno* f, int batch, const float* x, float* y) {
  if (!f || !x || !y) { fh::set_error("null argument"); return FH_ERR_ARG; }
  if (batch < 1 || batch > f->max_batch) { fh::set_error("batch out of range"); return FH_ERR_ARG; }
  cudaPointerAttributes attr{};
  const bool known = cudaPointerGetAttributes(&attr, y) == cudaSuccess;
  const bool direct = fh::writes_directly(known && attr.type == cudaMemoryTypeDevice, attr.device, f->device);
  cudaGetLastError();   // a host pointer may leave an error behind on some drivers
  fh_status rc = forward_all(f, batch, x, direct ? y : f->y, nullptr, nullptr);
  if (rc != FH_OK) return rc;
  if (!direct) FCK(cudaMemcpyAsync(y, f->y, (size_t)batch * f->d.cout * f->d.N3 * 4, cudaMemcpyDefault, f->stream));
  FCK(cudaStreamSynchronize(f->stream));
  return tc_status(f);
}

fh_status fh_fno_set_tensor_cores(fh_fno* f, int enable) {
  if (!f || (enable != 0 && enable != 1)) { fh::set_error("null network or enable not 0/1"); return FH_ERR_ARG; }
  f->tensor_cores = enable != 0;
  return FH_OK;
}

fh_status fh_fno_loss_grad(fh_fno* f, int batch, const float* x, const float* target, double* loss) {
  if (!f || !x || !target) { fh::set_error("null argument"); return FH_ERR_ARG; }
  if (batch < 1 || batch > f->max_batch) { fh::set_error("batch out of range"); return FH_ERR_ARG; }
  const FnoDims& d = f->d;
  const long long ny = (long long)batch * d.cout * d.N3;
  int gb = 0;
  fh_status rc = forward_all(f, batch, x, nullptr, target, &gb);
  if (rc != FH_OK) return rc;
  if (gb > f->nparts) { fh::set_error("more row blocks than partial sums"); return FH_ERR_INTERNAL; }
  const size_t act = (size_t)batch * d.W * d.N3;
  // projection: its weights' gradient, then gu = (Q^T gy) gelu'(u) of the last layer
  rc = weight_grad(f, batch, d.W, d.cout, f->gy, f->v + (size_t)d.L * act, f->off_Q, f->off_q);
  if (rc != FH_OK) return rc;
  fhrow::RowArgs a = row_args(f, batch, d.cout, f->gy, f->prm + f->off_Q, false, true, nullptr);
  a.u_in = f->u + (size_t)(d.L - 1) * act;
  float *gu = f->gb, *next = f->ga;
  a.out = gu;
  a.Yz = f->Yz;
  rc = launch_rows<2>(f, a);
  for (int l = d.L - 1; l >= 0 && rc == FH_OK; --l) {
    rc = weight_grad(f, batch, d.W, d.W, gu, f->v + (size_t)l * act, f->off_W + (long long)l * d.W * d.W, f->off_w + (long long)l * d.W);
    if (rc != FH_OK) return rc;
    // spectral adjoint: g = (w / N^3) DFT(gu); gin = R^H g, gR += g conj(vh); its inverse joins W^T gu
    if ((rc = dft_y(f, batch)) != FH_OK) return rc;
    if ((rc = mix_x<true>(f, batch, l, 1.f / (float)d.N3)) != FH_OK) return rc;
    if ((rc = idft_y(f, batch, 1.f, 0)) != FH_OK) return rc;
    a = row_args(f, batch, d.W, gu, f->Wbf + (size_t)l * d.W * d.W, true, true, nullptr);
    a.Iy = f->Yz;
    a.out = next;
    if (l > 0) {
      a.u_in = f->u + (size_t)(l - 1) * act;
      a.Yz = f->Yz;
      rc = hidden_rows<2>(f, a);
    } else {
      rc = hidden_rows<0>(f, a);
    }
    std::swap(gu, next);
  }
  if (rc != FH_OK) return rc;
  // lift
  rc = weight_grad(f, batch, d.cin, d.W, gu, x, f->off_P, f->off_p);
  if (rc != FH_OK) return rc;
  std::vector<double> parts(gb);
  FCK(cudaMemcpyAsync(parts.data(), f->part, gb * sizeof(double), cudaMemcpyDeviceToHost, f->stream));
  FCK(cudaStreamSynchronize(f->stream));
  if (loss) {
    double s = 0.0;
    for (double p : parts) s += p;
    *loss = s / (double)ny;
  }
  return tc_status(f);
}

fh_status fh_fno_adam_step(fh_fno* f, float lr, float beta1, float beta2, float eps, int step) {
  if (!f || step < 1) { fh::set_error("bad argument"); return FH_ERR_ARG; }
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adam<<<grid_for(f->nparam), kT, 0, f->stream>>>(f->nparam, f->prm, f->grd, f->m1, f->m2, lr, beta1, beta2, eps, c1, c2);
  FCK(cudaGetLastError());
  fh_status rc = refresh_bf16(f);
  if (rc != FH_OK) return rc;
  FCK(cudaStreamSynchronize(f->stream));
  return FH_OK;
}

}  // extern "C"
