// Learned warm start for the interior-point method: an MLP u -> GELU -> GELU -> linear that maps
// problem parameters (here the load vector of the SCOPF-shaped problem) to the solver's primal
// and dual starting point, trained by the library's own kernels:
//   forward   Z_1 = U W_1^T + b_1, H_1 = GELU(Z_1), Z_2 = H_1 W_2^T + b_2, H_2 = GELU(Z_2),
//             P = H_2 W_3^T + b_3                                   (GELU(z) = z Phi(z), erf form)
//   loss      L = mean((P - T)^2) over the batch, on standardized inputs and targets
//   backward  dP = 2 (P - T) / (B n_out); dW_l = dZ_l^T H_{l-1}; db_l = column sums of dZ_l;
//             dH_{l-1} = dZ_l W_l; dZ = dH * GELU'(Z)
//   Adam      (Kingma & Ba) on FP32 master weights, FP32 moments, BF16 operand copies.
// GEMMs: in the BF16 form the products run on the tcgen05 tensor cores (tc_plain: TMA-fed BF16
// operands, FP32 accumulation in tensor memory, bias added in the epilogue); the backward products
// take transposed operand copies written by the GELU, loss, GELU-derivative and Adam kernels.  Shapes the tensor cores cannot take (a batch that is not a multiple of 64 in the
// weight-gradient products, widths that are not multiples of 64) and the FP32 form use a
// shared-memory tiled CUDA-core kernel.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <numeric>
#include <random>
#include <string>
#include <vector>

#include "../../include/nnc.h"
#include "async.cuh"
#include "common.cuh"
#include "tc.cuh"

namespace nnc {
void set_last_error(const std::string& msg);
}
using namespace nnc;
using async::griddep_launch;
using async::griddep_wait;

namespace {

// C[m][n] = sum_k A(m, k) B(k, n) (+ bias[n]); A(m, k) = A[m * sam + k * sak] and likewise B,
// inputs of type T (BF16 or FP32), FP32 accumulation; optional GELU epilogue writes Z and H.
template <typename T>
__device__ __forceinline__ float ld(const T* p) {
  if constexpr (std::is_same<T, float>::value) return *p;
  else return __bfloat162float(*p);
}

// One 32 x 32 tile per CTA, 2 x 2 outputs a thread, the next K slice in registers while this one is
// multiplied.  Bound: latency (the products are small); 32 x 32 tiles give a 64 x 256 product 16 CTAs
// where 64 x 64 tiles gave it 4.
template <typename T>
__global__ void __launch_bounds__(256) k_ws_gemm(const T* __restrict__ A, long sam, long sak,
                                                 const T* __restrict__ B, long sbk, long sbn, int M,
                                                 int N, int K, const float* __restrict__ bias,
                                                 float* __restrict__ C, int ldc) {
  __shared__ float As[32][33], Bs[32][33];
  const int ntn = (N + 31) / 32;   // one grid dimension: the others end at 65535 tiles
  const int m0 = blockIdx.x / ntn * 32, n0 = blockIdx.x % ntn * 32;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int lo = threadIdx.x & 31, hi = threadIdx.x >> 5;   // neighbouring threads: neighbouring addresses
  float ra[4], rb[4];
  auto load = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int o = hi + 8 * j;
      const int ak = k0 + (sak == 1 ? lo : o), am = m0 + (sak == 1 ? o : lo);
      ra[j] = am < M && ak < K ? ld(A + am * sam + ak * sak) : 0.f;
      const int bk = k0 + (sbk == 1 ? lo : o), bn = n0 + (sbk == 1 ? o : lo);
      rb[j] = bn < N && bk < K ? ld(B + bk * sbk + bn * sbn) : 0.f;
    }
  };
  float acc[2][2] = {};
  griddep_wait();
  griddep_launch();
  load(0);
  for (int k0 = 0; k0 < K; k0 += 32) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int o = hi + 8 * j;
      if (sak == 1) As[lo][o] = ra[j];
      else As[o][lo] = ra[j];
      if (sbk == 1) Bs[lo][o] = rb[j];
      else Bs[o][lo] = rb[j];
    }
    __syncthreads();
    if (k0 + 32 < K) load(k0 + 32);
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) {
      const float a0 = As[kk][tx], a1 = As[kk][tx + 16], b0 = Bs[kk][ty], b1 = Bs[kk][ty + 16];
      acc[0][0] = fmaf(a0, b0, acc[0][0]);
      acc[0][1] = fmaf(a0, b1, acc[0][1]);
      acc[1][0] = fmaf(a1, b0, acc[1][0]);
      acc[1][1] = fmaf(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = m0 + tx + 16 * i;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int n = n0 + ty + 16 * j;
      if (m < M && n < N) C[(size_t)m * ldc + n] = acc[i][j] + (bias ? bias[n] : 0.f);
    }
  }
}

template <typename T>
cudaError_t gemm(const T* A, long sam, long sak, const T* B, long sbk, long sbn, int M, int N, int K,
                 const float* bias, float* C, int ldc, cudaStream_t st) {
  const long long tiles = (N + 31LL) / 32 * ((M + 31LL) / 32);
  if (tiles > INT_MAX) return cudaErrorInvalidValue;
  return launch_pdl(k_ws_gemm<T>, dim3((unsigned)tiles), dim3(256), 0, st, A, sam, sak, B, sbk, sbn, M, N, K, bias, C, ldc);
}

template <typename T>
__device__ __forceinline__ T to_op(float v) {
  if constexpr (std::is_same<T, float>::value) return v;
  else return __float2bfloat16_rn(v);
}

// H = GELU(Z) in the operand type (and, for the tensor-core backward products, its transposed copy) and
// D1 = GELU'(Z).  Bound: the FP64 pipe, two FMAs per clock and SM, so the elements are spread over the
// whole chip in CTAs of 64.  In the epilogue of the product the 64 x 256 values were one SM's work, and
// with them a training step of 64 rows (512 -> 256 -> 256 -> 713) took 1.1 ms; now 0.08 ms.
template <typename T>
__global__ void __launch_bounds__(64) k_ws_gelu(const float* __restrict__ Z, int n, T* __restrict__ Hl,
                                                float* __restrict__ D1, int cols,
                                                __nv_bfloat16* __restrict__ Ht, int ldt) {
  griddep_wait();
  griddep_launch();
  const int i = blockIdx.x * 64 + threadIdx.x;
  if (i >= n) return;
  double a, d1, d2;
  act_eval(NNC_GELU, (double)Z[i], a, d1, d2);
  const T h = to_op<T>((float)a);
  Hl[i] = h;
  D1[i] = (float)d1;
  if constexpr (!std::is_same<T, float>::value)
    if (Ht) Ht[(size_t)(i % cols) * ldt + i / cols] = h;
}

// Writes v of rows b .. b + 7 of one column of a transposed copy (16 bytes; ldt and b multiples of 8).
__device__ __forceinline__ void put8(__nv_bfloat16* dst, const float (&v)[8]) {
  __nv_bfloat162 h[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
  *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(h);
}

// dZ = dH * GELU'(Z) in the operand type and transposed, db[j] = sum_b dZ[b][j]: one thread per column,
// rows in order, eight loads in flight.
template <typename T>
__global__ void __launch_bounds__(32) k_ws_gelu_back(const float* __restrict__ dH,
                                                     const float* __restrict__ D1, int B, int cols,
                                                     T* __restrict__ dZl, float* __restrict__ db,
                                                     __nv_bfloat16* __restrict__ dZt, int ldt) {
  griddep_wait();
  griddep_launch();
  const int j = blockIdx.x * 32 + threadIdx.x;
  if (j >= cols) return;
  float s = 0.f;
  for (int b0 = 0; b0 < B; b0 += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const size_t o = (size_t)(b0 + u) * cols + j;
      v[u] = b0 + u < B ? __fmul_rn(dH[o], D1[o]) : 0.f;   // rounded before it is summed
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (b0 + u < B) {
        s += v[u];
        dZl[(size_t)(b0 + u) * cols + j] = to_op<T>(v[u]);
      }
    }
    if (dZt) put8(dZt + (size_t)j * ldt + b0, v);
  }
  db[j] = s;
}

// dP = 2 (P - T) / (B n_out) in the operand type and in the layouts of the tensor-core products (row
// stride padded to a multiple of 64, the padding stays zero; transposed), its column sums db and the
// loss's column sums part[j]: one thread per column as above.
template <typename T>
__global__ void __launch_bounds__(32) k_ws_loss(const float* __restrict__ P, const float* __restrict__ Tt,
                                                int B, int cols, float scale, T* __restrict__ dPl,
                                                float* __restrict__ db, double* __restrict__ part,
                                                __nv_bfloat16* __restrict__ dPp, int ldp,
                                                __nv_bfloat16* __restrict__ dPt, int ldt) {
  griddep_wait();
  griddep_launch();
  const int j = blockIdx.x * 32 + threadIdx.x;
  if (j >= cols) return;
  double l = 0.0;
  float s = 0.f;
  for (int b0 = 0; b0 < B; b0 += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const size_t o = (size_t)(b0 + u) * cols + j;
      v[u] = b0 + u < B ? P[o] - Tt[o] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      l += (double)v[u] * v[u];
      v[u] = __fmul_rn(2.f * v[u], scale);
      if (b0 + u < B) {
        s += v[u];
        if (dPp) dPp[(size_t)(b0 + u) * ldp + j] = __float2bfloat16_rn(v[u]);
        else dPl[(size_t)(b0 + u) * cols + j] = to_op<T>(v[u]);
      }
    }
    if (dPt) put8(dPt + (size_t)j * ldt + b0, v);
  }
  part[j] = l;
  db[j] = s;
}

// Adam on the six parameter arrays in one launch; refreshes a weight matrix's operand copy wl and, with
// wt given, its transposed BF16 copy (`cols` columns, row stride ldt).
struct AdamSeg {
  float *w, *m, *v;
  const float* g;
  void* wl;
  __nv_bfloat16* wt;
  int n, cols, ldt, blk0;   // blk0: the array's first block of 256 elements
};
struct AdamArgs {
  AdamSeg a[6];
  float lr, b1, b2, eps, c1, c2;
};
template <typename T>
__global__ void __launch_bounds__(256) k_ws_adam(const __grid_constant__ AdamArgs p) {
  griddep_wait();
  griddep_launch();
  int k = 5;
  while ((int)blockIdx.x < p.a[k].blk0) --k;
  const AdamSeg& q = p.a[k];
  const int i = ((int)blockIdx.x - q.blk0) * 256 + threadIdx.x;
  if (i >= q.n) return;
  const float gi = q.g[i];
  const float mi = fmaf(1.f - p.b1, gi, __fmul_rn(p.b1, q.m[i]));
  const float vi = fmaf(__fmul_rn(1.f - p.b2, gi), gi, __fmul_rn(p.b2, q.v[i]));
  q.m[i] = mi;
  q.v[i] = vi;
  const float wi = q.w[i] - p.lr * (mi / p.c1) / (sqrtf(vi / p.c2) + p.eps);
  q.w[i] = wi;
  if (q.wl) ((T*)q.wl)[i] = to_op<T>(wi);
  if (q.wt) q.wt[(size_t)(i % q.cols) * q.ldt + i / q.cols] = __float2bfloat16_rn(wi);
}

// One batch: rows idx[0 .. B) of the standardized inputs (operand type, transposed copy) and targets.
template <typename T>
__global__ void __launch_bounds__(256) k_ws_gather(const float* __restrict__ Ud, const float* __restrict__ Td,
                                                   const int* __restrict__ idx, int n_in, int n_out,
                                                   T* __restrict__ Ul, __nv_bfloat16* __restrict__ Ut,
                                                   int ldt, float* __restrict__ Tt) {
  griddep_wait();
  griddep_launch();
  const int per_row = (n_in + n_out + 255) / 256;   // blocks
  const int r = blockIdx.x / per_row, c = blockIdx.x % per_row * 256 + threadIdx.x;
  const size_t row = idx[r];
  if (c < n_in) {
    const float v = Ud[row * n_in + c];
    Ul[(size_t)r * n_in + c] = to_op<T>(v);
    if (Ut) Ut[(size_t)c * ldt + r] = __float2bfloat16_rn(v);
  } else if (c < n_in + n_out) {
    Tt[(size_t)r * n_out + c - n_in] = Td[row * n_out + c - n_in];
  }
}

// Mean and standard deviation of each column of X [N][cols], rows in order, 16 loads in flight.  The rows
// may come in several parts, rows [r0, r0 + n) of N at a time: all of them with pass = 0, then again with
// pass = 1.  With pass = 2 X is all N rows and one launch does both.
__global__ void __launch_bounds__(32) k_ws_stats(const double* __restrict__ X, int pass, int r0, int n, int N,
                                                 int cols, double* __restrict__ mean,
                                                 double* __restrict__ sd) {
  const int j = blockIdx.x * 32 + threadIdx.x;
  if (j >= cols) return;
  double mu = pass != 1 ? (r0 == 0 ? 0.0 : mean[j]) : mean[j], sq = pass != 1 || r0 == 0 ? 0.0 : sd[j];
#pragma unroll 1
  for (int p = pass == 1; p < (pass == 0 ? 1 : 2); ++p) {
    for (int b = 0; b < n; b += 16) {
      double v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = b + u < n ? X[(size_t)(b + u) * cols + j] : 0.0;
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        if (b + u >= n) break;
        if (p == 0) mu += v[u];
        else sq += (v[u] - mu) * (v[u] - mu);
      }
    }
    if (p == 0 && r0 + n == N) mu /= N;
  }
  mean[j] = mu;
  if (pass != 0) sd[j] = r0 + n == N ? fmax(sqrt(sq / N), 1e-12) : sq;
}
__global__ void __launch_bounds__(256) k_ws_standardize(const double* __restrict__ X, int cols,
                                                        const double* __restrict__ mean,
                                                        const double* __restrict__ sd,
                                                        float* __restrict__ Y) {
  const int per_row = (cols + 255) / 256;   // blocks
  const int c = blockIdx.x % per_row * 256 + threadIdx.x;
  if (c >= cols) return;
  const size_t o = (size_t)(blockIdx.x / per_row) * cols + c;
  Y[o] = (float)((X[o] - mean[c]) / sd[c]);
}

// dst = src in the operand type; with dstt also the transposed BF16 copy of a rows x cols matrix
template <typename T>
__global__ void k_ws_cast(const float* __restrict__ src, int n, T* __restrict__ dst, int cols = 1,
                          __nv_bfloat16* __restrict__ dstt = nullptr, int ldt = 0) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if constexpr (std::is_same<T, float>::value) dst[i] = src[i];
  else dst[i] = __float2bfloat16_rn(src[i]);
  if (dstt) dstt[(size_t)(i % cols) * ldt + i / cols] = __float2bfloat16_rn(src[i]);
}

int wfail(int code, const std::string& m) {
  set_last_error(m);
  return code;
}
#define WCK(expr)                                                                            \
  do {                                                                                       \
    cudaError_t e_ = (expr);                                                                 \
    if (e_ != cudaSuccess) return wfail(NNC_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_)); \
  } while (0)

}  // namespace

struct nnc_ws {
  int n_in = 0, h1 = 0, h2 = 0, n_out = 0, prec = NNC_BF16;
  int sizes[6];
  float *w[6] = {}, *g[6] = {}, *m[6] = {}, *v[6] = {};
  void* wl[6] = {};                // operand copies (BF16 or FP32)
  std::vector<double> in_mean, in_std, out_mean, out_std;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<void*> allocs;
  long long step = 0;
  // batch workspace (capacity cap rows)
  int cap = 0;
  float *U = nullptr, *Tt = nullptr, *Z1 = nullptr, *D1 = nullptr, *Z2 = nullptr, *D2 = nullptr,
        *P = nullptr, *dH = nullptr;   // D1, D2: GELU' of the two hidden layers
  void *Ul = nullptr, *H1l = nullptr, *H2l = nullptr, *dPl = nullptr, *dZl = nullptr;
  double* part = nullptr;   // [n_out] the loss's column sums
  // training set on the device (capacity nd rows): standardized, the epoch's order, the means and
  // deviations of the columns [2][n_in + n_out], and nr rows of it as given
  float *Ud = nullptr, *Td = nullptr;
  int* perm = nullptr;
  double *Ur = nullptr, *Tr = nullptr, *stats = nullptr;
  int nd = 0, nr = 0;
  // tensor-core path (BF16 form with n_in, h1, h2 multiples of 64): transposed BF16 operand copies
  // (row stride cap), dP with its row stride padded to n_out_p, W2^T and W3^T, and the plans of
  // the eight products (built for `plan_rows` batch rows)
  bool tc = false;
  int n_out_p = 0;
  __nv_bfloat16 *Ut = nullptr, *H1t = nullptr, *H2t = nullptr, *dPt = nullptr, *dZt = nullptr,
                *dPp = nullptr, *W2t = nullptr, *W3t = nullptr;
  int* d_err = nullptr;
  nnc::PlainPlan pl[8];
  int plan_rows = -1;
  int sm_count = 0;
};

namespace {

template <typename X>
int walloc(nnc_ws* s, X** p, size_t n) {
  void* q = nullptr;
  if (cudaMalloc(&q, std::max<size_t>(n, 1) * sizeof(X)) != cudaSuccess) {
    cudaGetLastError();   // reported here, not by the next launch
    return wfail(NNC_ERR_OOM, "cudaMalloc failed");
  }
  cudaMemsetAsync(q, 0, std::max<size_t>(n, 1) * sizeof(X), s->stream);
  s->allocs.push_back(q);
  *p = (X*)q;
  return NNC_OK;
}
#define WAL(p, n)                          \
  do {                                     \
    int r_ = walloc(s, &(p), (n));         \
    if (r_) return r_;                     \
  } while (0)

size_t esz(const nnc_ws* s) { return s->prec == NNC_FP32 ? 4 : 2; }

int ensure_cap(nnc_ws* s, int B) {
  if (B <= s->cap) return NNC_OK;
  if (s->tc) B = (B + 63) / 64 * 64;   // the transposed copies' row stride: a multiple of 64
  const int wmax = std::max(std::max(s->h1, s->h2), std::max(s->n_in, s->n_out));
  const size_t big = (size_t)B * wmax;
  WAL(s->U, big);
  WAL(s->Tt, big);
  WAL(s->Z1, big);
  WAL(s->D1, big);
  WAL(s->Z2, big);
  WAL(s->D2, big);
  WAL(s->P, big);
  WAL(s->dH, big);
  unsigned char* q;
  WAL(q, big * esz(s)); s->Ul = q;
  WAL(q, big * esz(s)); s->H1l = q;
  WAL(q, big * esz(s)); s->H2l = q;
  WAL(q, big * esz(s)); s->dPl = q;
  WAL(q, big * esz(s)); s->dZl = q;
  WAL(s->part, s->n_out);
  if (s->tc) {
    WAL(s->Ut, (size_t)s->n_in * B);
    WAL(s->H1t, (size_t)s->h1 * B);
    WAL(s->H2t, (size_t)s->h2 * B);
    WAL(s->dPt, (size_t)s->n_out * B);
    WAL(s->dZt, (size_t)std::max(s->h1, s->h2) * B);
    WAL(s->dPp, (size_t)B * s->n_out_p);
  }
  s->cap = B;
  s->plan_rows = -1;
  return NNC_OK;
}

// training-set buffers for N rows; a larger set replaces them.  The FP64 rows as given are needed until they
// are standardized: all at once where they take an eighth of the free memory or less, else in parts.
int ensure_set(nnc_ws* s, int N) {
  if (N <= s->nd) return NNC_OK;
  WCK(cudaStreamSynchronize(s->stream));
  for (void* p : {(void*)s->Ur, (void*)s->Tr, (void*)s->Ud, (void*)s->Td, (void*)s->perm}) {
    if (!p) continue;
    s->allocs.erase(std::find(s->allocs.begin(), s->allocs.end(), p));
    cudaFree(p);
  }
  s->Ur = s->Tr = nullptr;
  s->Ud = s->Td = nullptr;
  s->perm = nullptr;
  s->nd = 0;
  WAL(s->Ud, (size_t)N * s->n_in);
  WAL(s->Td, (size_t)N * s->n_out);
  WAL(s->perm, N);
  if (!s->stats) WAL(s->stats, 2 * (size_t)(s->n_in + s->n_out));
  size_t free_b = 0, total_b = 0;
  WCK(cudaMemGetInfo(&free_b, &total_b));
  const size_t row = sizeof(double) * ((size_t)s->n_in + s->n_out);
  s->nr = (int)std::min<size_t>(N, std::max<size_t>(1, free_b / 8 / row));
  WAL(s->Ur, (size_t)s->nr * s->n_in);
  WAL(s->Tr, (size_t)s->nr * s->n_out);
  s->nd = N;
  return NNC_OK;
}

// the eight tensor-core products for batches of B rows (tensor maps of the current buffers)
int make_plans(nnc_ws* s, int B) {
  if (s->plan_rows == B) return NNC_OK;
  using nnc::tc_plain_plan;
  const int cap = s->cap, sms = s->sm_count;
  const __nv_bfloat16* w1 = (const __nv_bfloat16*)s->wl[0];
  const __nv_bfloat16* w2 = (const __nv_bfloat16*)s->wl[2];
  const __nv_bfloat16* w3 = (const __nv_bfloat16*)s->wl[4];
  int r = tc_plain_plan(s->pl[0], s->Ul, B, s->n_in, w1, s->h1, s->n_in, B, s->h1, s->n_in, sms);
  if (!r) r = tc_plain_plan(s->pl[1], s->H1l, B, s->h1, w2, s->h2, s->h1, B, s->h2, s->h1, sms);
  if (!r) r = tc_plain_plan(s->pl[2], s->H2l, B, s->h2, w3, s->n_out, s->h2, B, s->n_out, s->h2, sms);
  if (!r && B % 64 == 0) {
    r = tc_plain_plan(s->pl[3], s->dPt, s->n_out, cap, s->H2t, s->h2, cap, s->n_out, s->h2, B, sms);
    if (!r) r = tc_plain_plan(s->pl[4], s->dPp, B, s->n_out_p, s->W3t, s->h2, s->n_out_p, B, s->h2, s->n_out_p, sms);
    if (!r) r = tc_plain_plan(s->pl[5], s->dZt, s->h2, cap, s->H1t, s->h1, cap, s->h2, s->h1, B, sms);
    if (!r) r = tc_plain_plan(s->pl[6], s->dZl, B, s->h2, s->W2t, s->h1, s->h2, B, s->h1, s->h2, sms);
    if (!r) r = tc_plain_plan(s->pl[7], s->dZt, s->h1, cap, s->Ut, s->n_in, cap, s->h1, s->n_in, B, sms);
  }
  if (r) return wfail(r, "warm start: tensor-core plan failed");
  s->plan_rows = B;
  return NNC_OK;
}
#define TCK(expr)                                                                            \
  do {                                                                                       \
    cudaError_t e_ = (expr);                                                                 \
    if (e_ != cudaSuccess) return wfail(NNC_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <typename T>
cudaError_t gelu(nnc_ws* s, const float* Z, int B, int cols, void* Hl, float* D1, __nv_bfloat16* Ht) {
  const int rows = std::max(1, (1 << 30) / cols);   // of a launch, whose elements an int counts
  for (int r = 0; r < B; r += rows) {
    const int n = std::min(rows, B - r) * cols;
    const size_t o = (size_t)r * cols;
    const cudaError_t e = launch_pdl(k_ws_gelu<T>, dim3((n + 63) / 64), dim3(64), 0, s->stream, Z + o, n,
                                     (T*)Hl + o, D1 + o, cols, Ht ? Ht + r : nullptr, s->cap);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// forward on the first B rows of s->Ul (operand type): P = net(U)
template <typename T>
int forward(nnc_ws* s, int B) {
  cudaStream_t st = s->stream;
  if constexpr (!std::is_same<T, float>::value) {
    if (s->tc) {
      int r = make_plans(s, B);
      if (r) return r;
      TCK(nnc::tc_plain(s->pl[0], s->w[1], s->Z1, s->h1, s->d_err, st));
      TCK(gelu<T>(s, s->Z1, B, s->h1, s->H1l, s->D1, s->H1t));
      TCK(nnc::tc_plain(s->pl[1], s->w[3], s->Z2, s->h2, s->d_err, st));
      TCK(gelu<T>(s, s->Z2, B, s->h2, s->H2l, s->D2, s->H2t));
      TCK(nnc::tc_plain(s->pl[2], s->w[5], s->P, s->n_out, s->d_err, st));
      return NNC_OK;
    }
  }
  TCK(gemm<T>((const T*)s->Ul, s->n_in, 1, (const T*)s->wl[0], 1, s->n_in, B, s->h1, s->n_in, s->w[1], s->Z1,
          s->h1, st));
  TCK(gelu<T>(s, s->Z1, B, s->h1, s->H1l, s->D1, nullptr));
  TCK(gemm<T>((const T*)s->H1l, s->h1, 1, (const T*)s->wl[2], 1, s->h1, B, s->h2, s->h1, s->w[3], s->Z2, s->h2,
          st));
  TCK(gelu<T>(s, s->Z2, B, s->h2, s->H2l, s->D2, nullptr));
  TCK(gemm<T>((const T*)s->H2l, s->h2, 1, (const T*)s->wl[4], 1, s->h2, B, s->n_out, s->h2, s->w[5], s->P,
          s->n_out, st));
  return NNC_OK;
}

// loss and gradients on the first B rows (targets in s->Tt); returns the loss through *loss
template <typename T>
int loss_grad(nnc_ws* s, int B, double* loss) {
  cudaStream_t st = s->stream;
  int rf = forward<T>(s, B);
  if (rf) return rf;
  const int nP = B * s->n_out;
  // tensor-core backward products need the batch (their K) to be a multiple of 64
  const bool tcb = !std::is_same<T, float>::value && s->tc && B % 64 == 0;
  __nv_bfloat16* dZt = tcb ? s->dZt : nullptr;
  auto back = [&](const float* D, int cols, float* db) {
    return launch_pdl(k_ws_gelu_back<T>, dim3((cols + 31) / 32), dim3(32), 0, st, s->dH, D, B, cols,
                      (T*)s->dZl, db, dZt, s->cap);
  };
  TCK(launch_pdl(k_ws_loss<T>, dim3((s->n_out + 31) / 32), dim3(32), 0, st, s->P, s->Tt, B, s->n_out,
                 1.f / (float)nP, (T*)s->dPl, s->g[5], s->part, tcb ? s->dPp : nullptr, s->n_out_p,
                 tcb ? s->dPt : nullptr, s->cap));
  // layer by layer: dW = dZ^T H (db with dZ), dH = dZ W, dZ = dH * GELU'
  if (tcb) {
    TCK(nnc::tc_plain(s->pl[3], nullptr, s->g[4], s->h2, s->d_err, st));
    TCK(nnc::tc_plain(s->pl[4], nullptr, s->dH, s->h2, s->d_err, st));
    TCK(back(s->D2, s->h2, s->g[3]));
    TCK(nnc::tc_plain(s->pl[5], nullptr, s->g[2], s->h1, s->d_err, st));
    TCK(nnc::tc_plain(s->pl[6], nullptr, s->dH, s->h1, s->d_err, st));
    TCK(back(s->D1, s->h1, s->g[1]));
    TCK(nnc::tc_plain(s->pl[7], nullptr, s->g[0], s->n_in, s->d_err, st));
  } else {
    TCK(gemm<T>((const T*)s->dPl, 1, s->n_out, (const T*)s->H2l, s->h2, 1, s->n_out, s->h2, B, nullptr, s->g[4],
            s->h2, st));
    TCK(gemm<T>((const T*)s->dPl, s->n_out, 1, (const T*)s->wl[4], s->h2, 1, B, s->h2, s->n_out, nullptr, s->dH,
            s->h2, st));
    TCK(back(s->D2, s->h2, s->g[3]));
    TCK(gemm<T>((const T*)s->dZl, 1, s->h2, (const T*)s->H1l, s->h1, 1, s->h2, s->h1, B, nullptr, s->g[2], s->h1,
            st));
    TCK(gemm<T>((const T*)s->dZl, s->h2, 1, (const T*)s->wl[2], s->h1, 1, B, s->h1, s->h2, nullptr, s->dH, s->h1,
            st));
    TCK(back(s->D1, s->h1, s->g[1]));
    TCK(gemm<T>((const T*)s->dZl, 1, s->h1, (const T*)s->Ul, s->n_in, 1, s->h1, s->n_in, B, nullptr, s->g[0],
            s->n_in, st));
  }
  if (loss) {
    std::vector<double> h(s->n_out);
    WCK(cudaMemcpyAsync(h.data(), s->part, sizeof(double) * s->n_out, cudaMemcpyDeviceToHost, st));
    WCK(cudaStreamSynchronize(st));
    double t = 0;
    for (double x : h) t += x;
    *loss = t / nP;
  }
  return NNC_OK;
}

template <typename T>
cudaError_t adam(nnc_ws* s, float lr, float b1, float b2, float eps) {
  s->step += 1;
  AdamArgs p{};
  p.lr = lr;
  p.b1 = b1;
  p.b2 = b2;
  p.eps = eps;
  p.c1 = 1.f - std::pow(b1, (float)s->step);
  p.c2 = 1.f - std::pow(b2, (float)s->step);
  int blocks = 0;
  for (int i = 0; i < 6; ++i) {
    // W2^T and W3^T feed the tensor-core backward products
    __nv_bfloat16* wt = !s->tc ? nullptr : i == 2 ? s->W2t : i == 4 ? s->W3t : nullptr;
    p.a[i] = AdamSeg{s->w[i], s->m[i], s->v[i], s->g[i], i % 2 == 0 ? s->wl[i] : nullptr, wt, s->sizes[i],
                     i == 2 ? s->h1 : i == 4 ? s->h2 : 1, i == 2 ? s->h2 : i == 4 ? s->n_out_p : 0, blocks};
    blocks += (s->sizes[i] + 255) / 256;
  }
  return launch_pdl(k_ws_adam<T>, dim3(blocks), dim3(256), 0, s->stream, p);
}

template <typename T>
cudaError_t stage_rows(nnc_ws* s, int B) {
  // s->U (B x n_in) is on the device in standardized FP32
  k_ws_cast<T><<<(B * s->n_in + 255) / 256, 256, 0, s->stream>>>(s->U, B * s->n_in, (T*)s->Ul, s->n_in,
                                                                  s->tc ? s->Ut : nullptr, s->cap);
  note_launch();
  return cudaGetLastError();
}

int upload_std(nnc_ws* s, const double* U, const double* Tt, int N, bool with_t) {
  std::vector<float> hu((size_t)N * s->n_in), ht(with_t ? (size_t)N * s->n_out : 0);
  for (int r = 0; r < N; ++r) {
    for (int c = 0; c < s->n_in; ++c)
      hu[(size_t)r * s->n_in + c] = (float)((U[(size_t)r * s->n_in + c] - s->in_mean[c]) / s->in_std[c]);
    if (with_t)
      for (int c = 0; c < s->n_out; ++c)
        ht[(size_t)r * s->n_out + c] = (float)((Tt[(size_t)r * s->n_out + c] - s->out_mean[c]) / s->out_std[c]);
  }
  int r = ensure_cap(s, N);
  if (r) return r;
  WCK(cudaMemcpyAsync(s->U, hu.data(), sizeof(float) * hu.size(), cudaMemcpyHostToDevice, s->stream));
  if (with_t)
    WCK(cudaMemcpyAsync(s->Tt, ht.data(), sizeof(float) * ht.size(), cudaMemcpyHostToDevice, s->stream));
  WCK(cudaStreamSynchronize(s->stream));
  return NNC_OK;
}

// the tensor-core kernels' bounded waits record an error word; a set word fails the call
int check_ws_err(nnc_ws* s) {
  if (!s->d_err) return NNC_OK;
  int e = 0;
  WCK(cudaMemcpyAsync(&e, s->d_err, sizeof(int), cudaMemcpyDeviceToHost, s->stream));
  WCK(cudaStreamSynchronize(s->stream));
  if (e) {
    cudaMemsetAsync(s->d_err, 0, sizeof(int), s->stream);
    return wfail(NNC_ERR_TIMEOUT, "warm start: a bounded device-side wait ran out");
  }
  return NNC_OK;
}

}  // namespace

extern "C" {

int nnc_ws_create(nnc_ws** out, int n_in, int h1, int h2, int n_out, const double* const* params,
                  int prec, void* stream) {
  if (!out || n_in < 1 || h1 < 1 || h2 < 1 || n_out < 1 || !params || (prec != NNC_BF16 && prec != NNC_FP32))
    return wfail(NNC_ERR_ARG, "nnc_ws_create: bad arguments");
  *out = nullptr;
  nnc_ws* s = new nnc_ws();
  s->n_in = n_in;
  s->h1 = h1;
  s->h2 = h2;
  s->n_out = n_out;
  s->prec = prec;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    delete s;
    return wfail(NNC_ERR_CUDA, "no CUDA device");
  }
  if (stream) s->stream = (cudaStream_t)stream;
  else {
    if (cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete s;
      return wfail(NNC_ERR_CUDA, "no CUDA device");
    }
    s->own_stream = true;
  }
  const int sz[6] = {h1 * n_in, h1, h2 * h1, h2, n_out * h2, n_out};
  s->tc = prec == NNC_BF16 && n_in % 64 == 0 && h1 % 64 == 0 && h2 % 64 == 0;
  s->n_out_p = (n_out + 63) / 64 * 64;
  if (s->tc) {
    int r = walloc(s, &s->W2t, (size_t)h1 * h2);
    if (!r) r = walloc(s, &s->W3t, (size_t)h2 * s->n_out_p);
    if (!r) r = walloc(s, &s->d_err, 1);
    if (r) {
      nnc_ws_free(s);
      return r;
    }
  }
  for (int i = 0; i < 6; ++i) {
    s->sizes[i] = sz[i];
    if (!params[i]) {
      nnc_ws_free(s);
      return wfail(NNC_ERR_ARG, "NULL parameter array");
    }
    int r = walloc(s, &s->w[i], sz[i]);
    if (!r) r = walloc(s, &s->g[i], sz[i]);
    if (!r) r = walloc(s, &s->m[i], sz[i]);
    if (!r) r = walloc(s, &s->v[i], sz[i]);
    unsigned char* q = nullptr;
    if (!r) r = walloc(s, &q, (size_t)sz[i] * esz(s));
    if (r) {
      nnc_ws_free(s);
      return r;
    }
    s->wl[i] = q;
    std::vector<float> h(params[i], params[i] + sz[i]);
    cudaMemcpyAsync(s->w[i], h.data(), sizeof(float) * sz[i], cudaMemcpyHostToDevice, s->stream);
    if (prec == NNC_FP32) k_ws_cast<float><<<(sz[i] + 255) / 256, 256, 0, s->stream>>>(s->w[i], sz[i], (float*)q);
    else {
      __nv_bfloat16* wt = !s->tc ? nullptr : i == 2 ? s->W2t : i == 4 ? s->W3t : nullptr;
      k_ws_cast<__nv_bfloat16><<<(sz[i] + 255) / 256, 256, 0, s->stream>>>(
          s->w[i], sz[i], (__nv_bfloat16*)q, i == 2 ? h1 : i == 4 ? h2 : 1, wt,
          i == 2 ? h2 : i == 4 ? s->n_out_p : 0);
    }
    note_launch();
    cudaStreamSynchronize(s->stream);
  }
  s->in_mean.assign(n_in, 0.0);
  s->in_std.assign(n_in, 1.0);
  s->out_mean.assign(n_out, 0.0);
  s->out_std.assign(n_out, 1.0);
  if (cudaGetLastError() != cudaSuccess) {
    nnc_ws_free(s);
    return wfail(NNC_ERR_CUDA, "nnc_ws_create: CUDA error");
  }
  *out = s;
  return NNC_OK;
}

void nnc_ws_free(nnc_ws* s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  for (void* p : s->allocs) cudaFree(p);
  if (s->own_stream && s->stream) cudaStreamDestroy(s->stream);
  delete s;
}

int nnc_ws_set_scaling(nnc_ws* s, const double* in_mean, const double* in_std,
                       const double* out_mean, const double* out_std) {
  if (!s || !in_mean || !in_std || !out_mean || !out_std) return wfail(NNC_ERR_ARG, "bad scaling");
  s->in_mean.assign(in_mean, in_mean + s->n_in);
  s->in_std.assign(in_std, in_std + s->n_in);
  s->out_mean.assign(out_mean, out_mean + s->n_out);
  s->out_std.assign(out_std, out_std + s->n_out);
  return NNC_OK;
}

int nnc_ws_loss_grad(nnc_ws* s, const double* U, const double* Tt, int B, double* loss,
                     double* const* grads) {
  if (!s || !U || !Tt || B < 1) return wfail(NNC_ERR_ARG, "nnc_ws_loss_grad: bad arguments");
  int r = upload_std(s, U, Tt, B, true);
  if (r) return r;
  if (s->prec == NNC_FP32) {
    WCK(stage_rows<float>(s, B));
    r = loss_grad<float>(s, B, loss);
  } else {
    WCK(stage_rows<__nv_bfloat16>(s, B));
    r = loss_grad<__nv_bfloat16>(s, B, loss);
  }
  if (r) return r;
  r = check_ws_err(s);
  if (r) return r;
  if (grads) {
    for (int i = 0; i < 6; ++i) {
      if (!grads[i]) continue;
      std::vector<float> h(s->sizes[i]);
      WCK(cudaMemcpyAsync(h.data(), s->g[i], sizeof(float) * s->sizes[i], cudaMemcpyDeviceToHost, s->stream));
      WCK(cudaStreamSynchronize(s->stream));
      for (int j = 0; j < s->sizes[i]; ++j) grads[i][j] = h[j];
    }
  }
  return NNC_OK;
}

int nnc_ws_adam_step(nnc_ws* s, double lr, double beta1, double beta2, double eps) {
  if (!s) return wfail(NNC_ERR_ARG, "ws is NULL");
  WCK(s->prec == NNC_FP32 ? adam<float>(s, (float)lr, (float)beta1, (float)beta2, (float)eps)
                          : adam<__nv_bfloat16>(s, (float)lr, (float)beta1, (float)beta2, (float)eps));
  return NNC_OK;
}

int nnc_ws_train(nnc_ws* s, const double* U, const double* Tt, int N, int epochs, int batch,
                 double lr, double beta1, double beta2, double eps, unsigned long long seed,
                 double* final_loss) {
  if (!s || !U || !Tt || N < 1 || epochs < 0 || batch < 1) return wfail(NNC_ERR_ARG, "nnc_ws_train: bad arguments");
  const int B = std::min(batch, N), n_in = s->n_in, n_out = s->n_out, nc = n_in + n_out;
  int r = ensure_cap(s, B);
  if (!r) r = ensure_set(s, N);
  if (r) return r;
  cudaStream_t st = s->stream;
  // the data set goes to the device as given and is standardized there, per coordinate; batches are
  // gathered by index.  A set that does not fit beside its standardized copy is sent three times in parts:
  // for the means, the deviations and the standardized values.
  double *mean = s->stats, *sd = s->stats + nc;
  const int part = std::min(s->nr, N);
  for (int pass = part == N ? 2 : 0; pass <= 2; ++pass) {
    for (int r0 = 0; r0 < N; r0 += part) {
      const int n = std::min(part, N - r0);
      const size_t ou = (size_t)r0 * n_in, ot = (size_t)r0 * n_out;
      WCK(cudaMemcpyAsync(s->Ur, U + ou, sizeof(double) * (size_t)n * n_in, cudaMemcpyHostToDevice, st));
      WCK(cudaMemcpyAsync(s->Tr, Tt + ot, sizeof(double) * (size_t)n * n_out, cudaMemcpyHostToDevice, st));
      if (pass < 2 || part == N) {
        k_ws_stats<<<(n_in + 31) / 32, 32, 0, st>>>(s->Ur, pass, r0, n, N, n_in, mean, sd);
        k_ws_stats<<<(n_out + 31) / 32, 32, 0, st>>>(s->Tr, pass, r0, n, N, n_out, mean + n_in, sd + n_in);
        note_launch(2);
      }
      if (pass == 2) {
        k_ws_standardize<<<(unsigned)n * ((n_in + 255) / 256), 256, 0, st>>>(s->Ur, n_in, mean, sd, s->Ud + ou);
        k_ws_standardize<<<(unsigned)n * ((n_out + 255) / 256), 256, 0, st>>>(s->Tr, n_out, mean + n_in,
                                                                             sd + n_in, s->Td + ot);
        note_launch(2);
      }
      WCK(cudaGetLastError());
    }
  }
  std::vector<double> h(2 * (size_t)nc);
  WCK(cudaMemcpyAsync(h.data(), s->stats, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, st));
  WCK(cudaStreamSynchronize(st));
  std::copy_n(h.begin(), n_in, s->in_mean.begin());
  std::copy_n(h.begin() + n_in, n_out, s->out_mean.begin());
  std::copy_n(h.begin() + nc, n_in, s->in_std.begin());
  std::copy_n(h.begin() + nc + n_in, n_out, s->out_std.begin());
  std::mt19937_64 rng(seed);
  std::vector<int> perm(N);
  std::iota(perm.begin(), perm.end(), 0);
  double last = 0.0;
  const dim3 gg((unsigned)B * ((nc + 255) / 256));
  for (int e = 0; e < epochs; ++e) {
    std::shuffle(perm.begin(), perm.end(), rng);
    WCK(cudaMemcpyAsync(s->perm, perm.data(), sizeof(int) * N, cudaMemcpyHostToDevice, st));
    WCK(cudaStreamSynchronize(st));   // `perm` is shuffled again
    for (int b0 = 0; b0 + B <= N; b0 += B) {
      const bool want = (e == epochs - 1) && (b0 + 2 * B > N);
      if (s->prec == NNC_FP32) {
        WCK(launch_pdl(k_ws_gather<float>, gg, dim3(256), 0, st, s->Ud, s->Td, s->perm + b0, n_in, n_out,
                       (float*)s->Ul, nullptr, 0, s->Tt));
        r = loss_grad<float>(s, B, want ? &last : nullptr);
        if (r) return r;
        WCK(adam<float>(s, (float)lr, (float)beta1, (float)beta2, (float)eps));
      } else {
        WCK(launch_pdl(k_ws_gather<__nv_bfloat16>, gg, dim3(256), 0, st, s->Ud, s->Td, s->perm + b0, n_in,
                       n_out, (__nv_bfloat16*)s->Ul, s->tc ? s->Ut : nullptr, s->cap, s->Tt));
        r = loss_grad<__nv_bfloat16>(s, B, want ? &last : nullptr);
        if (r) return r;
        WCK(adam<__nv_bfloat16>(s, (float)lr, (float)beta1, (float)beta2, (float)eps));
      }
    }
  }
  WCK(cudaStreamSynchronize(s->stream));
  WCK(cudaGetLastError());
  r = check_ws_err(s);
  if (r) return r;
  if (final_loss) *final_loss = last;
  return NNC_OK;
}

int nnc_ws_predict(nnc_ws* s, const double* U, int N, double* P) {
  if (!s || !U || !P || N < 1) return wfail(NNC_ERR_ARG, "nnc_ws_predict: bad arguments");
  int r = upload_std(s, U, nullptr, N, false);
  if (r) return r;
  if (s->prec == NNC_FP32) {
    WCK(stage_rows<float>(s, N));
    r = forward<float>(s, N);
  } else {
    WCK(stage_rows<__nv_bfloat16>(s, N));
    r = forward<__nv_bfloat16>(s, N);
  }
  if (r) return r;
  r = check_ws_err(s);
  if (r) return r;
  std::vector<float> h((size_t)N * s->n_out);
  WCK(cudaMemcpyAsync(h.data(), s->P, sizeof(float) * h.size(), cudaMemcpyDeviceToHost, s->stream));
  WCK(cudaStreamSynchronize(s->stream));
  for (int i = 0; i < N; ++i)
    for (int c = 0; c < s->n_out; ++c)
      P[(size_t)i * s->n_out + c] = h[(size_t)i * s->n_out + c] * s->out_std[c] + s->out_mean[c];
  return NNC_OK;
}

int nnc_ws_get_params(nnc_ws* s, double* const* params) {
  if (!s || !params) return wfail(NNC_ERR_ARG, "bad arguments");
  for (int i = 0; i < 6; ++i) {
    if (!params[i]) continue;
    std::vector<float> h(s->sizes[i]);
    WCK(cudaMemcpyAsync(h.data(), s->w[i], sizeof(float) * s->sizes[i], cudaMemcpyDeviceToHost, s->stream));
    WCK(cudaStreamSynchronize(s->stream));
    for (int j = 0; j < s->sizes[i]; ++j) params[i][j] = h[j];
  }
  return NNC_OK;
}

}  // extern "C"
