// CUDA-core GEMMs of the FP64 and FP32 forms: the forward tangent sweep of the Hessian
// (Zdot_l = W_l Adot_{l-1}, n_in tangent columns) and the symmetric product
// H = sum_l Zdot_l^T diag(c_l) Zdot_l, every sum in order of k.  k_sgemm is the FP32 form's; k_simt_gemm
// the FP64 form's, which comes here only where the residue products of k_rns.cu do not serve: their residues
// take four times the memory of the FP64 weights, and keep too few bits of uneven weights.
#include <algorithm>

#include "async.cuh"
#include "kernels.cuh"

namespace nnc {

enum { EPI_TANGENT = 0, EPI_SYRK = 1 };

// FP64: D[m][n] = sum_k A[m][k] B[n][k] on a 64 x 64 tile with 256 threads; thread (tx, ty)
// owns rows m0 + tx + 16 i and columns n0 + ty + 16 j.  K must be a multiple of 16 (all
// packed dimensions are multiples of 128).
template <int EPI>
__global__ void __launch_bounds__(256) k_simt_gemm(const double* __restrict__ A, int lda,
                                                   const double* __restrict__ B, int ldb, int M, int N,
                                                   int K, int k_per_split,
                                                   const double* __restrict__ s1,
                                                   const double* __restrict__ c,
                                                   double* __restrict__ At, double* __restrict__ Zt,
                                                   double* __restrict__ Yt, int ldo, int ldz,
                                                   double* __restrict__ Hp) {
  constexpr int TM = 4, TN = 4, BM = 16 * TM, BN = 16 * TN, BK = 16;
  __shared__ double As[BK][BM + 1];
  __shared__ double Bs[BK][BN + 1];
  const int bm = blockIdx.y, bn = blockIdx.x, split = blockIdx.z;
  if (EPI == EPI_SYRK && bn > bm) return;  // upper-triangle tiles are mirrored at the end
  const int m0 = bm * BM, n0 = bn * BN;
  const int kbeg = split * k_per_split;
  const int kend = min(K, kbeg + k_per_split);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;

  for (int k0 = kbeg; k0 < kend; k0 += BK) {
    for (int i = threadIdx.x; i < BM * BK; i += 256) {
      const int r = i >> 4, kk = i & 15;
      const int gm = m0 + r;
      As[kk][r] = gm < M ? A[(size_t)gm * lda + k0 + kk] : 0.0;
    }
    for (int i = threadIdx.x; i < BN * BK; i += 256) {
      const int r = i >> 4, kk = i & 15;
      const int gn = n0 + r;
      Bs[kk][r] = gn < N ? B[(size_t)gn * ldb + k0 + kk] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      double a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][tx + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][ty + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

  if (EPI == EPI_TANGENT) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int m = m0 + tx + 16 * i;
      if (m >= M) continue;
      const double sm = s1[m], cm = c[m];
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int n = n0 + ty + 16 * j;
        if (n >= N) continue;
        const double v = acc[i][j];
        if (At) At[(size_t)n * ldo + m] = sm * v;
        if (Zt) {
          const size_t oz = (size_t)n * ldz + m;
          Zt[oz] = v;
          Yt[oz] = cm * v;
        }
      }
    }
  } else {
    double* hp = Hp + (size_t)split * M * N;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int m = m0 + tx + 16 * i;
      if (m >= M) continue;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int n = n0 + ty + 16 * j;
        if (n >= N) continue;
        hp[(size_t)m * N + n] += acc[i][j];
      }
    }
  }
}

// FP32: D[m][n] = sum_k A[m][k] B[n][k], k in order.  A warp owns 32 rows m of 4 C columns n, eight lanes
// along the rows (rows lane & 7, + 8, ...), four along the columns (lane >> 3, + 4, ...): 4 x C outputs a
// lane; a CTA of 4 x 2 warps 128 x 8 C.  Both operands go to shared memory as they lie, by 16-byte
// asynchronous copies, in a ring of four stages of 16 columns of K; rows of 20 floats there put the eight
// lanes of a quarter warp on different banks.
// Bound: what shared memory returns to registers, 128 bytes per clock and SM (a load that all lanes share
// returns as much as any other): 4 + C clocks per k and warp, against C clocks of FMAs.  Larger tiles a
// lane need fewer loads but leave a scheduler one warp.  1024 x 784 x 1024: 62 us; 69 us with 2 x 12
// outputs a lane, about 90 us with 8 x 8; 252 us with 8 x 8, single-buffered, one float at a time.
// SYRK: A = Ydot^T, B = Zdot^T, split blockIdx.z of K, tiles that reach the lower triangle n >= m.
constexpr int kSgM = 128, kSgK = 16, kSgThreads = 256, kSgStages = 4;
constexpr int kSgLd = kSgK + 4;   // floats per row in shared memory

struct SgArgs {
  const float *A, *B;
  int lda, ldb, M, N, K, k_per_split;
  const double *s1, *c;
  float *At, *Zt, *Yt;
  int ldo, ldz;
  double* Hp;   // [splits][N][M] (SYRK: N = M)
};

// 16 bytes from global `src` (zeros if !valid) to shared `dst`.
__device__ __forceinline__ void cp16(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(async::smem_u32(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}

template <int C, int EPI>
__global__ void __launch_bounds__(kSgThreads) k_sgemm(const SgArgs p) {
  constexpr int BN = 8 * C, ROWS = kSgM + BN, STAGE = ROWS * kSgLd;
  constexpr int Q = (ROWS * 4 + kSgThreads - 1) / kSgThreads;   // 16-byte copies per thread and stage
  extern __shared__ __align__(16) float sg_smem[];   // [kSgStages][kSgM + BN][kSgLd]
  const int m0 = blockIdx.x * kSgM, n0 = blockIdx.y * BN, split = blockIdx.z;
  if (EPI == EPI_SYRK && m0 > n0 + BN - 1) return;   // above the diagonal: mirrored at the end
  const int kbeg = split * p.k_per_split, kend = min(p.K, kbeg + p.k_per_split);
  const int tid = threadIdx.x, lane = tid & 31;
  const int lm = (tid >> 6) * 32 + (lane & 7), ln = (tid >> 5 & 1) * 4 * C + (lane >> 3);   // first row, column
  auto load = [&](int k0, int stage) {
    if (k0 < kend) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int e = tid + q * kSgThreads, r = e >> 2, k = k0 + 4 * (e & 3);
        if (ROWS * 4 % kSgThreads && e >= ROWS * 4) break;
        const bool isa = r < kSgM;
        const int g = isa ? m0 + r : n0 + r - kSgM;
        const bool valid = g < (isa ? p.M : p.N);
        const float* src = isa ? p.A + (size_t)(valid ? g : 0) * p.lda + k : p.B + (size_t)(valid ? g : 0) * p.ldb + k;
        cp16(sg_smem + stage * STAGE + r * kSgLd + 4 * (e & 3), src, valid);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[4][C];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < C; ++j) acc[i][j] = 0.f;
  for (int s = 0; s < kSgStages - 1; ++s) load(kbeg + s * kSgK, s);
  int stage = 0;
  for (int k0 = kbeg; k0 < kend; k0 += kSgK) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kSgStages - 2) : "memory");
    __syncthreads();   // this stage is there, and nobody reads the one before it any more
    load(k0 + (kSgStages - 1) * kSgK, stage == 0 ? kSgStages - 1 : stage - 1);
    const float* as = sg_smem + stage * STAGE + lm * kSgLd;
    const float* bs = sg_smem + stage * STAGE + (kSgM + ln) * kSgLd;
#pragma unroll
    for (int kk = 0; kk < kSgK; kk += 4) {
      float4 a[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(as + 8 * i * kSgLd + kk);
#pragma unroll
      for (int j = 0; j < C; ++j) {
        const float4 b = *reinterpret_cast<const float4*>(bs + 4 * j * kSgLd + kk);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = fmaf(a[i].x, b.x, acc[i][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = fmaf(a[i].y, b.y, acc[i][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = fmaf(a[i].z, b.z, acc[i][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][j] = fmaf(a[i].w, b.w, acc[i][j]);
      }
    }
    stage = stage + 1 == kSgStages ? 0 : stage + 1;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + lm + 8 * i;
    if (m >= p.M) break;
    const double sm = EPI == EPI_TANGENT ? p.s1[m] : 0.0, cm = EPI == EPI_TANGENT ? p.c[m] : 0.0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
      const int n = n0 + ln + 4 * j;
      if (n >= p.N) break;
      const double v = (double)acc[i][j];
      if (EPI == EPI_TANGENT) {
        if (p.At) p.At[(size_t)n * p.ldo + m] = (float)(sm * v);
        if (p.Zt) {
          p.Zt[(size_t)n * p.ldz + m] = acc[i][j];
          p.Yt[(size_t)n * p.ldz + m] = (float)(cm * v);
        }
      } else {
        p.Hp[((size_t)split * p.N + n) * p.M + m] = v;
      }
    }
  }
}

template <int C, int EPI>
cudaError_t launch_sgemm_c(const SgArgs& a, int splits, cudaStream_t st) {
  constexpr int smem = kSgStages * (kSgM + 8 * C) * kSgLd * (int)sizeof(float);
  static bool attr = false;
  if (!attr) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_sgemm<C, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const dim3 grid((a.M + kSgM - 1) / kSgM, (a.N + 8 * C - 1) / (8 * C), splits);
  k_sgemm<C, EPI><<<grid, kSgThreads, smem, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

template <int EPI>
cudaError_t launch_sgemm(const SgArgs& a, int splits, int sm_count, cudaStream_t st) {
  // columns per lane: the least time of the busiest SM, tiles times 4 + C (the bound above)
  int best = 8;
  long long least = -1;
  for (int c : {8, 6, 4, 2}) {
    const long long t = (long long)((a.M + kSgM - 1) / kSgM) * ((a.N + 8 * c - 1) / (8 * c)) * splits;
    const long long cost = (t + sm_count - 1) / sm_count * (4 + c);
    if (least < 0 || cost < least) {
      least = cost;
      best = c;
    }
  }
  switch (best) {
    case 8: return launch_sgemm_c<8, EPI>(a, splits, st);
    case 6: return launch_sgemm_c<6, EPI>(a, splits, st);
    case 4: return launch_sgemm_c<4, EPI>(a, splits, st);
    default: return launch_sgemm_c<2, EPI>(a, splits, st);
  }
}

cudaError_t launch_simt_tangent(bool fp64, const void* A, int lda, const void* B, int ldb, int M,
                                int N, int K, const double* s1, const double* c, void* At, int ldo,
                                void* Zt, void* Yt, int ldz, int sm_count, cudaStream_t st) {
  if (fp64) {
    dim3 grid((N + 63) / 64, (M + 63) / 64, 1);
    k_simt_gemm<EPI_TANGENT><<<grid, 256, 0, st>>>(
        (const double*)A, lda, (const double*)B, ldb, M, N, K, K, s1, c, (double*)At, (double*)Zt,
        (double*)Yt, ldo, ldz, nullptr);
  } else {
    return launch_sgemm<EPI_TANGENT>(SgArgs{(const float*)A, (const float*)B, lda, ldb, M, N, K, K, s1, c,
                                            (float*)At, (float*)Zt, (float*)Yt, ldo, ldz, nullptr},
                                     1, sm_count, st);
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_simt_syrk(bool fp64, const void* Zt, const void* Yt, int ld, int n, int K,
                             int splits, double* Hp, int sm_count, cudaStream_t st) {
  const int kps = ((K + splits - 1) / splits + 15) / 16 * 16;
  if (fp64) {
    dim3 grid((n + 63) / 64, (n + 63) / 64, splits);
    k_simt_gemm<EPI_SYRK><<<grid, 256, 0, st>>>(
        (const double*)Zt, ld, (const double*)Yt, ld, n, n, K, kps, nullptr, nullptr, nullptr,
        nullptr, nullptr, 0, 0, Hp);
  } else {
    return launch_sgemm<EPI_SYRK>(SgArgs{(const float*)Yt, (const float*)Zt, ld, ld, n, n, K, kps, nullptr,
                                         nullptr, nullptr, nullptr, nullptr, 0, 0, Hp},
                                  splits, sm_count, st);
  }
  note_launch();
  return cudaGetLastError();
}

}  // namespace nnc
