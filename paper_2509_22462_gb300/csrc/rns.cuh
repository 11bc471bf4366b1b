// FP64 matrix products on the BF16 tensor cores by a residue number system (k_rns.cu), host side.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace nnc {

constexpr int kRns = 16;   // residues per number

// Moduli and the constants of one product's number system, passed to the kernels by value.
struct RnsSet {
  int bits = 0;                 // operands are integers of magnitude <= 2^bits
  float p[kRns], pinv[kRns];
  float r16[kRns], r32[kRns], r48[kRns];   // 2^16, 2^32, 2^48 mod p, in [-p/2, p/2]
  float q[kRns];                // (P / p)^-1 mod p, in [-p/2, p/2]
  unsigned c0[kRns], c1[kRns], c2[kRns];   // round(2^96 / p), low word first
  double scale = 0.0;           // P 2^-64
};
// The system of a product over K terms (K <= 65664).
RnsSet rns_set(int K);

struct RnsPlan {
  CUtensorMap ta, tb;
  int M = 0, N = 0, nkb = 0, bn = 0, lower = 0, rev = 0, a_rows = 0, b_rows = 0;
  bool ready = false;
};
// D = A B^T for every residue: A [kRns][a_rows][K] and B [kRns][b_rows][K] (BF16 integers, K-major,
// row stride K, a multiple of 64); M <= a_rows rounded up to 128, N <= b_rows.  lower: only the
// tiles on and below the diagonal.
int rns_plan(RnsPlan& p, const void* A, int a_rows, const void* B, int b_rows, int M, int N, int K,
             bool lower);
// C[i][n][m] = (sum_k A_i[m][k] B_i[n][k]) mod p_i, one byte each, rows of ldc (>= M rounded up to
// 128) bytes, N rows per residue.
cudaError_t rns_gemm(const RnsPlan& p, const RnsSet& s, unsigned char* C, int ldc, int* err,
                     int sm_count, cudaStream_t st);

// Powers of two 2^de[k] that even out the columns of W [m][k] (row stride ldw): the residues are those of
// W[r][k] 2^-de[k], the operand beside them is multiplied by 2^de[k].  Scratch: rns_even_scratch(k)
// bytes.  *flags receives kRnsUneven where the rounding of a row would cost too much all the same (the
// net's products then stay on the CUDA cores), kRnsScaled where de is needed (else
// it is left out).
constexpr int kRnsUneven = 1, kRnsScaled = 2;
size_t rns_even_scratch(int k);
cudaError_t rns_even_out(const RnsSet& s, const double* W, int ldw, int m, int k, void* scratch, int* de,
                         int* flags, cudaStream_t st);

// Weights W [mp][kp] (FP64): residues [kRns][mp][kp] of W 2^-de (de [kp] or NULL) with q folded in, and
// the row scales sa[mp].
cudaError_t rns_pack_weights(const RnsSet& s, const double* W, int mp, int kp, const int* de, void* res,
                             double* sa, cudaStream_t st);

// One layer's tangents, row by row (n rows of K = mp columns).
struct RnsRows {
  // source: residues C [kRns][n][ldc] of Zdot with the scales sa[m], sb[row], or FP64 Z
  const unsigned char* C = nullptr;
  int ldc = 0;
  const double *sa = nullptr, *sb = nullptr;
  double* Z = nullptr;          // [n][ldz]: read if C is NULL, else written
  int ldz = 0;
  int n = 0, K = 0;             // K: columns handled (a multiple of 128)
  const double* s1 = nullptr;   // sigma' of the layer
  const double *c = nullptr, *rc = nullptr;   // curvature weight and sqrt|c|
  const int* de = nullptr;      // the next layer's column exponents [K], or NULL
  void* At = nullptr;           // residues of s1 * Z * 2^de [kRns][n][K], or NULL
  double* sat = nullptr;        // their row scales [n]
  void *Sa = nullptr, *Sb = nullptr;   // residues of rc Z (q folded in) and sign(c) rc Z, or NULL
  double* ss = nullptr;         // their row scales [n]
};
cudaError_t rns_rows(const RnsSet& s, const RnsRows& a, cudaStream_t st);

// One step between two reverse products: seeds s < S, K columns (the output layer's rows, or the
// columns of the layer just multiplied, padded).
struct RnsRev {
  const unsigned char* C = nullptr;   // planes of rns_gemm on an rns_plan_rev plan, or NULL: seeds
  int chunks = 0, seeds = 0;          // seeds: rows of a plane (S rounded up to 16)
  const double* sb = nullptr;         // scales of the seeds that were multiplied [S]
  const int* de = nullptr;            // column exponents of the weights that were multiplied [K], or NULL
  int K = 0, kvalid = 0, nJ = 0, lam_col = -1;
  const double *s1 = nullptr, *s2 = nullptr;   // of the layer that owns the K columns; NULL: x
  const double *lam = nullptr, *soft_p = nullptr;   // seeds (out_seed)
  const double* sa = nullptr;         // that layer's row scales of W
  double *c_out = nullptr, *rc_out = nullptr;   // its curvature weights c (lambda column), and sqrt|c| or NULL
  double *J = nullptr, *g = nullptr;  // x: J [nJ][kvalid], gradient (each may be NULL)
  double* Zs = nullptr;               // scratch [S][K]
  void* Zr = nullptr;                 // residues [n][seeds][K] of the scaled seeds
  double* sb_out = nullptr;           // their scales [S]
};
cudaError_t rns_rev_rows(const RnsSet& s, const RnsRev& a, int S, cudaStream_t st);
// Product W^T Z over the mp rows of the residues W [kRns][mp][kp], Z [kRns][seeds rounded up to 16][mp].
// rns_gemm then writes C[chunk][i][seed][k] (rows of kp bytes), chunks = rows / 1024 rounded up.
int rns_plan_rev(RnsPlan& p, const void* W, int mp, int kp, const void* Z, int seeds);

// The rank-two part of a softmax layer's curvature as two more columns m, m + 1 of its block:
// Z[j][m + k] = w_k[j], c[m + k] = g'_k, rc likewise (see k_softmax_ext).
cudaError_t rns_softmax_ext(int n, int m, int col, const double* p, const double* lam, double* Z,
                            int ldz, double* c, double* rc, cudaStream_t st);

// H[i][j] = H[j][i] = sum_l ss_l[i] ss_l[j] D_l[i][j] over `layers` residue planes
// U [layers][kRns][n][ldu] (entry [j][i], i >= j), ss [layers][n].
cudaError_t rns_h_finish(const RnsSet& s, int layers, const unsigned char* U, int ldu,
                         const double* ss, int n, double* H, cudaStream_t st);

}  // namespace nnc
