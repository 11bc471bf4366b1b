// FP64 matrix products of the FP64 form on the BF16 tensor cores.
//
// GB300 issues about two FP64 FMAs per clock and SM, so the two contractions of the Hessian
// (tangents Zdot_l = W_l Adot_{l-1}, and H = sum_l Zdot_l^T diag(c_l) Zdot_l) took 181 ms of a
// 104M-parameter evaluation in an FP64 GEMM on the CUDA cores.  The residue scheme of Ozaki, Uchino
// and Imamura ("Ozaki scheme II", 2025) does them with integer products instead:
//   - every row of either operand is scaled by a power of two and rounded to integers of at most
//     `bits` + 1 bits below its largest entry (bits = 57 at K = 1024, 56 at 4096, 54 at 65664);
//   - so an entry 2^j below its row's largest has j bits fewer.  Powers of two even out the columns of the
//     weights beforehand (k_rns_colsum), which makes the rounding independent of the units in which
//     inputs, hidden units and outputs are measured; weights that stay uneven (k_rns_spread) keep the
//     FP64 products;
//   - an integer is kept as its residues modulo 16 pairwise coprime numbers p_i <= 256, each
//     in [-p/2, p/2], which BF16 holds exactly;
//   - one BF16 product per modulus gives the result's residue: products are at most 2^14, so 1024
//     terms add up exactly in the tensor core's FP32 accumulator, which is reduced mod p_i after
//     every 1024 terms of K;
//   - the Chinese remainder theorem gives the integer result: D / P = frac(sum_i y_i / p_i) with
//     y_i = D_i (P/p_i)^-1 mod p_i (the inverse is folded into one operand) and P = prod p_i,
//     summed in 96-bit fixed point, where integer overflow is the frac().
// The adjoints of the reverse sweep, W_l^T Zbar, take the same residues of W (REV below): n_out + 1
// FP64 FMAs per weight would be 2.5 ms of the same evaluation.
// The only roundings are those of the operands and of the result, so the error does not grow with
// K as a sum of FP64 products does.  Chosen over slicing into 8-bit digits, which needs 28 products
// where this needs 16.  Rows holding a NaN or an infinity give NaN.
//
// Every kernel waits for the one before it itself (programmatic dependent launch): a small net's evaluation
// is twenty short launches.
//
// Measured, residual + J + H + gradient at one iterate: 784 -> 4096 x 7 -> 10 181 ms with FP64 products, 4.00 ms
// so (error of H against 64-bit sums 5.7e-15, 3.5e-15), 784 -> 128 x 2 -> 10 912 and 113 us (8e-16, 7e-16).
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "async.cuh"
#include "rns.cuh"
#include "umma.cuh"

namespace nnc {
using namespace umma;

namespace {

constexpr int kModuli[kRns] = {256, 255, 253, 251, 247, 241, 239, 233,
                                  229, 227, 223, 217, 211, 199, 197, 193};

// ------------------------------------------------------------------ residue arithmetic
// x - p rint(x / p) for |x| <= 2^24 (all steps exact but the quotient's rounding, which can only
// move a value next to +-p/2 to the other end).
__device__ __forceinline__ float rns_mod(float x, float p, float pinv) {
  const float q = __fsub_rn(__fmaf_rn(x, pinv, 12582912.f), 12582912.f);
  return __fmaf_rn(-q, p, x);
}

// The four 16-bit limbs of a (signed, |a| <= 2^60) as floats in [-2^15, 2^15).
struct Limbs {
  float l0, l1, l2, l3;
};
__device__ __forceinline__ Limbs rns_limbs(long long a) {
  const unsigned long long u = (unsigned long long)a + 0x8000800080008000ull;
  const unsigned lo = (unsigned)u, hi = (unsigned)(u >> 32);
  const float off = 8388608.f + 32768.f;
  return Limbs{__uint_as_float(0x4B000000u | (lo & 0xFFFFu)) - off,
               __uint_as_float(0x4B000000u | (lo >> 16)) - off,
               __uint_as_float(0x4B000000u | (hi & 0xFFFFu)) - off,
               __uint_as_float(0x4B000000u | (hi >> 16)) - off};
}
__device__ __forceinline__ float rns_res(const RnsSet& s, int i, const Limbs& l) {
  const float x = __fmaf_rn(l.l3, s.r48[i], __fmaf_rn(l.l2, s.r32[i], __fmaf_rn(l.l1, s.r16[i], l.l0)));
  return rns_mod(x, s.p[i], s.pinv[i]);
}
// BF16 bits of an integer of at most 8 significant bits: the upper half of its FP32 bits.
__device__ __forceinline__ unsigned bf2(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// Scale of a row whose values are below 2^(ex - 1022) in size (ex: biased exponent, 0x7FF for a row
// with a NaN or an infinity).  *sh = bits - e makes the integers v 2^sh, the return value 2^-sh undoes it
// (NaN for a row with a NaN or an infinity).
__device__ __forceinline__ double rns_scale(int ex, int bits, int* sh) {
  const int e = max(ex - 1022, -900);
  *sh = bits - e;
  return ex == 0x7FF ? __longlong_as_double(0x7FF8000000000000ll)
                     : __hiloint2double((e - bits + 1023) << 20, 0);
}
__device__ __forceinline__ int expo(double v) { return (__double2hiint(v) >> 20) & 0x7FF; }

// GB300 issues one FP64 instruction of a warp every 16 clocks of an SM; the helpers below do in a dozen
// integer instructions (a clock or less each) what would be two or three FP64 ones per element.

// Biased exponent that bounds |a b| < 2^(e - 1022) (0x7FF: a NaN, an infinity or an overflow): from the
// top 21 bits of both mantissas, rounded up.
__device__ __forceinline__ int prod_expo(double a, double b) {
  const int ha = __double2hiint(a), hb = __double2hiint(b);
  const int ea = (ha >> 20) & 0x7FF, eb = (hb >> 20) & 0x7FF;
  const unsigned p = __umulhi(((unsigned)ha << 11) | 0x800007FFu, ((unsigned)hb << 11) | 0x800007FFu);
  const int e = ea + eb - 1023 + (p >= 0x7FFFFFFCu ? 1 : 0);
  return max(ea, eb) == 0x7FF ? 0x7FF : min(max(e, 0), 0x7FF);
}
// v 2^sh as an integer, to nearest; |v 2^sh| <= 2^60.
__device__ __forceinline__ long long to_int(double v, int sh) {
  const long long u = __double_as_longlong(v);
  const int e = (int)(u >> 52) & 0x7FF;
  const unsigned long long m = ((unsigned long long)u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int s = e - 1075 + sh;   // |v| 2^sh = m 2^s
  const int t = min(max(-s, 0), 63);
  const unsigned long long half = t > 0 ? 1ull << (t - 1) : 0ull;
  unsigned long long r = s >= 0 ? m << min(s, 8) : (m + half) >> t;
  if (e == 0) r = 0;
  return u < 0 ? -(long long)r : (long long)r;
}

// 96-bit fixed-point value of D / P from the residues y_i (0 .. p_i - 1), as D 2^64 / P.
struct Crt {
  unsigned long long lo = 0, mid = 0;
  unsigned hi = 0;
  __device__ __forceinline__ void add(const RnsSet& s, int i, unsigned y) {
    lo += (unsigned long long)y * s.c0[i];
    mid += (unsigned long long)y * s.c1[i];
    hi += y * s.c2[i];
  }
  // rounded to nearest by hand: sign and size, 64 leading bits, 53 of them
  __device__ __forceinline__ double value() const {
    const unsigned long long m = mid + (lo >> 32);
    const unsigned h = hi + (unsigned)(m >> 32);
    unsigned long long t = ((unsigned long long)h << 32) | (unsigned)m;
    unsigned l = (unsigned)lo;
    const bool neg = (int)h < 0;
    if (neg) {   // ones' complement: off by 2^-32 of a unit of t
      t = ~t;
      l = ~l;
    }
    if (t == 0) {   // below 2^-64 P
      const double v = (double)l * 2.3283064365386963e-10;
      return neg ? -v : v;
    }
    const int z = __clzll((long long)t);
    t = z ? (t << z) | (((unsigned long long)l << 32) >> (64 - z)) : t;
    t = (t >> 11) + ((t >> 10) & 1ull);   // 2^52 .. 2^53, times 2^(11 - z)
    t += ((unsigned long long)(1085 - z)) << 52;
    return __longlong_as_double((long long)(t | (neg ? 0x8000000000000000ull : 0ull)));
  }
};

// The biased exponent of v 2^d from that of v.
__device__ __forceinline__ int shift_expo(int e, int d) {
  return e == 0x7FF ? e : min(max(e + d, 0), 0x7FF);
}

__device__ __forceinline__ int block_max(int v, int* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = __reduce_max_sync(0xffffffffu, v);
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  int r = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = max(r, sh[w]);
  __syncthreads();
  return r;
}
__device__ __forceinline__ int block_sum(int v, int* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = __reduce_add_sync(0xffffffffu, v);
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  int r = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sh[w];
  __syncthreads();
  return r;
}

// ------------------------------------------------------------------ weights (once, at load)
// Column exponents.  A row of W is rounded relative to its largest entry, so a column that is small in
// every row (an input in small units, the outgoing weights of a hidden unit in large ones) would lose
// what it is smaller by: inputs spread over 2^40 left 1e-6 of a column of J, where FP64 products leave
// 2e-15.  2^de[k] is the geometric mean of column k's entries in units of the first column's, which sees
// through rows of any size.  The mean is taken of 16 bits of mantissa behind the exponent, in integers, so
// that the order of the sums does not matter.  A matrix whose means all lie within 2^2.5 of the first one
// (2^4.5 for less than 64 rows, whose means scatter more), as those of evenly scaled weights do, stays as it
// is: 784 -> 128 x 2 -> 10 takes 129 us with its exponents of -1, 0 and 1, 126 without, and
// 784 -> 4096 x 7 -> 10 3.87 ms with those of its last layer, 3.84 without.
struct RnsEven {
  unsigned long long* sum;   // [k] of the nonzero entries' logarithms, times 2^16
  int *cnt, *small;          // [k] nonzero entries; entries in nonzero rows that are small there
  unsigned long long* total; // [3] entries looked at, small ones, nonzero rows
};
constexpr int kEvenRows = 256;   // rows of W per CTA

__global__ void __launch_bounds__(256) k_rns_colsum(const double* __restrict__ W, int ldw, int m, int k,
                                                    const RnsEven e, int* __restrict__ flags) {
  __shared__ unsigned long long s[8][32];
  __shared__ int c[8][32];
  const int col = blockIdx.x * 32 + threadIdx.x, y = threadIdx.y;
  const int r1 = min(m, (int)(blockIdx.y + 1) * kEvenRows);
  unsigned long long sum = 0;
  int cnt = 0;
  bool odd = false;
  if (col < k) {
    for (int r = blockIdx.y * kEvenRows + y; r < r1; r += 8) {
      const double w = W[(size_t)r * ldw + col];
      const int ex = expo(w);
      // the exponents of products and scales stay in range for weights of 2^-200 to 2^200
      odd |= w != 0.0 && (ex < 1023 - 200 || ex > 1023 + 200);
      if (ex > 0) {
        sum += (unsigned)(__double2hiint(w) & 0x7FFFFFFF) >> 4;
        ++cnt;
      }
    }
  }
  if (odd) atomicOr(flags, kRnsUneven);
  s[y][threadIdx.x] = sum;
  c[y][threadIdx.x] = cnt;
  __syncthreads();
  if (y > 0 || col >= k) return;
  for (int j = 1; j < 8; ++j) {
    sum += s[j][threadIdx.x];
    cnt += c[j][threadIdx.x];
  }
  atomicAdd(e.sum + col, sum);
  atomicAdd(e.cnt + col, cnt);
}

__global__ void __launch_bounds__(256) k_rns_colexp(int m, int k, const RnsEven e,
                                                    int* __restrict__ de, int* __restrict__ flags) {
  const int col = blockIdx.x * 256 + threadIdx.x;
  if (col >= k) return;
  int q = 0;   // the first column that is not zero
  while (q < k - 1 && e.cnt[q] == 0) ++q;
  int d = 0;
  if (e.cnt[col] > 0) {   // sum / cnt against sum_q / cnt_q, to nearest: |difference| < 2^59
    const long long c = e.cnt[col], cq = e.cnt[q], den = c * cq << 16;
    const long long num = 2 * ((long long)e.sum[col] * cq - (long long)e.sum[q] * c) + den;
    d = (int)(num >= 0 ? num / (2 * den) : -((2 * den - 1 - num) / (2 * den)));
  }
  de[col] = d;
  if (abs(d) > (m >= 64 ? 2 : 4)) atomicOr(flags, kRnsScaled);
}

// How uneven W 2^-de is: an entry is small if it lies more than 2^(bits - 44) below its row's largest, so
// that fewer than 44 of its bits are kept.  Sums in which such entries are outnumbered lose nothing to
// speak of (a few percent of normally distributed entries are small); a row or column that consists of
// them would.  So of 64 entries or more in a row or a column at most a quarter may be small, of 16 or
// more half, and of the whole matrix a quarter.  Rows and columns of zeros do not count.  No row's largest
// entry may lie more than 2^(bits - 44) above the geometric mean of its nonzero ones either, however short the
// row: its scale is multiplied into the seeds, and would push those of the other rows down.
__device__ __forceinline__ bool rns_uneven(int small, int n) {
  return n >= 64 ? 4 * (long long)small > n : n >= 16 && 2 * small > n;
}
__global__ void __launch_bounds__(256) k_rns_spread(const double* __restrict__ W, int ldw, int k, int bits,
                                                    const int* __restrict__ de, const RnsEven e,
                                                    int* __restrict__ flags) {
  __shared__ int sh[8];
  const double* w = W + (size_t)blockIdx.x * ldw;
  int ex = 0;
  for (int j = threadIdx.x; j < k; j += 256)
    if (expo(w[j]) > 0) ex = max(ex, expo(w[j]) - de[j]);
  ex = block_max(ex, sh);
  if (ex <= 0) return;   // a row of zeros
  int small = 0, n = 0, nz = 0, below = 0;   // below: sum of log2(largest / entry) over the nonzero ones
  for (int j = threadIdx.x; j < k; j += 256) {
    if (e.cnt[j] == 0) continue;
    ++n;
    if (expo(w[j]) > 0) {
      ++nz;
      below += ex - (expo(w[j]) - de[j]);
    }
    if (expo(w[j]) == 0 || expo(w[j]) - de[j] < ex - (bits - 44)) {
      ++small;
      atomicAdd(e.small + j, 1);
    }
  }
  n = block_sum(n, sh);
  small = block_sum(small, sh);
  nz = block_sum(nz, sh);
  below = block_sum(below, sh);   // at most 65536 times 1200
  if (threadIdx.x == 0) {
    if (rns_uneven(small, n) || below > (bits - 44) * nz) atomicOr(flags, kRnsUneven);
    atomicAdd(e.total, (unsigned long long)n);
    atomicAdd(e.total + 1, (unsigned long long)small);
    atomicAdd(e.total + 2, 1ull);
  }
}
__global__ void __launch_bounds__(256) k_rns_colspread(int k, const RnsEven e, int* __restrict__ flags) {
  const int col = blockIdx.x * 256 + threadIdx.x;
  if (col < k && rns_uneven(e.small[col], (int)e.total[2])) atomicOr(flags, kRnsUneven);
  if (col == 0 && 4 * e.total[1] > e.total[0]) atomicOr(flags, kRnsUneven);
}

__global__ void __launch_bounds__(256) k_rns_pack(const __grid_constant__ RnsSet s,
                                                  const double* __restrict__ W, int mp, int kp,
                                                  const int* __restrict__ de,
                                                  __nv_bfloat16* __restrict__ res,
                                                  double* __restrict__ sa) {
  __shared__ int sh[8];
  const int r = blockIdx.x;
  const double* w = W + (size_t)r * kp;
  int ex = 0, sc;
  for (int k = threadIdx.x; k < kp; k += blockDim.x)
    if (expo(w[k]) > 0) ex = max(ex, expo(w[k]) - (de ? de[k] : 0));
  const double back = rns_scale(block_max(ex, sh), s.bits, &sc);
  if (threadIdx.x == 0) sa[r] = back;
  for (int k = 4 * threadIdx.x; k < kp; k += 4 * blockDim.x) {
    Limbs l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) l[j] = rns_limbs(to_int(w[k + j], sc - (de ? de[k + j] : 0)));
#pragma unroll 4
    for (int i = 0; i < kRns; ++i) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = rns_mod(rns_res(s, i, l[j]) * s.q[i], s.p[i], s.pinv[i]);
      *reinterpret_cast<uint2*>(res + ((size_t)i * mp + r) * kp + k) =
          make_uint2(bf2(v[0], v[1]), bf2(v[2], v[3]));
    }
  }
}

// ------------------------------------------------------------------ tangent rows
// One CTA per tangent (row of Zdot^T): the row's residues become FP64 (or the row is read as FP64),
// the row's largest |sigma' z| and |sqrt|c| z| give its scales, and the residues of both are written:
// the operand of the next layer's product and the two operands of the symmetric product, which
// takes sqrt|c| z on both sides (sign(c) on one) so that one scale per row fits every column.
// Bound: 96 bytes written per element (16 residues x 3 operands) and about 450 instructions; four of them
// on the FP64 pipe.
// DE: the next layer's weights have column exponents.
template <bool CRT, bool DE>
__global__ void __launch_bounds__(256) k_rns_rows(const __grid_constant__ RnsSet set,
                                                  const RnsRows a) {
  __shared__ int sh[8];
  const int r = blockIdx.x;
  double* zrow = a.Z + (size_t)r * a.ldz;
  griddep_wait();
  griddep_launch();
  const double sb = CRT ? set.scale * a.sb[r] : 0.0;
  int ha = 0, hs = 0;
  for (int k = 4 * threadIdx.x; k < a.K; k += 4 * blockDim.x) {
    double z[4];
    if (CRT) {
      Crt t[4];
      const unsigned char* c = a.C + (size_t)r * a.ldc + k;
      const size_t plane = (size_t)a.n * a.ldc;
#pragma unroll 4
      for (int i = 0; i < kRns; ++i) {
        const unsigned y = __ldg(reinterpret_cast<const unsigned*>(c + i * plane));
        t[0].add(set, i, y & 0xFFu);
        t[1].add(set, i, (y >> 8) & 0xFFu);
        t[2].add(set, i, (y >> 16) & 0xFFu);
        t[3].add(set, i, y >> 24);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) z[j] = t[j].value() * sb * __ldg(a.sa + k + j);
      *reinterpret_cast<double2*>(zrow + k) = make_double2(z[0], z[1]);
      *reinterpret_cast<double2*>(zrow + k + 2) = make_double2(z[2], z[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) z[j] = zrow[k + j];
    }
    int d[4];
    if (DE) *reinterpret_cast<int4*>(d) = __ldg(reinterpret_cast<const int4*>(a.de + k));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (a.At) {
        const int e = prod_expo(__ldg(a.s1 + k + j), z[j]);
        ha = max(ha, DE ? shift_expo(e, d[j]) : e);
      }
      if (a.Sa) hs = max(hs, prod_expo(__ldg(a.rc + k + j), z[j]));
    }
  }
  if (!a.At && !a.Sa) return;
  int sca, scs;
  ha = block_max(ha, sh);
  hs = block_max(hs, sh);
  const double ba = rns_scale(ha, set.bits, &sca), bs = rns_scale(hs, set.bits, &scs);
  if (threadIdx.x == 0) {
    if (a.At) a.sat[r] = ba;
    if (a.Sa) a.ss[r] = bs;
  }
  const size_t plane = (size_t)a.n * a.K;
  for (int k = 4 * threadIdx.x; k < a.K; k += 4 * blockDim.x) {
    double z[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) z[j] = zrow[k + j];
    const size_t o = (size_t)r * a.K + k;
    if (a.At) {
      Limbs l[4];
      int d[4] = {0, 0, 0, 0};
      if (DE) *reinterpret_cast<int4*>(d) = __ldg(reinterpret_cast<const int4*>(a.de + k));
#pragma unroll
      for (int j = 0; j < 4; ++j) l[j] = rns_limbs(to_int(__ldg(a.s1 + k + j) * z[j], sca + d[j]));
      __nv_bfloat16* dst = (__nv_bfloat16*)a.At + o;
#pragma unroll 4
      for (int i = 0; i < kRns; ++i)
        *reinterpret_cast<uint2*>(dst + i * plane) =
            make_uint2(bf2(rns_res(set, i, l[0]), rns_res(set, i, l[1])),
                       bf2(rns_res(set, i, l[2]), rns_res(set, i, l[3])));
    }
    if (a.Sa) {
      Limbs l[4];
      unsigned neg0, neg1;   // sign bits of c, in the places of the packed BF16 pairs
      {
        unsigned s4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s4[j] = (unsigned)__double2hiint(__ldg(a.c + k + j)) & 0x80000000u;
          l[j] = rns_limbs(to_int(__ldg(a.rc + k + j) * z[j], scs));
        }
        neg0 = (s4[0] >> 16) | s4[1];
        neg1 = (s4[2] >> 16) | s4[3];
      }
      __nv_bfloat16 *da = (__nv_bfloat16*)a.Sa + o, *db = (__nv_bfloat16*)a.Sb + o;
#pragma unroll 4
      for (int i = 0; i < kRns; ++i) {
        float v[4], w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          v[j] = rns_res(set, i, l[j]);
          w[j] = rns_mod(v[j] * set.q[i], set.p[i], set.pinv[i]);
        }
        *reinterpret_cast<uint2*>(da + i * plane) = make_uint2(bf2(w[0], w[1]), bf2(w[2], w[3]));
        *reinterpret_cast<uint2*>(db + i * plane) =
            make_uint2(bf2(v[0], v[1]) ^ neg0, bf2(v[2], v[3]) ^ neg1);
      }
    }
  }
}

// ------------------------------------------------------------------ reverse rows
// One cluster of eight CTAs per seed column s: Abar[k][s] from the residue planes of W_l^T Zbar (or,
// for the output layer, the seeds), then sigma' Abar of the layer below as residues, one scale per
// seed (the row scales of that layer's weights are multiplied in, since its product sums over rows).
// First layer: J and the gradient instead.  Bound: latency, so a thread has one column up to 4096, and
// its loads, 32 at a time, are in flight together.
// DE: the weights just multiplied have column exponents.
constexpr int kRevCl = 8;
template <bool DE>
__global__ void __launch_bounds__(512) k_rns_rev_rows(const __grid_constant__ RnsSet set,
                                                      const RnsRev a) {
  __shared__ int sh[16], mine;
  const int s = blockIdx.y;
  const int k0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  const bool is_lam = s == a.lam_col;
  double* zrow = a.Zs + (size_t)s * a.K;
  griddep_wait();
  griddep_launch();
  int ex = 0;
  double keep = 0.0;   // of column k0
  for (int k = k0; k < a.K; k += step) {
    double z;
    if (a.C) {
      const int de = DE ? __ldg(a.de + k) : 0;
      Crt t;
      const unsigned char* c = a.C + (size_t)s * a.K + k;
      const size_t plane = (size_t)a.seeds * a.K;
      for (int i0 = 0; i0 < kRns; i0 += 8) {
        unsigned y[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int c0 = 0; c0 < a.chunks; c0 += 4) {
          unsigned q[8][4];
#pragma unroll
          for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int w = 0; w < 4; ++w)
              q[u][w] = c0 + w < a.chunks ? __ldg(c + (size_t)((c0 + w) * kRns + i0 + u) * plane) : 0u;
#pragma unroll
          for (int u = 0; u < 8; ++u) y[u] += q[u][0] + q[u][1] + q[u][2] + q[u][3];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          float r = rns_mod((float)y[u], set.p[i0 + u], set.pinv[i0 + u]);
          r += r < 0.f ? set.p[i0 + u] : 0.f;
          t.add(set, i0 + u, __float_as_uint(r + 8388608.f) & 0x1FFu);
        }
      }
      double v = t.value() * (set.scale * a.sb[s]);
      if (DE) v *= __hiloint2double((de + 1023) << 20, 0);
      if (!a.s1) {
        if (k < a.kvalid) {
          if (a.J && s < a.nJ) a.J[(size_t)s * a.kvalid + k] = v;
          if (a.g && is_lam) a.g[k] = v;
        }
        continue;
      }
      z = a.s1[k] * v;
      if (is_lam) {
        const double cv = a.s2[k] * v;
        a.c_out[k] = cv;
        if (a.rc_out) a.rc_out[k] = sqrt(fabs(cv));
      }
    } else {
      double cv = 0.0;
      z = k < a.kvalid ? out_seed(k, s, a.kvalid, a.nJ, a.lam_col, a.s1, a.s2, a.lam, a.soft_p, &cv) : 0.0;
      if (is_lam) {
        a.c_out[k] = cv;
        if (a.rc_out) a.rc_out[k] = sqrt(fabs(cv));
      }
    }
    z *= a.sa[k];
    ex = max(ex, expo(z));
    if (k == k0) keep = z;
    else zrow[k] = z;
  }
  if (a.C && !a.s1) return;   // the whole cluster: nothing is exchanged on the first layer
  ex = block_max(ex, sh);
  if (threadIdx.x == 0) mine = ex;
  __syncthreads();
  async::cluster_sync();
  for (int q = 0; q < kRevCl; ++q)
    ex = max(ex, __float_as_int(async::ld_dsmem_f32(smem_u32(&mine), (uint32_t)q)));
  async::cluster_sync();      // no CTA leaves while another still reads its shared memory
  int sc;
  const double back = rns_scale(ex, set.bits, &sc);
  if (blockIdx.x == 0 && threadIdx.x == 0) a.sb_out[s] = back;
  for (int k = k0; k < a.K; k += step) {
    const Limbs l = rns_limbs(to_int(k == k0 ? keep : zrow[k], sc));
    __nv_bfloat16* dst = (__nv_bfloat16*)a.Zr + (size_t)s * a.K + k;
    const size_t plane = (size_t)a.seeds * a.K;
#pragma unroll 4
    for (int i = 0; i < kRns; ++i)
      dst[i * plane] = __ushort_as_bfloat16((unsigned short)(__float_as_uint(rns_res(set, i, l)) >> 16));
  }
}

__global__ void k_rns_softmax_ext(int n, int m, int col, const double* __restrict__ p,
                                  const double* __restrict__ lam, double* __restrict__ Z, int ldz,
                                  double* __restrict__ c, double* __restrict__ rc) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  griddep_wait();
  griddep_launch();
  if (j >= n) return;
  double lb = 0.0;
  for (int i = 0; i < m; ++i) lb += lam[i] * p[i];
  const double r = sqrt(lb * lb + 1.0);
  const double g[2] = {lb + r, lb - r};
  double w[2] = {0.0, 0.0};
  for (int i = 0; i < m; ++i) {
    const double z = Z[(size_t)j * ldz + i];
    const double pl = p[i] * lam[i];
#pragma unroll
    for (int k = 0; k < 2; ++k) w[k] += z * (p[i] + (2.0 * lb - g[k]) * pl);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double t = 2.0 * lb - g[k], gp = g[k] / (1.0 + t * t);
    Z[(size_t)j * ldz + col + k] = w[k];
    if (j == 0) {
      c[col + k] = gp;
      rc[col + k] = sqrt(fabs(gp));
    }
  }
}

// ------------------------------------------------------------------ H from the residue planes
__global__ void __launch_bounds__(256) k_rns_h(const __grid_constant__ RnsSet s, int layers,
                                               const unsigned char* __restrict__ U, int ldu,
                                               const double* __restrict__ ss, int n,
                                               double* __restrict__ H) {
  __shared__ double t[8][129];
  const int i0 = blockIdx.x * 128, j0 = blockIdx.y * 8;
  griddep_wait();
  griddep_launch();
  if (i0 + 127 < j0) return;           // strictly above the diagonal
  const int x = threadIdx.x, y = threadIdx.y;
  const int i = i0 + 4 * x, j = j0 + y;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (j < n && i < n) {
    for (int l = 0; l < layers; ++l) {
      const unsigned char* u = U + ((size_t)l * kRns * n + j) * ldu + i;
      const size_t plane = (size_t)n * ldu;
      Crt r[4];
#pragma unroll 4
      for (int q = 0; q < kRns; ++q) {
        const unsigned b = __ldg(reinterpret_cast<const unsigned*>(u + q * plane));
        r[0].add(s, q, b & 0xFFu);
        r[1].add(s, q, (b >> 8) & 0xFFu);
        r[2].add(s, q, (b >> 16) & 0xFFu);
        r[3].add(s, q, b >> 24);
      }
      const double* sl = ss + (size_t)l * n;
      const double sj = s.scale * sl[j];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k < n) v[k] = fma(r[k].value() * sj, sl[i + k], v[k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k < n && i + k >= j) H[(size_t)j * n + i + k] = v[k];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) t[y][4 * x + k] = v[k];
  __syncthreads();
  // mirror: rows i0 .. i0 + 127, columns j0 .. j0 + 7
  for (int e = threadIdx.y * 32 + threadIdx.x; e < 128 * 8; e += 256) {
    const int ii = i0 + e / 8, jj = j0 + e % 8;
    if (ii < n && jj < n && ii > jj) H[(size_t)ii * n + jj] = t[e % 8][e / 8];
  }
}

// ------------------------------------------------------------------ residue GEMM
// Persistent: CTA b takes the (modulus, tile) pairs b, b + gridDim.x, ... of 128 x BN tiles.  Warp 0
// copies the operands (TMA, 64-element K blocks, 128-byte swizzle) through a ring of stages, warp 1
// issues the MMAs into one of two TMEM accumulators, which it changes every 1024 terms of K, and
// eight epilogue warps (two per 32-lane TMEM quadrant, each half of the columns) reduce the finished
// accumulator mod p into registers while the next one fills; after a tile's last accumulator they
// store its residues, one byte each.
// Bound: the tensor pipe.  A reduction costs three FP32 operations per element and 1024 terms of K,
// 0.2 of the MMA time on 8 warps, and runs under the next accumulator's MMAs; the tile is as wide as
// two accumulators in TMEM allow.
//
// REV: the reverse sweep's product W^T Zbar over the rows of W, BN = 16, 32 or 48 seed columns.  A is
// the same residue array read the other way round: its stages are two boxes of 64 rows x 64 columns,
// which the MMA takes as an MN-major operand.  Each item is one 128-column strip of one modulus and
// one chunk of up to 1024 rows, whose residues go to a plane of their own (the reader adds the
// chunks).  Bound: HBM, 32 bytes per weight; up to 12 stages of 18 KB keep 200 KB per SM in flight.
constexpr int kGBM = 128, kGBK = 64;
constexpr int kGThreads = 320;                 // producer, MMA, eight epilogue warps
constexpr int kGChunk = 1024 / kGBK;           // K blocks that add up exactly

struct RnsGemm {
  int chunks;            // REV: chunks of 1024 rows
  int M, N, nkb, lower, ntm, ntn, tiles, a_rows, b_rows;
  unsigned char* C;
  int ldc;
  int* err;
  float p[kRns], pinv[kRns];
};

template <int BN, bool REV>
struct GCfg {
  static constexpr int STAGE = (kGBM + BN) * 128;
  static constexpr int FIT = (227 * 1024 - 2048) / STAGE, CAP = REV ? 12 : 6;
  static constexpr int STAGES = FIT > CAP ? CAP : FIT;
  static constexpr int SMEM = STAGES * STAGE + 1024 + 256;
  static_assert((2 * STAGES + 5) * 8 + 12 <= 256, "barriers fit behind the stages");
  // FP32 sums of BF16 products, A MN-major (bit 15) in the reverse sweep
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (REV ? 1u << 15 : 0u) |
                                    ((uint32_t)(kGBM >> 4) << 24);
  static_assert(BN % 16 == 0 && BN <= 256 && (BN * 128) % 1024 == 0, "tile width");
};

// Descriptor of an MN-major operand in 128-byte swizzled rows of 64 elements: 8 rows of K per KB
// (stride byte offset 1024), the next 64 elements of M `lbo` bytes on.
__device__ __forceinline__ uint64_t sdesc_mn(uint32_t addr, uint32_t lbo) {
  return sdesc<2, 1024>(addr) | ((uint64_t)(lbo >> 4) << 16);
}

template <int BN, bool REV>
__global__ void __launch_bounds__(kGThreads, 1)
    k_rns_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
               const __grid_constant__ RnsGemm g) {
  using C = GCfg<BN, REV>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + C::STAGES * C::STAGE);
  uint64_t* empty = full + C::STAGES;
  uint64_t* accf = empty + C::STAGES;   // [2]: accumulator b holds finished sums
  uint64_t* tfree = accf + 2;           // [2]: the epilogue has read accumulator b
  uint64_t* mdone = tfree + 2;          // every MMA issued has completed
  uint32_t* tmem_slot = (uint32_t*)(mdone + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  volatile int* consumed_sh = (volatile int*)(tmem_slot + 2);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per_mod = g.tiles, total = g.tiles * kRns;
  // REV: tn is the chunk of rows
  auto decode = [&](int t, int& mod, int& tm, int& tn) {
    mod = t / per_mod;
    int r = t - mod * per_mod;
    if (g.lower) {          // BN = 128: row tm holds the tiles tn = 0 .. tm
      tm = 0;
      while (r > tm) r -= ++tm;
      tn = r;
    } else {
      tn = r / g.ntm;
      tm = r - tn * g.ntm;
    }
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&accf[b]), 1);
      mbar_init(smem_u32(&tfree[b]), 8);   // one arrival per epilogue warp
    }
    mbar_init(smem_u32(mdone), 1);
    *abort_flag = 0;
    *consumed_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  griddep_wait();     // the operands are written, and the last reader of C is done
  griddep_launch();

  int issued = 0;  // producer only
  if (warp == 0) {
    if (lane == 0) {
      int i = 0;
      bool stop = false;
      for (int t = blockIdx.x; t < total && !stop; t += gridDim.x) {
        int mod, tm, tn;
        decode(t, mod, tm, tn);
        const int kb_beg = REV ? tn * kGChunk : 0;
        const int kb_end = REV ? min(g.nkb, kb_beg + kGChunk) : g.nkb;
        const int ar = mod * g.a_rows + (REV ? 0 : tm * kGBM);
        const int br = mod * g.b_rows + (REV ? 0 : tn * BN);
        for (int kb = kb_beg; kb < kb_end; ++kb, ++i) {
          const int s = i % C::STAGES;
          const uint32_t ph = (uint32_t)(i / C::STAGES) & 1u;
          if (!mbar_wait(smem_u32(&empty[s]), ph ^ 1u, g.err, 71, abort_flag)) {
            stop = true;
            break;
          }
          uint8_t* st = smem + s * C::STAGE;
          const uint32_t fb = smem_u32(&full[s]);
          mbar_expect_tx(fb, C::STAGE);
          if (REV) {
            tma_load_2d(smem_u32(st), &ta, fb, tm * kGBM, ar + kb * kGBK);
            tma_load_2d(smem_u32(st + kGBK * 128), &ta, fb, tm * kGBM + 64, ar + kb * kGBK);
          } else {
            tma_load_2d(smem_u32(st), &ta, fb, kb * kGBK, ar);
          }
          tma_load_2d(smem_u32(st + kGBM * 128), &tb, fb, kb * kGBK, br);
          issued = i + 1;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int i = 0, ai = 0;   // stages consumed, accumulators started
      bool stop = false;
      for (int t = blockIdx.x; t < total && !stop; t += gridDim.x) {
        int mod, tm, tn;
        decode(t, mod, tm, tn);
        const int n_eff = REV ? BN : (min(BN, g.N - tn * BN) + 15) / 16 * 16;
        const uint32_t idesc = C::IDESC | ((uint32_t)(n_eff >> 3) << 17);
        const int kb_beg = REV ? tn * kGChunk : 0;
        const int kb_end = REV ? min(g.nkb, kb_beg + kGChunk) : g.nkb;
        for (int kb0 = kb_beg; kb0 < kb_end && !stop; kb0 += kGChunk, ++ai) {
          const int b = ai & 1;
          if (ai >= 2 &&
              !mbar_wait(smem_u32(&tfree[b]), (uint32_t)((ai - 2) >> 1) & 1u, g.err, 72, abort_flag)) {
            stop = true;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(b * 256);
          const int kb1 = min(g.nkb, kb0 + kGChunk);
          for (int kb = kb0; kb < kb1; ++kb, ++i) {
            const int s = i % C::STAGES;
            const uint32_t ph = (uint32_t)(i / C::STAGES) & 1u;
            if (!mbar_wait(smem_u32(&full[s]), ph, g.err, 73, abort_flag)) {
              stop = true;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + s * C::STAGE), sb = sa + kGBM * 128;
#pragma unroll
            for (int kk = 0; kk < kGBK / 16; ++kk)
              umma_bf16(d, REV ? sdesc_mn(sa + kk * 16 * 128, kGBK * 128) : sdesc<2, 1024>(sa + kk * 32),
                        sdesc<2, 1024>(sb + kk * 32), idesc,
                        (kb > kb0 || kk > 0) ? 1u : 0u);
            umma_commit(smem_u32(&empty[s]));
          }
          if (!stop) umma_commit(smem_u32(&accf[b]));
        }
      }
      *consumed_sh = i;
      umma_commit(smem_u32(mdone));
    }
  } else {
    const int q = warp & 3;              // TMEM lanes 32q .. 32q + 31 belong to this warp
    const int half = (warp - 2) >> 2;    // columns half * BN / 2 ..
    constexpr int NH = BN / 2;
    int ai = 0;
    bool stop = false;
    for (int t = blockIdx.x; t < total && !stop; t += gridDim.x) {
      int mod, tm, tn;
      decode(t, mod, tm, tn);
      const int n_eff = REV ? g.N : min(BN, g.N - tn * BN);
      const float p = g.p[mod], pinv = g.pinv[mod];
      float res[NH];
#pragma unroll
      for (int j = 0; j < NH; ++j) res[j] = 0.f;
      const int kb_beg = REV ? tn * kGChunk : 0;
      const int kb_end = REV ? min(g.nkb, kb_beg + kGChunk) : g.nkb;
      for (int kb0 = kb_beg; kb0 < kb_end; kb0 += kGChunk, ++ai) {
        const int b = ai & 1;
        const bool ok = mbar_wait(smem_u32(&accf[b]), (uint32_t)(ai >> 1) & 1u, g.err, 74, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) {
          stop = true;
          break;
        }
        tc_fence_after();
        const uint32_t src = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * 256 + half * NH);
#pragma unroll
        for (int c0 = 0; c0 < NH; c0 += 8) {
          if (half * NH + c0 < n_eff) {
            uint32_t v[8];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                  "=r"(v[7])
                : "r"(src + (uint32_t)c0));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 8; ++j) res[c0 + j] += rns_mod(__uint_as_float(v[j]), p, pinv);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tfree[b]));
      }
      if (stop) break;
      const int n0 = (REV ? 0 : tn * BN) + half * NH;
      const size_t plane = REV ? (size_t)(tn * kRns + mod) * BN : (size_t)mod * g.N;
      unsigned char* dst = g.C + (plane + n0) * g.ldc + tm * kGBM + q * 32 + lane;
#pragma unroll
      for (int j = 0; j < NH; ++j) {
        if (n0 + j < g.N) {
          float r = rns_mod(res[j], p, pinv);
          r += r < 0.f ? p : 0.f;
          dst[(size_t)j * g.ldc] = (unsigned char)__float_as_uint(r + 8388608.f);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1 && lane == 0) {
    volatile int no_abort = 0;
    mbar_wait(smem_u32(mdone), 0, g.err, 76, &no_abort, *abort_flag ? kWaitCycles / 8 : kWaitCycles);
  }
  if (*abort_flag && warp == 0 && lane == 0) {
    for (int i = *consumed_sh; i < issued; ++i) {
      volatile int no_abort = 0;
      mbar_wait(smem_u32(&full[i % C::STAGES]), (uint32_t)(i / C::STAGES) & 1u, g.err, 77, &no_abort,
                kWaitCycles / 8);
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  }
}

PFN_cuTensorMapEncodeTiled_v12000 rns_encode() {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
          cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    return nullptr;
  return (PFN_cuTensorMapEncodeTiled_v12000)p;
}

bool rns_map(CUtensorMap* m, const void* base, long long rows, int cols, int box_rows) {   // 64-column boxes
  auto enc = rns_encode();
  if (!enc || !base) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kGBK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, bool REV = false>
cudaError_t launch_gemm(const RnsPlan& p, const RnsGemm& g, int grid, cudaStream_t st) {
  using C = GCfg<BN, REV>;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(k_rns_gemm<BN, REV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         C::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  return launch_pdl(k_rns_gemm<BN, REV>, dim3(grid), dim3(kGThreads), C::SMEM, st, p.ta, p.tb, g);
}

}  // namespace

RnsSet rns_set(int K) {
  // 16 moduli leave 57 bits at K = 1024, 56 at 4096 and 54 at 65664.  Error of J, the gradient and H against
  // 128-bit sums, FP64 products / 15 moduli (four bits less) / 16: 30 -> 1100 x 2 -> 3 4.5e-16 1.2e-15 3.1e-16,
  // 4.1e-16 1.3e-15 2.7e-16, 1.2e-15 1.3e-15 4.0e-16; 16 -> 4096 x 2 -> 3 5.9e-16 1.9e-15 3.0e-16, 5.3e-16
  // 1.6e-15 2.5e-16, 1.8e-15 2.0e-15 3.6e-16.  So 15, with 784 -> 4096 x 7 -> 10 in 3.86 ms instead of 4.00, would
  // be less exact than FP64 products.
  RnsSet s;
  double bits = 0.0;
  unsigned __int128 P = 1;   // below 2^126; a product in FP64 would round fifteen times, the same way for all
  for (int i = 0; i < kRns; ++i) {
    bits += std::log2((double)kModuli[i]);
    P *= (unsigned)kModuli[i];
  }
  s.scale = std::ldexp((double)P, -64);
  s.bits = std::min(60, (int)std::floor((bits - 1.0 - std::log2((double)K)) / 2.0 - 1e-9));
  auto sym = [](long long v, int p) {
    v %= p;
    return (float)(v > p / 2 ? v - p : v);
  };
  for (int i = 0; i < kRns; ++i) {
    const int p = kModuli[i];
    s.p[i] = (float)p;
    s.pinv[i] = 1.0f / (float)p;
    const long long r16 = 65536 % p, r32 = r16 * r16 % p, r48 = r32 * r16 % p;
    s.r16[i] = sym(r16, p);
    s.r32[i] = sym(r32, p);
    s.r48[i] = sym(r48, p);
    long long m = 1;
    for (int j = 0; j < kRns; ++j)
      if (j != i) m = m * (kModuli[j] % p) % p;
    long long inv = 1;
    while (m * inv % p != 1) ++inv;   // the moduli are pairwise coprime
    s.q[i] = sym(inv, p);
    const unsigned __int128 c = ((((unsigned __int128)1) << 97) / p + 1) / 2;
    s.c0[i] = (unsigned)c;
    s.c1[i] = (unsigned)(c >> 32);
    s.c2[i] = (unsigned)(c >> 64);
  }
  return s;
}

int rns_plan(RnsPlan& p, const void* A, int a_rows, const void* B, int b_rows, int M, int N, int K,
             bool lower) {
  p = RnsPlan();
  if (K % kGBK || K <= 0 || M <= 0 || N <= 0 || N > b_rows) return NNC_ERR_ARG;
  p.M = M;
  p.N = N;
  p.nkb = K / kGBK;
  p.a_rows = a_rows;
  p.b_rows = b_rows;
  p.lower = lower ? 1 : 0;
  // tile width: the least padded work, a tile counting 8 columns of overhead and at least 96 (narrower
  // MMAs are bound by reading A from shared memory)
  p.bn = 128;
  if (!lower) {
    long long best = -1;
    for (int bn : {128, 208, 256}) {
      long long cost = 0;
      for (int n = 0; n < N; n += bn) cost += std::max((std::min(bn, N - n) + 15) / 16 * 16, 96) + 8;
      if (best < 0 || cost < best) {
        best = cost;
        p.bn = bn;
      }
    }
  }
  if (!rns_map(&p.ta, A, (long long)kRns * a_rows, K, kGBM) ||
      !rns_map(&p.tb, B, (long long)kRns * b_rows, K, p.bn))
    return NNC_ERR_CUDA;
  p.ready = true;
  return NNC_OK;
}

int rns_plan_rev(RnsPlan& p, const void* W, int mp, int kp, const void* Z, int seeds) {
  p = RnsPlan();
  if (mp % 128 || kp % 128 || seeds < 1 || seeds > 48) return NNC_ERR_ARG;
  p.M = kp;
  p.nkb = mp / kGBK;
  p.bn = (seeds + 15) / 16 * 16;
  p.N = p.bn;
  p.a_rows = mp;
  p.b_rows = p.bn;
  p.rev = 1;
  if (!rns_map(&p.ta, W, (long long)kRns * mp, kp, kGBK) ||
      !rns_map(&p.tb, Z, (long long)kRns * p.bn, mp, p.bn))
    return NNC_ERR_CUDA;
  p.ready = true;
  return NNC_OK;
}

cudaError_t rns_gemm(const RnsPlan& p, const RnsSet& s, unsigned char* C, int ldc, int* err,
                     int sm_count, cudaStream_t st) {
  RnsGemm g{};
  g.ntm = (p.M + kGBM - 1) / kGBM;
  g.chunks = (p.nkb + kGChunk - 1) / kGChunk;
  g.ntn = p.rev ? g.chunks : (p.N + p.bn - 1) / p.bn;
  if (!p.ready || ldc < g.ntm * kGBM) return cudaErrorInvalidValue;
  g.M = p.M;
  g.N = p.N;
  g.nkb = p.nkb;
  g.lower = p.lower;
  g.tiles = p.lower ? g.ntm * (g.ntm + 1) / 2 : g.ntm * g.ntn;
  g.a_rows = p.a_rows;
  g.b_rows = p.b_rows;
  g.C = C;
  g.ldc = ldc;
  g.err = err;
  for (int i = 0; i < kRns; ++i) {
    g.p[i] = s.p[i];
    g.pinv[i] = s.pinv[i];
  }
  const int grid = std::min(sm_count, g.tiles * kRns);
  switch (p.rev ? -p.bn : p.bn) {
    case -16: return launch_gemm<16, true>(p, g, grid, st);
    case -32: return launch_gemm<32, true>(p, g, grid, st);
    case -48: return launch_gemm<48, true>(p, g, grid, st);
    case 128: return launch_gemm<128>(p, g, grid, st);
    case 208: return launch_gemm<208>(p, g, grid, st);
    case 256: return launch_gemm<256>(p, g, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

size_t rns_even_scratch(int k) { return (size_t)k * 16 + 24; }

cudaError_t rns_even_out(const RnsSet& s, const double* W, int ldw, int m, int k, void* scratch, int* de,
                         int* flags, cudaStream_t st) {
  RnsEven e;
  e.sum = (unsigned long long*)scratch;
  e.total = e.sum + k;
  e.cnt = (int*)(e.total + 3);
  e.small = e.cnt + k;
  const cudaError_t r = cudaMemsetAsync(scratch, 0, rns_even_scratch(k), st);
  if (r != cudaSuccess) return r;
  k_rns_colsum<<<dim3((k + 31) / 32, (m + kEvenRows - 1) / kEvenRows), dim3(32, 8), 0, st>>>(W, ldw, m, k, e,
                                                                                             flags);
  k_rns_colexp<<<(k + 255) / 256, 256, 0, st>>>(m, k, e, de, flags);
  k_rns_spread<<<m, 256, 0, st>>>(W, ldw, k, s.bits, de, e, flags);
  k_rns_colspread<<<(k + 255) / 256, 256, 0, st>>>(k, e, flags);
  note_launch(4);
  return cudaGetLastError();
}

cudaError_t rns_pack_weights(const RnsSet& s, const double* W, int mp, int kp, const int* de, void* res,
                             double* sa, cudaStream_t st) {
  k_rns_pack<<<mp, 256, 0, st>>>(s, W, mp, kp, de, (__nv_bfloat16*)res, sa);
  note_launch();
  return cudaGetLastError();
}

cudaError_t rns_rows(const RnsSet& s, const RnsRows& a, cudaStream_t st) {
  if (a.K % 128 || a.n < 1 || (a.ldz & 1)) return cudaErrorInvalidValue;
  const int threads = std::min(256, std::max(32, a.K / 4));
  auto kernel = a.At && a.de ? (a.C ? k_rns_rows<true, true> : k_rns_rows<false, true>)
                             : (a.C ? k_rns_rows<true, false> : k_rns_rows<false, false>);
  return launch_pdl(kernel, dim3(a.n), dim3(threads), 0, st, s, a);
}

cudaError_t rns_rev_rows(const RnsSet& s, const RnsRev& a, int S, cudaStream_t st) {
  if (a.K % 128 || S < 1 || S > a.seeds) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kRevCl, S);
  cfg.blockDim = dim3(std::min(512, std::max(32, (a.K / kRevCl + 31) / 32 * 32)));
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kRevCl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, a.C && a.de ? k_rns_rev_rows<true> : k_rns_rev_rows<false>, s, a);
  note_launch();
  const cudaError_t last = cudaGetLastError();
  return e != cudaSuccess ? e : last;
}

cudaError_t rns_softmax_ext(int n, int m, int col, const double* p, const double* lam, double* Z,
                            int ldz, double* c, double* rc, cudaStream_t st) {
  return launch_pdl(k_rns_softmax_ext, dim3((n + 127) / 128), dim3(128), 0, st, n, m, col, p, lam, Z, ldz, c,
                    rc);
}

cudaError_t rns_h_finish(const RnsSet& s, int layers, const unsigned char* U, int ldu,
                         const double* ss, int n, double* H, cudaStream_t st) {
  dim3 grid((n + 127) / 128, (n + 7) / 8);
  return launch_pdl(k_rns_h, grid, dim3(32, 8), 0, st, s, layers, U, ldu, ss, n, H);
}

}  // namespace nnc
