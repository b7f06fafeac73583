// FP64-grade matrix products on the BF16 tensor cores.
//
// FP64 runs at 1.9 FMA/clk/SM on this GPU (1.2 TFLOP/s); BF16 tensor cores at about 1.7
// PFLOP/s.  A product C = A B^T of FP64 matrices is therefore formed from digits.  With
// 2^E the power of two just above a row's max |x|, an element is the integer
// V = round(x 2^(62 - E)) in 7 balanced base-512 digits d_0 .. d_6, each in [-256, 256] and so
// exact in BF16.  Digit products d_a e_b of order t = a + b <= 6 (28 of 49) accumulate in FP32
// tensor memory, one accumulator per order.  Over at most 64 terms of K an accumulator of
// order t <= 3 stays within 4 * 64 * 2^16 = 2^24, so its sum is exact whatever the data; the
// epilogue then moves all orders into a 79-bit fixed-point sum in units of 2^-58 (row max of
// A)(row max of B), and clears the accumulators for the next 64 terms.  The result is rounded to
// FP64 once.  Its error is about 2^-62 sqrt(K) of those maxima: what the dropped products of order
// 7 and the last bit of the fixed-point sum leave.  A plain FP64 sum rounds each of its K steps
// by 2^-53 of the running sum: less for an element whose own terms are all below 2^-9 of the maxima,
// more for all others (K of 12 and 40 centres against extended precision, units of 2^-53
// sqrt(K_mm K_nn): 15 to 28 at most with FP64 sums, 1.2 to 1.7 here).
// Slicing into digits whose products sum exactly is the scheme of Ozaki, Ogita, Oishi and Rump
// (error-free transformations of matrix multiplication, 2012), here with fixed-point digits per row
// and integer sums.
//
// Rows with an infinity or a NaN carry no digits; the epilogue recomputes the outputs of such
// rows and columns by plain FP64 dot products of the original operands.
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"

namespace dfscf {
namespace digits {

constexpr int NS = 7;        // digits per element
constexpr int BM = 128;      // rows of A per tile
constexpr int BK = 32;       // K per shared-memory stage (one 64-byte swizzle row)
constexpr int CHUNK = 64;    // K between two drains of the accumulators: exact orders 0..3

// Leading dimension (elements) of a digit plane over K: 16-byte rows for TMA.
inline long plane_ld(long K) { return (K + 7) / 8 * 8; }
inline size_t plane_bytes(long rows, long K) { return (size_t)NS * rows * plane_ld(K) * sizeof(__nv_bfloat16); }

// High word of |x| as the row-maximum key (0 only for x = 0; 0x7ff00000 and above: inf, NaN).
__device__ __forceinline__ unsigned high_key(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned h = (unsigned)(u >> 32) & 0x7fffffffu;
  return h ? h : ((unsigned)u ? 1u : 0u);
}
// Biased exponent field f of a row key (denormals count as 1): |x| < 2^(f - 1022).
__device__ __forceinline__ int key_field(unsigned key) { return max((int)(key >> 20), 1); }
__device__ __forceinline__ bool key_bad(unsigned key) { return key >= 0x7ff00000u; }

// The NS digits of x, most significant first, for a row of exponent field f.
__device__ __forceinline__ void split_digits(double x, int f, int (&d)[NS]) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int fx = (int)((u >> 52) & 0x7ffu);
  unsigned long long m = u & 0xfffffffffffffull;
  if (fx) m |= 1ull << 52;
  const int s = 9 * NS - 54 - (f - max(fx, 1));
  if (s >= 0) m <<= s;
  else if (s > -55) m = (m + (1ull << (-s - 1))) >> (-s);
  else m = 0;
  long long v = (long long)u < 0 ? -(long long)m : (long long)m;  // |v| <= 2^62
#pragma unroll
  for (int j = NS - 1; j >= 3; --j) {
    d[j] = ((int)v << 23) >> 23;
    v = (v + 256) >> 9;
  }
  int w = (int)v;  // the digits 0..2: at most 2^26
#pragma unroll
  for (int j = 2; j >= 1; --j) {
    d[j] = (w << 23) >> 23;
    w = (w + 256) >> 9;
  }
  d[0] = w;
}

// BF16 bits of two digits, a in the low half (integers up to 256 are exact).
__device__ __forceinline__ unsigned pack_digits(int a, int b) {
  const float fa = __int_as_float(0x4B400000 + a) - 12582912.0f, fb = __int_as_float(0x4B400000 + b) - 12582912.0f;
  return __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
}

// Eight consecutive K elements of a row into its NS planes (16-byte stores).
__device__ __forceinline__ void store_digits8(const double (&x)[8], int f, __nv_bfloat16* out, size_t plane) {
  unsigned w[NS][4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    int a[NS], b[NS];
    split_digits(x[2 * u], f, a);
    split_digits(x[2 * u + 1], f, b);
#pragma unroll
    for (int j = 0; j < NS; ++j) w[j][u] = pack_digits(a[j], b[j]);
  }
#pragma unroll
  for (int j = 0; j < NS; ++j) *reinterpret_cast<uint4*>(out + j * plane) = make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
}

}  // namespace digits

// Digit planes of a matrix operand [NS][rows][ld] over K, and the row keys.
struct DigitOperand {
  __nv_bfloat16* p = nullptr;
  unsigned* key = nullptr;
  long rows = 0, K = 0;
};
size_t digit_operand_bytes(long rows, long K);
DigitOperand digit_operand(void* mem, long rows, long K);

// Digits of op rows: element (r, k) = A[r * lda + k] (trans = false) or A[k * lda + r].
int slice_matrix(const double* A, long lda, bool trans, const DigitOperand& o, cudaStream_t s);
// Digits of rows r = (P, m), P = p0 .. p0 + np - 1, m < nao, of the symmetric matrices packed
// in rows P of B (row stride ldb), over n < nao.
int slice_packed(const double* B, long ldb, int nao, int p0, int np, const DigitOperand& o, cudaStream_t s);
// Digits of A with the row keys already in o.key.
int slice_with_keys(const double* A, long lda, const DigitOperand& o, cudaStream_t s);

// C[z][m][n] = alpha sum_k a_mk b_nk + beta C[z][m][n], K split in `splits` ranges (slices sC apart);
// DIGIT_LOWER: only tiles that reach n <= m; DIGIT_TRANSPOSED: C[n ldc + m], whose lanes store
// consecutive m.  A0 (a_mk = A0[m sam + k sak]) and B0 are the operands'
// FP64 originals.  err: device flag raised when a bounded wait gave up (C is then incomplete).
enum DigitShape { DIGIT_FULL = 0, DIGIT_LOWER = 1, DIGIT_TRANSPOSED = 2 };
struct DigitSource {
  const double* p;
  long sr, sk;
};
int digit_gemm(const DigitOperand& A, const DigitOperand& B, DigitSource A0, DigitSource B0, double alpha, double beta,
               double* C, long ldc, long sC, int splits, int shape, int* err, cudaStream_t s);
// Half-transform X[m][(P - p0) nocc + i] = sum_n B_P[m][n] C[n][i] (row stride ldx) of the rows
// of slice_packed, and xkey[m] = max over the row (atomicMax: zero it first).
int digit_half_transform(const DigitOperand& A, const DigitOperand& Ct, const double* B, long ldb, int nao, int p0,
                         const double* C, int nocc, double* X, long ldx, long xcol0, unsigned* xkey, int* err,
                         cudaStream_t s);
int digits_prepare();

}  // namespace dfscf
