// FP64 dense linear algebra on CUDA cores: a register-tiled GEMM (batched, split-K,
// lower-triangle-only), the blocked Cholesky factorisation of the Coulomb metric
// M = L L^T and the blocked forward substitution B = L^-1 R of the density-fitting
// whitening (arXiv 2506.06661, Section "Density fitting").  On this GPU FP64 runs at
// about 1.9 FMA/clk/SM, so these kernels are FP64-ALU bound by design; they only need
// coalesced loads and enough independent FMAs per thread.
#include <algorithm>

#include "common.cuh"
#include "digits.cuh"
#include "kernels.cuh"

namespace dfscf {

constexpr int GB_M = 64, GB_N = 64, GB_K = 16;

// C = alpha * op(A) op(B) + beta * C.
//   op(A)(m,k) = TA ? A[k*lda + m] : A[m*lda + k];  op(B)(k,n) = TB ? B[n*ldb + k] : B[k*ldb + n].
// blockIdx.z: batch index (strides sA, sB, sC) or, when kchunk > 0, a split of the K range
// [z*kchunk, min(K, (z+1)*kchunk)) with output slice C + z*sC.
// lower_only: tiles strictly above the diagonal are skipped.
template <bool TA, bool TB>
__global__ void __launch_bounds__(256) dgemm_kernel(int M, int N, int K, double alpha, const double* __restrict__ A,
                                                    long lda, long sA, const double* __restrict__ B, long ldb, long sB,
                                                    double beta, double* __restrict__ C, long ldc, long sC,
                                                    long kchunk, int lower_only) {
  int mt = blockIdx.y, nt = blockIdx.x;
  if (lower_only && mt < nt) return;
  __shared__ double As[GB_K][GB_M + 1];
  __shared__ double Bs[GB_K][GB_N + 1];
  long k_begin = 0, k_end = K;
  if (kchunk > 0) {
    k_begin = (long)blockIdx.z * kchunk;
    k_end = min((long)K, k_begin + kchunk);
    C += (size_t)blockIdx.z * sC;
  } else {
    A += (size_t)blockIdx.z * sA;
    B += (size_t)blockIdx.z * sB;
    C += (size_t)blockIdx.z * sC;
  }
  int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  int m0 = mt * GB_M, n0 = nt * GB_N;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;

  for (long k0 = k_begin; k0 < k_end; k0 += GB_K) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int idx = threadIdx.x + 256 * r;
      int mm, kk;
      if (TA) { kk = idx >> 6; mm = idx & 63; } else { mm = idx >> 4; kk = idx & 15; }
      long gk = k0 + kk;
      int gm = m0 + mm;
      double v = 0.0;
      if (gm < M && gk < k_end) v = TA ? A[gk * lda + gm] : A[(long)gm * lda + gk];
      As[kk][mm] = v;
      int nn;
      if (TB) { nn = idx >> 4; kk = idx & 15; } else { kk = idx >> 6; nn = idx & 63; }
      gk = k0 + kk;
      int gn = n0 + nn;
      v = 0.0;
      if (gn < N && gk < k_end) v = TB ? B[(long)gn * ldb + gk] : B[gk * ldb + gn];
      Bs[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GB_K; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int gm = m0 + ty + 16 * i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int gn = n0 + tx + 16 * j;
      if (gn >= N) continue;
      double* c = C + (long)gm * ldc + gn;
      *c = (beta == 0.0) ? alpha * acc[i][j] : fma(alpha, acc[i][j], beta * *c);
    }
  }
}

// The same product in tiles of 16 x 8, one output per thread.  FP64 issues one warp instruction per
// 64 clocks on each partition of an SM, so four warps fill it and a tile's time is its share of
// the multiplications: 300^3 in 64 x 64 tiles put them on 25 of 152 SMs, 309 us; in 16 x 8 tiles
// 722 CTAs spread over all of them, 52 us (48 are the FP64 units' own); 100^3 125 us, now 11.  The
// tiles of the next 32 of K are on their way while this one's are multiplied.
constexpr int GS_M = 16, GS_N = 8, GS_K = 32;
template <bool TA, bool TB>
__global__ void __launch_bounds__(128) dgemm_small_kernel(int M, int N, int K, double alpha, const double* __restrict__ A,
                                                          long lda, long sA, const double* __restrict__ B, long ldb,
                                                          long sB, double beta, double* __restrict__ C, long ldc,
                                                          long sC) {
  __shared__ double As[GS_K][GS_M + 1], Bs[GS_K][GS_N + 1];
  A += (size_t)blockIdx.z * sA;
  B += (size_t)blockIdx.z * sB;
  C += (size_t)blockIdx.z * sC;
  const int tid = threadIdx.x, tx = tid % GS_N, ty = tid / GS_N;
  const int m0 = blockIdx.y * GS_M, n0 = blockIdx.x * GS_N;
  double a[4], b[2], acc = 0.0;
  auto fetch = [&](int k0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int q = tid + 128 * r, mm = TA ? q % GS_M : q / GS_K, kk = TA ? q / GS_M : q % GS_K;
      const long gm = m0 + mm, gk = k0 + kk;
      a[r] = gm < M && gk < K ? (TA ? A[gk * lda + gm] : A[gm * lda + gk]) : 0.0;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int q = tid + 128 * r, nn = TB ? q / GS_K : q % GS_N, kk = TB ? q % GS_K : q / GS_N;
      const long gn = n0 + nn, gk = k0 + kk;
      b[r] = gn < N && gk < K ? (TB ? B[gn * ldb + gk] : B[gk * ldb + gn]) : 0.0;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < K; k0 += GS_K) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int q = tid + 128 * r;
      As[TA ? q / GS_M : q % GS_K][TA ? q % GS_M : q / GS_K] = a[r];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int q = tid + 128 * r;
      Bs[TB ? q % GS_K : q / GS_N][TB ? q / GS_K : q % GS_N] = b[r];
    }
    __syncthreads();
    if (k0 + GS_K < K) fetch(k0 + GS_K);
    if (k0 + GS_K <= K) {
#pragma unroll
      for (int kk = 0; kk < GS_K; ++kk) acc = fma(As[kk][ty], Bs[kk][tx], acc);
    } else {
      for (int kk = 0; kk < K - k0; ++kk) acc = fma(As[kk][ty], Bs[kk][tx], acc);
    }
  }
  const int gm = m0 + ty, gn = n0 + tx;
  if (gm >= M || gn >= N) return;
  double* c = C + (size_t)gm * ldc + gn;
  *c = beta == 0.0 ? alpha * acc : fma(alpha, acc, beta * *c);
}

int dgemm(bool ta, bool tb, int M, int N, int K, double alpha, const double* A, long lda, long sA, const double* B,
          long ldb, long sB, double beta, double* C, long ldc, long sC, int batch, cudaStream_t s, long kchunk,
          int lower_only) {
  if (M <= 0 || N <= 0 || batch <= 0) return DF_OK;
  dim3 grid((N + GB_N - 1) / GB_N, (M + GB_M - 1) / GB_M, batch);
  DF_REQUIRE(grid.y <= 65535 && grid.z <= 65535, DF_ERR_ARG, "dgemm: grid too large (M=%d batch=%d)", M, batch);
  // Few large tiles leave SMs idle; up to about four per SM the small ones spread better, and their
  // reads (3 bytes per multiplication from L2) are still far below what L2 gives.
  const dim3 small((N + GS_N - 1) / GS_N, (M + GS_M - 1) / GS_M, batch);
  if (kchunk == 0 && !lower_only && (long)grid.x * grid.y * grid.z <= 4 * 152 && small.y <= 65535) {
    auto k = !ta && !tb ? dgemm_small_kernel<false, false>
                        : !ta ? dgemm_small_kernel<false, true> : !tb ? dgemm_small_kernel<true, false> : dgemm_small_kernel<true, true>;
    k<<<small, 128, 0, s>>>(M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC);
    DF_LAUNCHED("dgemm_small_kernel");
    return DF_OK;
  }
  if (!ta && !tb)
    dgemm_kernel<false, false><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, kchunk, lower_only);
  else if (!ta && tb)
    dgemm_kernel<false, true><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, kchunk, lower_only);
  else if (ta && !tb)
    dgemm_kernel<true, false><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, kchunk, lower_only);
  else
    dgemm_kernel<true, true><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, kchunk, lower_only);
  DF_LAUNCHED("dgemm_kernel");
  return DF_OK;
}

// ---- Cholesky ----------------------------------------------------------------------
// Right-looking in blocks of 32: one warp factors the diagonal block in registers, one lane per
// row solves the panel below it and writes its digits, and the trailing update runs on digit
// products.  The chain of 3 launches per block bounds it (n / 32 blocks): small blocks keep
// the serial FP64 part of each link short.
constexpr int CH_NB = 32;

__global__ void chol_init_kernel(const double* __restrict__ A, int n, double* maxdiag, int* status) {
  __shared__ double sh[32];
  double m = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, A[(size_t)i * n + i]);
  // block max via warp shuffles
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t = fmax(t, sh[i]);
    *maxdiag = t;
    *status = -1;
  }
}

// Factor the b x b diagonal block at (k0, k0): lane i holds row i (right-looking).
__global__ void __launch_bounds__(32) chol_diag_kernel(double* __restrict__ A, int n, int k0, int b,
                                                       const double* maxdiag, int* status, double tol) {
  if (*status >= 0) return;
  const int i = threadIdx.x;
  double row[CH_NB];
#pragma unroll
  for (int j = 0; j < CH_NB; ++j) row[j] = (i < b && j <= i) ? A[(size_t)(k0 + i) * n + k0 + j] : 0.0;
  const double thr = tol * *maxdiag;
  int fail = -1;
#pragma unroll
  for (int j = 0; j < CH_NB; ++j) {
    if (j < b && fail < 0) {
      const double piv = __shfl_sync(0xffffffffu, row[j], j);
      if (!(piv > thr)) {
        fail = j;
      } else {
        const double l = sqrt(piv);
        row[j] = i == j ? l : row[j] / l;  // rows above j hold zeros there
#pragma unroll
        for (int c = j + 1; c < CH_NB; ++c) {
          const double lc = __shfl_sync(0xffffffffu, row[j], c);
          if (c <= i) row[c] = fma(-row[j], lc, row[c]);
        }
      }
    }
  }
  if (fail >= 0) {
    if (i == 0) atomicCAS(status, -1, k0 + fail);
    return;
  }
#pragma unroll
  for (int j = 0; j < CH_NB; ++j)
    if (i < b && j < b) A[(size_t)(k0 + i) * n + k0 + j] = row[j];
}

// Panel below the diagonal block: L[i, k0:k0+32] = A[i, k0:k0+32] L_kk^-T, one lane per row, few
// lanes per CTA to spread the FP64 work over the SMs; the row's digits for the trailing update.
__global__ void __launch_bounds__(32) chol_panel_kernel(double* __restrict__ A, int n, int k0, const int* status,
                                                        __nv_bfloat16* __restrict__ out, unsigned* __restrict__ key) {
  __shared__ double Lk[CH_NB][CH_NB];
  __shared__ double rinv[CH_NB];
  if (*status >= 0) return;
  for (int e = threadIdx.x; e < CH_NB * CH_NB; e += blockDim.x)
    Lk[e / CH_NB][e % CH_NB] = A[(size_t)(k0 + e / CH_NB) * n + k0 + e % CH_NB];
  rinv[threadIdx.x] = 1.0 / A[(size_t)(k0 + threadIdx.x) * n + k0 + threadIdx.x];
  __syncthreads();
  const int r = blockIdx.x * blockDim.x + threadIdx.x, rows = n - k0 - CH_NB;
  if (r >= rows) return;
  double* a = A + (size_t)(k0 + CH_NB + r) * n + k0;
  double x[CH_NB];
#pragma unroll
  for (int j = 0; j < CH_NB; ++j) x[j] = a[j];
  unsigned t = 0;
#pragma unroll
  for (int j = 0; j < CH_NB; ++j) {
    double v = x[j];
#pragma unroll
    for (int m = 0; m < j; ++m) v = fma(-Lk[j][m], x[m], v);
    const double q = v * rinv[j];  // pivots are positive and normal: one correction rounds the quotient
    x[j] = fma(fma(-Lk[j][j], q, v), rinv[j], q);
    t = max(t, digits::high_key(x[j]));
  }
#pragma unroll
  for (int j = 0; j < CH_NB; ++j) a[j] = x[j];
  key[r] = t;
  const bool bad = digits::key_bad(t);
  const int f = digits::key_field(t);
#pragma unroll
  for (int j = 0; j < CH_NB; j += 8) {
    double y[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) y[u] = bad ? 0.0 : x[j + u];
    digits::store_digits8(y, f, out + (size_t)r * CH_NB + j, (size_t)rows * CH_NB);
  }
}

__global__ void zero_upper_kernel(double* __restrict__ A, int n) {
  long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long)n * n) return;
  int i = (int)(e / n), j = (int)(e % n);
  if (j > i) A[e] = 0.0;
}

// A wait of the tensor-core updates gave up: no row may pass for a result.
__global__ void poison_kernel(const int* __restrict__ err, double* __restrict__ R, long n) {
  if (*err)
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
      R[i] = __longlong_as_double(0x7ff8000000000000LL);
}

size_t cholesky_bytes(int n) { return 256 + (n > CH_NB ? digit_operand_bytes(n, CH_NB) : 0); }

int cholesky_inplace(double* A, int n, int* d_status, double* d_maxdiag, double tol, void* work, cudaStream_t s) {
  int* err = (int*)work;
  chol_init_kernel<<<1, 1024, 0, s>>>(A, n, d_maxdiag, d_status);
  DF_LAUNCHED("chol_init_kernel");
  for (int k0 = 0; k0 < n; k0 += CH_NB) {
    int b = min(CH_NB, n - k0);
    chol_diag_kernel<<<1, 32, 0, s>>>(A, n, k0, b, d_maxdiag, d_status, tol);
    DF_LAUNCHED("chol_diag_kernel");
    int rest = n - k0 - b;
    if (rest <= 0) break;
    const DigitOperand l = digit_operand((char*)work + 256, rest, CH_NB);
    chol_panel_kernel<<<(rest + 31) / 32, 32, 0, s>>>(A, n, k0, d_status, l.p, l.key);
    DF_LAUNCHED("chol_panel_kernel");
    int k1 = k0 + b;
    const DigitSource src{A + (size_t)k1 * n + k0, n, 1};
    DF_TRY(digit_gemm(l, l, src, src, -1.0, 1.0, A + (size_t)k1 * n + k1, n, 0, 1, DIGIT_LOWER, err, s));
  }
  long nn = (long)n * n;
  zero_upper_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(A, n);
  DF_LAUNCHED("zero_upper_kernel");
  poison_kernel<<<1, 256, 0, s>>>(err, A, n);
  DF_LAUNCHED("poison_kernel");
  return DF_OK;
}

// ---- forward substitution B = L^-1 R ---------------------------------------------------
// Rows k0..k0+NB of R are solved against the diagonal block of L, one lane per column.  FP64-bound
// (NB (NB - 1) / 2 FMAs per column and block), so divisions are a product with the reciprocal and
// one correction step.  With `out`, the digits (digits.cuh) of the solved rows, as row c over the
// NB terms, are written from registers for the update that follows.
template <int NB>
__global__ void __launch_bounds__(128) trsm_diag_kernel(double* __restrict__ R, long ld, long ncol,
                                                        const double* __restrict__ L, int naux, int k0,
                                                        __nv_bfloat16* __restrict__ out, unsigned* __restrict__ key) {
  __shared__ double Lk[NB][NB];
  __shared__ double rinv[NB];
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    int i = e / NB, j = e % NB;
    Lk[i][j] = (j <= i) ? L[(size_t)(k0 + i) * naux + k0 + j] : 0.0;
    if (i == j) rinv[i] = 1.0 / L[(size_t)(k0 + i) * naux + k0 + i];
  }
  __syncthreads();
  long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncol) return;
  double x[NB];
#pragma unroll
  for (int p = 0; p < NB; ++p) x[p] = R[(size_t)(k0 + p) * ld + c];
#pragma unroll
  for (int p = 0; p < NB; ++p) {
    double v = x[p];
#pragma unroll
    for (int q = 0; q < p; ++q) v = fma(-Lk[p][q], x[q], v);
    const double r = rinv[p], q = v * r;
    const double q1 = fma(fma(-Lk[p][p], q, v), r, q);
    x[p] = isfinite(r) && r != 0.0 ? (isfinite(q1) ? q1 : q) : v / Lk[p][p];
  }
  unsigned t = 0;
#pragma unroll
  for (int p = 0; p < NB; ++p) {
    R[(size_t)(k0 + p) * ld + c] = x[p];
    t = max(t, digits::high_key(x[p]));
  }
  if (out) {
    key[c] = t;
    const bool bad = digits::key_bad(t);
    const int f = digits::key_field(t);
#pragma unroll
    for (int p = 0; p < NB; p += 8) {
      double y[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) y[u] = bad ? 0.0 : x[p + u];
      digits::store_digits8(y, f, out + (size_t)c * NB + p, (size_t)ncol * NB);
    }
  }
}

__global__ void trsm_diag_generic_kernel(double* __restrict__ R, long ld, long ncol, const double* __restrict__ L,
                                         int naux, int k0, int b) {
  long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncol) return;
  for (int p = 0; p < b; ++p) {
    double v = R[(size_t)(k0 + p) * ld + c];
    for (int q = 0; q < p; ++q) v -= L[(size_t)(k0 + p) * naux + k0 + q] * R[(size_t)(k0 + q) * ld + c];
    R[(size_t)(k0 + p) * ld + c] = v / L[(size_t)(k0 + p) * naux + k0 + p];
  }
}

// Two levels of blocks.  A block of 32 rows is solved in FP64 (FP64 work grows with the block);
// its digits update the rest of the 128 rows around it; the 128 solved rows together update all
// rows below, so that those are read and written once per 128 rows.  Columns go through in
// chunks, which bounds the digits of X to 120 MB.
constexpr int FS_NB = 32, FS_NBO = 128;
constexpr long FS_COLS = 65536;

size_t forward_substitution_bytes(long ncol, int naux) {
  if (naux <= FS_NB) return 256;  // (also enough for cholesky_bytes(naux), which comes first)
  return digit_operand_bytes(std::min(ncol, FS_COLS), FS_NBO) + digit_operand_bytes(naux, FS_NBO) + 256;
}

int forward_substitution(double* R, long ld, long ncol, const double* L, int naux, void* work, cudaStream_t s) {
  const long cmax = std::min(ncol, FS_COLS);
  char* xmem = (char*)work + 256;
  char* lmem = xmem + digit_operand_bytes(cmax, FS_NBO);
  int* err = (int*)work;
  // R[r0.., :] -= L[r0.., k0..k0+b) R[k0..k0+b, :] over nr rows and the columns of chunk c0 (digits
  // of R's rows k0.. in x)
  auto update = [&](int r0, int nr, int k0, int b, long c0, const DigitOperand& x, const DigitOperand& l) -> int {
    return digit_gemm(x, l, DigitSource{R + (size_t)k0 * ld + c0, 1, ld}, DigitSource{L + (size_t)r0 * naux + k0, naux, 1},
                      -1.0, 1.0, R + (size_t)r0 * ld + c0, ld, 0, 1, DIGIT_TRANSPOSED, err, s);
  };
  for (int j0 = 0; j0 < naux; j0 += FS_NBO) {
    const int nb = std::min(FS_NBO, naux - j0);
    for (int k0 = j0; k0 < j0 + nb; k0 += FS_NB) {
      const int b = std::min(FS_NB, j0 + nb - k0);
      const int rest = j0 + nb - k0 - b;  // rows of this 128-row block still to solve
      DigitOperand l;
      if (rest > 0) {
        l = digit_operand(lmem, rest, b);
        DF_TRY(slice_matrix(L + (size_t)(k0 + b) * naux + k0, naux, false, l, s));
      }
      for (long c0 = 0; c0 < ncol; c0 += FS_COLS) {
        const long nc = std::min(FS_COLS, ncol - c0);
        const unsigned blocks = (unsigned)((nc + 127) / 128);
        const DigitOperand x = digit_operand(xmem, nc, b);
        if (b == FS_NB)
          trsm_diag_kernel<FS_NB><<<blocks, 128, 0, s>>>(R + c0, ld, nc, L, naux, k0, rest > 0 ? x.p : nullptr, x.key);
        else
          trsm_diag_generic_kernel<<<blocks, 128, 0, s>>>(R + c0, ld, nc, L, naux, k0, b);
        DF_LAUNCHED("trsm_diag_kernel");
        if (rest > 0) DF_TRY(update(k0 + b, rest, k0, b, c0, x, l));
      }
    }
    const int r0 = j0 + nb, rest = naux - r0;
    if (rest <= 0) break;
    const DigitOperand l = digit_operand(lmem, rest, nb);
    DF_TRY(slice_matrix(L + (size_t)r0 * naux + j0, naux, false, l, s));
    for (long c0 = 0; c0 < ncol; c0 += FS_COLS) {
      const DigitOperand x = digit_operand(xmem, std::min(FS_COLS, ncol - c0), nb);
      DF_TRY(slice_matrix(R + (size_t)j0 * ld + c0, ld, true, x, s));
      DF_TRY(update(r0, rest, j0, nb, c0, x, l));
    }
  }
  if (naux > FS_NB) {
    poison_kernel<<<64, 256, 0, s>>>(err, R, ncol);
    DF_LAUNCHED("poison_kernel");
  }
  return DF_OK;
}

}  // namespace dfscf

using namespace dfscf;

extern "C" size_t df_metric_chol_work_bytes(int naux) {
  return kWorkAlign + 512 + sizeof(double) * align_up(boys_table_doubles(), 32) + (naux > 0 ? cholesky_bytes(naux) : 0);
}

extern "C" int df_metric_chol(const double* aux_xyz, const double* aux_exp, int naux, double* L, double* M_out,
                              int* bad_pivot, void* work, size_t work_bytes, cudaStream_t s) {
  clear_error();
  DF_REQUIRE(naux > 0 && aux_xyz && aux_exp && L && bad_pivot, DF_ERR_ARG, "df_metric_chol: bad arguments");
  DF_REQUIRE(work && work_bytes >= df_metric_chol_work_bytes(naux), DF_ERR_NOMEM,
             "df_metric_chol: workspace of %zu bytes is smaller than %zu", work_bytes, df_metric_chol_work_bytes(naux));
  *bad_pivot = -1;
  work = aligned_work(work);
  int* d_status = (int*)work;
  double* d_maxdiag = (double*)((char*)work + 256);
  DF_TRY(launch_int2c(aux_xyz, aux_exp, naux, L, (double*)((char*)work + 512), s));
  if (M_out) DF_CUDA(cudaMemcpyAsync(M_out, L, sizeof(double) * naux * naux, cudaMemcpyDeviceToDevice, s));
  void* chol = (char*)work + 512 + sizeof(double) * align_up(boys_table_doubles(), 32);
  DF_TRY(reset_tc_errors((int*)chol, 1, TC_SETUP, s));
  DF_TRY(cholesky_inplace(L, naux, d_status, d_maxdiag, 1e-14, chol, s));
  int h_status = -1;
  DF_CUDA(cudaMemcpyAsync(&h_status, d_status, sizeof(int), cudaMemcpyDeviceToHost, s));
  DF_TRY(check_tc_errors((const int*)chol, 1, "df_metric_chol", s));  // (synchronises) before the pivot, which it may spoil
  if (h_status >= 0) {
    *bad_pivot = h_status;
    set_error("df_metric_chol: metric not positive definite at pivot %d", h_status);
    return DF_ERR_NOT_SPD;
  }
  return DF_OK;
}

DF_BOUNDS_READER(bounds_read_linalg)
