// Internal launchers shared between the library's translation units.
#pragma once
#include <cstddef>
#include <vector>
#include <algorithm>

#include <algorithm>

#include "common.cuh"

namespace dfscf {

// ---- integrals (integrals.cu) ------------------------------------------------------
int launch_int1e(const double* ao_xyz, const double* ao_exp, int nao, const double* nuc_xyz, const double* nuc_z,
                 int natm, double* S, double* T, double* V, cudaStream_t s);
// Per packed orbital pair: exponent p, centre (x, y, z) and factor K_ab = N_a N_b e^{-mu R^2}
// 2 pi^{5/2} / p, as five arrays of npair doubles in pair_tab (pair_tab_doubles(nao) in launch_int3c).
int launch_pair_table(const double* ao_xyz, const double* ao_exp, int nao, double* pair_tab, cudaStream_t s);
// Doubles of a pair table with the Boys table behind it (pair_tab_boys; 16-byte aligned).
size_t boys_table_doubles();
inline size_t pair_tab_boys_offset(int nao) { return align_up(5 * (size_t)npair_of(nao), 2); }
inline size_t pair_tab_doubles(int nao) { return pair_tab_boys_offset(nao) + boys_table_doubles(); }
inline double* pair_tab_boys(double* pair_tab, int nao) { return pair_tab + pair_tab_boys_offset(nao); }
// omega > 0: the long-range operator erf(omega r)/r instead of 1/r (LRDF); table: scratch of
// boys_table_doubles()
int launch_int2c(const double* xyz, const double* ex, int naux, double* M, double* table, cudaStream_t s,
                 double omega = 0.0);
int launch_int3c(const double* ao_xyz, const double* ao_exp, int nao, const double* aux_xyz, const double* aux_exp,
                 int naux, double* R, long ld, double* pair_tab, cudaStream_t s, double omega = 0.0);
int launch_enuc(const double* xyz, const double* z, int natm, double* out, cudaStream_t s);

// ---- FP64 linear algebra (linalg.cu) -----------------------------------------------
int dgemm(bool ta, bool tb, int M, int N, int K, double alpha, const double* A, long lda, long sA, const double* B,
          long ldb, long sB, double beta, double* C, long ldc, long sC, int batch, cudaStream_t s, long kchunk,
          int lower_only);
// work: cholesky_bytes(n), at most forward_substitution_bytes(_, n)
size_t cholesky_bytes(int n);
int cholesky_inplace(double* A, int n, int* d_status, double* d_maxdiag, double tol, void* work, cudaStream_t s);
// work: forward_substitution_bytes(ncol, naux)
size_t forward_substitution_bytes(long ncol, int naux);
int forward_substitution(double* R, long ld, long ncol, const double* L, int naux, void* work, cudaStream_t s);

// Error words of the tensor-core kernels (digit products, split-BF16 GEMMs): a bounded wait that
// gives up raises its word, and every later launch with that word skips its work.  reset before the
// launches of a call; check reads them back (synchronising; not inside a stream capture) and
// returns DF_ERR_TIMEOUT.  cholesky_inplace and forward_substitution use the word at the start of
// work, which their caller resets.
enum TcUser { TC_SETUP = 1, TC_EXCHANGE = 2 };  // values of the test hook "tc_give_up"
int reset_tc_errors(int* err, int n, TcUser user, cudaStream_t s);
int check_tc_errors(const int* err, int n, const char* who, cudaStream_t s);

// ---- eigensolver (eig.cu) ------------------------------------------------------------
size_t eigh_scratch_doubles(int n);
int eigh_rows(double* A, int n, double* w, double* ZT, double* scratch, int* status, cudaStream_t s);
size_t eigh_lowest_scratch_doubles(int n, int k);
size_t eigh_coop_aux_bytes(int n);
size_t eigh_full_scratch_doubles(int n);
// exact: the rounding of the eigensolver's own entry points; false: that of an SCF's iterations
// (tridiag.cu).
int eigh_full_rows(double* A, int n, double* w, double* ZT, double* scratch, int* status, cudaStream_t s, void* aux,
                   bool exact);
// S^p over the eigenvalues of S above lindep, from its eigenvector rows ZT and eigenvalues (lowdin.cu).
int lowdin_power(const double* ZT, const double* s_eig, int n, double lindep, double power, double* scratch,
                 double* out, cudaStream_t s);
int eigh_lowest_rows(double* A, int n, int k, double* w, double* ZT, double* scratch, int* status, cudaStream_t s,
                     void* aux, bool exact);
int transpose(const double* in, int rows, int cols, double* out, cudaStream_t s);

// ---- B layout and J/K (jk.cu, umma.cu) --------------------------------------------------
// Most BF16 planes a mixed-precision B can hold; a B keeps as many as the knob "mixed_planes"
// asked for when it was sized and built (3, 4 or 5).
constexpr int kMixedPlanes = 5;

struct BLayout {
  long ld;       // packed row stride (elements)
  int npad;      // padded orbital dimension of the BF16 planes
  int planes;    // BF16 planes held (0 for DF_FP64)
  size_t off64, offp[kMixedPlanes], bytes;
};

struct MixedKWork {
  void* Cp[kMixedPlanes];  // bf16 [ncpad][npad]  planes of C^T
  void* Xp[kMixedPlanes];  // bf16 [npad][naux * ncpad]  planes of X (row m, column P*ncpad + i)
  float* X32;              // fp32 [2][npad][naux * ncpad]  X from the half transform as a pair
                           //   (order-0 accumulator, higher-order accumulator)
  unsigned* xmax;          // [npad] max |X| of row m (FP32 bits)
  float* Kpart;            // fp32 [nsplit][npad][npad] partial K tiles
  int* err;                // device error flag of the tensor-core kernels
  int ncpad;               // padded occupied count (multiple of 16, >= 16)
  int nsplit;              // K-dimension splits of the exchange contraction
  int planes;              // BF16 planes per operand (3, 4, 5: 6, 10, 15 plane products)
};

// FP64 exchange on digit products (digits.cuh): auxiliary rows go through in blocks of px (X, its
// digits and one SYRK per block) whose half-transforms run pb rows of B at a time.
struct Fp64KWork {
  void* Ct;        // digits of C^T
  void* Bp;        // digits of pb symmetric B_P
  void* Xd;        // digits of X [nao][px * nocc]
  double* X;       // [nao][px * nocc]
  double* Kpart;   // [nsplit][nao][nao]
  int* err;        // a bounded wait gave up
  int pb, px, nsplit;
};

struct JKWork {
  int* err;  // error words of the FP64 and of the mixed exchange (reset_tc_errors before run_jk)
  double* Dw;
  double* d;
  double* Jpart;
  int nsplit_j;
  char* scratch;  // the region of fk, of mk and of the caller's shared scratch
  Fp64KWork fk;
  MixedKWork mk;
};

long B_ld(int nao);
int nao_pad(int nao);
// planes: BF16 planes of a mixed B (ignored for DF_FP64); plane j sits at the same offset
// whatever the count, so a B with more planes serves an exchange that uses fewer.
BLayout B_layout(int nao, int naux, int precision, int planes);
int mixed_planes();
// Host-side record of the plane count each mixed B was built with (keyed by its address),
// checked before an exchange reads the planes; -1 if the address was never recorded.
void record_B_planes(const void* B, int planes);
int recorded_B_planes(const void* B);
JKWork jk_work_layout(int nao, int naux, int nocc, int precision, Arena* a, Sizer* z, bool fp64_k, size_t shared = 0);
int umma_prepare();
void mixed_k_work_layout(int nao, int naux, int nocc, Arena* a, Sizer* z, MixedKWork* w);
int build_K_mixed(const void* B, const BLayout& L, int nao, int naux, const double* C, int nocc, double* K,
                  const MixedKWork& w, cudaStream_t s);
int build_J(const void* Bbuf, const BLayout& L, int nao, int naux, int precision, const double* D, double* J,
            const JKWork& w, cudaStream_t s);
// A workspace sized for more occupied columns serves fewer, though the size of the FP64 exchange's blocks
// does not grow with every column: the number of columns from nocc on whose layout fits in
// work_bytes (at most `most`), -1 if there is none.  bytes(n): the size for n columns.
template <typename Bytes>
int layout_columns(int nocc, int most, size_t work_bytes, Bytes bytes) {
  for (int n = nocc; n <= std::max(nocc, most); ++n)
    if (work_bytes >= bytes(n)) return n;
  return -1;
}
int run_jk(const void* B, int nao, int naux, int precision, const double* D, const double* C, int nocc, double* J,
           double* K, const JKWork& w, cudaStream_t s);
int build_B(const double* ao_xyz, const double* ao_exp, int nao, const double* aux_xyz, const double* aux_exp,
            int naux, const double* Lfac, int precision, void* Bbuf, double* pair_tab, void* subst, cudaStream_t s);

// Bounds-check records of the translation units with kernels (checking build; all zero
// otherwise).
int bounds_read_dferr(BoundsRecord*);
int bounds_read_digits(BoundsRecord*);
int bounds_read_eig(BoundsRecord*);
int bounds_read_integrals(BoundsRecord*);
int bounds_read_jk(BoundsRecord*);
int bounds_read_linalg(BoundsRecord*);
int bounds_read_lowdin(BoundsRecord*);
int bounds_read_lrdf(BoundsRecord*);
int bounds_read_mlp(BoundsRecord*);
int bounds_read_scf(BoundsRecord*);
int bounds_read_tridiag(BoundsRecord*);
int bounds_read_trivec(BoundsRecord*);
int bounds_read_umma(BoundsRecord*);

}  // namespace dfscf
