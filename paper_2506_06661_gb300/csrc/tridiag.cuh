// Interface between the multi-SM tridiagonalisation (tridiag.cu), the eigenpairs of the
// tridiagonal matrix (trivec.cu) and the eigensolver's entry points (eig.cu).
#pragma once
#include "common.cuh"

namespace dfscf {

// Control record of one solve, zeroed on the stream before it starts.
struct EigControl {
  unsigned count;  // arrivals at the grid barrier since launch (monotone)
  unsigned extra;  // arrivals expected beyond the grid's own CTAs: 0, except in the test of
                   // the bounded wait (knob "eig_barrier_extra"), where no wait can complete
  int err;         // 1: a wait gave up; 2: inverse iteration failed
  unsigned limit;  // polls before a wait gives up (knob "eig_barrier_polls")
  int bad;         // the direct eigenvectors of T cannot be used: take inverse iteration
  int pad;
  unsigned long long emax[4];  // bits of max |Z Z^T - 1| before each re-orthonormalisation
};

constexpr int kPanel = 16;  // reflectors applied at once in the back-transformation

struct TridiagPlan {
  int G = 0;  // CTAs (0: the size does not fit)
  int R = 0;  // rows per CTA
  int vps = 2;  // vectors of pending updates in shared memory
  bool exact = true;
  size_t smem = 0;
};

// forced: CTA count asked for by the caller (0: choose).  exact: which rounding (tridiag.cu).
TridiagPlan tridiag_plan(int n, int forced, bool exact);
size_t tridiag_exchange_bytes(int n);  // zeroed by the caller before each launch
// A [n][n] symmetric -> d, e, beta; reflector r in row r of A, columns r + 1 .. n - 1.
int tridiag_launch(double* A, int n, double* d, double* e, double* beta, const TridiagPlan& P, void* exchange,
                   EigControl* ctl, cudaStream_t s);

// The k lowest eigenpairs from the output of tridiag_launch: w [k], ZT [k][n].  Scratch:
// trivec_scratch_doubles(n, k).  exact: the vectors are corrected once.  Leaves ctl->bad or ctl->emax for eig_needs_fallback.
size_t trivec_scratch_doubles(int n, int k);
bool trivec_fits(int n);
int trivec_launch(const double* A, int n, int k, const double* d, const double* e, const double* beta, double* w,
                  double* ZT, double* scratch, bool exact, EigControl* ctl, cudaStream_t s);

// Re-orthonormalisation Z <- Z - (Z Z^T - 1) Z / 2 leaves 3/4 ||Z Z^T - 1||^2.
constexpr double kOrthoDone = 1e-8;
__device__ __forceinline__ bool eig_needs_fallback(const EigControl* c, int k) {
  if (c->bad) return true;
  return !(k * __longlong_as_double((long long)c->emax[0]) <= kOrthoDone ||
           k * __longlong_as_double((long long)c->emax[2]) <= kOrthoDone);
}

}  // namespace dfscf
