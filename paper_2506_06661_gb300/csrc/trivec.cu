// Eigenpairs of a symmetric tridiagonal matrix T, one CTA per eigenvalue, and their
// transformation back to the full matrix.
//
// FP64 issues one warp instruction per 64 clocks and partition, and a division is about ten of them,
// so the recurrences here have none: the leading minors p_i = (d_i - x) p_{i-1} - e_{i-1}^2
// p_{i-2} of T - x (scaled so that ||T|| < 1, and by powers of two when they leave the middle of
// the FP64 range) take a product and two additions a step.  Their sign changes count the
// eigenvalues below x (Givens), and their ratios are the pivots of the factorisations from
// either end, whose meeting point gives the eigenvector directly (the twisted factorisation of
// Fernando, Parlett and Dhillon).
//   1. bisection into 129 parts a round, one thread per point: in FP32 down to about 2^-20, then
//      in FP64 to the last bit; a bracket that FP64 does not confirm starts over in FP64;
//   2. minors from both ends, pivots q+ and q-, the index r with the least |q+_r + q-_r - (d_r - l)|,
//      and z outward from z_r = 1: z_i = -(e_i / q+_i) z_{i+1} and z_{i+1} = -(e_i / q-_{i+1}) z_i;
//      then, where the caller wants exact vectors, one correction of z: its residual in twice the
//      precision, solved with the same factors;
//   3. reflectors in panels of 16: z -= V (T (V^T z));
//   4. Z <- Z - (Z Z^T - 1) Z / 2, three times when the vectors need it.
// Eigenvalues equal to rounding are told apart by the blocks into which T falls, each with the
// eigenvalue of its own block, and inside a block by inverse iteration with projections.  What that
// cannot repair is left to inverse iteration and Gram-Schmidt over the whole matrix, or to implicit
// QL (eig.cu).
// Device time at n = 900, k = 91 against 33-way bisection with a division a step, inverse iteration
// from global memory, one reflector at a time and Gram-Schmidt with five grid barriers a vector:
// eigenvalues 5.2 -> 0.57 ms, eigenvectors 3.1 -> 0.36 (0.23 without the correction),
// back-transformation 2.5 -> 0.71, orthonormalisation 3.0 -> 0.07; at n = 100, k = 11 (one CTA before)
// 936 -> 72 us, 213 -> 52, 112 -> 32, 100 -> 22.
#include <algorithm>
#include <cfloat>

#include "kernels.cuh"
#include "tridiag.cuh"

namespace dfscf {

namespace {
constexpr int NT = 128;

__device__ __forceinline__ double sum4(double v, double* sh) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  return (sh[0] + sh[1]) + (sh[2] + sh[3]);
}

__device__ __forceinline__ double max4(double v, double* sh) {
  for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  return fmax(fmax(sh[0], sh[1]), fmax(sh[2], sh[3]));
}

__device__ __forceinline__ int exponent_of(double a) { return (__double2hiint(a) >> 20) & 0x7ff; }

// a 2^k, k a small integer; what leaves the FP64 range becomes zero.
__device__ __forceinline__ double shifted(double a, int k) {
  const int ex = exponent_of(a) + k;
  return ex <= 0 ? 0.0 : __hiloint2double(__double2hiint(a) + (k << 20), __double2loint(a));
}

// Exponent shift that brings the larger of two minors back to the middle of the range (0: fine).
// Eight steps grow a minor by at most 3^8 and shrink the larger of a pair by at most 2^-520.
__device__ __forceinline__ int rescale(double a, double b) {
  const int ex = max(exponent_of(a), exponent_of(b));
  return (ex < 1023 - 300 || ex > 1023 + 300) ? 1023 - ex : 0;
}

struct __align__(16) Row {
  double d, e2;  // diagonal and squared subdiagonal below it, scaled
};

// Eigenvalues of T below x.
__device__ int count_below(const Row* __restrict__ T, int n, double x) {
  double p0 = 1.0, p1 = T[0].d - x;
  int c = (unsigned)__double2hiint(p1) >> 31;
  double e2 = T[0].e2;
  int i = 1;
  for (; i + 8 <= n; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const Row t = T[i + u];
      const double p = fma(t.d - x, p1, -(e2 * p0));
      c += (unsigned)(__double2hiint(p) ^ __double2hiint(p1)) >> 31;
      p0 = p1;
      p1 = p;
      e2 = t.e2;
    }
    const int k = rescale(p0, p1);
    if (k) {
      p0 = shifted(p0, k);
      p1 = shifted(p1, k);
    }
  }
  for (; i < n; ++i) {
    const Row t = T[i];
    const double p = fma(t.d - x, p1, -(e2 * p0));
    c += (unsigned)(__double2hiint(p) ^ __double2hiint(p1)) >> 31;
    p0 = p1;
    p1 = p;
    e2 = t.e2;
  }
  return c;
}

__device__ int count_below_f(const float2* __restrict__ T, int n, float x) {
  float p0 = 1.0f, p1 = T[0].x - x, e2 = T[0].y;
  int c = (unsigned)__float_as_int(p1) >> 31;
  int i = 1;
  for (; i + 4 <= n; i += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float2 t = T[i + u];
      const float p = fmaf(t.x - x, p1, -(e2 * p0));
      c += (unsigned)(__float_as_int(p) ^ __float_as_int(p1)) >> 31;
      p0 = p1;
      p1 = p;
      e2 = t.y;
    }
    const int ex = max((__float_as_int(p0) >> 23) & 0xff, (__float_as_int(p1) >> 23) & 0xff);
    if (ex < 127 - 30 || ex > 127 + 30) {
      const float f = __int_as_float(min(254, max(1, 254 - ex)) << 23);
      p0 *= f;
      p1 *= f;
    }
  }
  for (; i < n; ++i) {
    const float2 t = T[i];
    const float p = fmaf(t.x - x, p1, -(e2 * p0));
    c += (unsigned)(__float_as_int(p) ^ __float_as_int(p1)) >> 31;
    p0 = p1;
    p1 = p;
    e2 = t.y;
  }
  return c;
}

// First thread of the CTA (in order) whose predicate holds, NT if none.
__device__ __forceinline__ int first_thread(bool p, unsigned* sh) {
  const unsigned m = __ballot_sync(0xffffffffu, p);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  for (int w = 0; w < NT / 32; ++w)
    if (sh[w]) return 32 * w + __ffs(sh[w]) - 1;
  return NT;
}

// Minors of T - l from one end (dir +1: leading, -1: trailing), by one warp; p[i] is stored before
// its block's rescaling, sc[block] is that rescaling's exponent.
__device__ void minors(const Row* __restrict__ T, int n, double l, int dir, double* __restrict__ p, int* __restrict__ sc) {
  const bool lead = (threadIdx.x & 31) == 0;
  int at = dir > 0 ? 0 : n - 1;
  double p0 = 1.0, p1 = T[at].d - l, e2 = 0.0;
  if (p1 == 0.0) p1 = 0x1p-60;
  if (lead) p[at] = p1;
  for (int i0 = 1; i0 < n; i0 += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (i0 + u < n) {
        at += dir;
        e2 = dir > 0 ? T[at - 1].e2 : T[at].e2;
        double q = fma(T[at].d - l, p1, -(e2 * p0));
        if (q == 0.0) q = p1 * 0x1p-60;  // a diagonal entry moved by 2^-60 ||T||
        p0 = p1;
        p1 = q;
        if (lead) p[at] = q;
      }
    }
    const int k = rescale(p0, p1);
    if (k) {
      p0 = shifted(p0, k);
      p1 = shifted(p1, k);
    }
    if (lead) sc[(i0 - 1) / 8] = k;
  }
}

// Block-reflector factor of panel b: T upper triangular, H_r0 .. H_r0+15 = 1 - V T V^T
// (columns of V: the reflectors; T_jj = beta_j, T_0:j,j = -beta_j T_0:j,0:j V_0:j^T v_j).
__device__ void panel_factor(const double* __restrict__ A, int n, int b, const double* __restrict__ beta,
                             double* __restrict__ Tout, double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r0 = b * kPanel, nr = min(kPanel, n - 2 - r0);
  double* Gm = sh;  // [16][16], Gm[i][j] = v_i . v_j for i < j
  double* Tm = sh + kPanel * kPanel;
  for (int q = threadIdx.x; q < kPanel * kPanel; q += NT) Tm[q] = 0.0;
  for (int q = wid; q < nr * (nr - 1) / 2; q += NT / 32) {
    int j = 1;
    while (j * (j + 1) / 2 <= q) ++j;
    const int i = q - j * (j - 1) / 2;
    const double *vi = A + (size_t)(r0 + i) * n, *vj = A + (size_t)(r0 + j) * n;
    double s = 0.0;
#pragma unroll 4
    for (int c = r0 + j + 1 + lane; c < n; c += 32) s = fma(vi[c], vj[c], s);
    s = warp_sum(s);
    if (lane == 0) Gm[i * kPanel + j] = s;
  }
  __syncthreads();
  if (wid == 0) {
    for (int j = 0; j < nr; ++j) {
      const double bj = beta[r0 + j];
      double s = 0.0;
      if (lane < j)
        for (int l = lane; l < j; ++l) s = fma(Tm[lane * kPanel + l], Gm[l * kPanel + j], s);
      __syncwarp();
      if (lane < j) Tm[lane * kPanel + j] = -bj * s;
      if (lane == j) Tm[j * kPanel + j] = bj;
      __syncwarp();
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < kPanel * kPanel; q += NT) Tout[(size_t)b * kPanel * kPanel + q] = Tm[q];
}

// Gershgorin interval of T and its exponent; false when T is zero, not finite or extreme.
__device__ __forceinline__ bool interval(const double* __restrict__ d, const double* __restrict__ e, int n, double* sh,
                                         double& lo, double& hi, int& ex) {
  lo = INFINITY;
  hi = -INFINITY;
  for (int i = threadIdx.x; i < n; i += NT) {
    const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0);
    lo = fmin(lo, d[i] - r);
    hi = fmax(hi, d[i] + r);
  }
  lo = -max4(-lo, sh);
  hi = max4(hi, sh);
  ex = exponent_of(fmax(fabs(lo), fabs(hi)));
  return ex >= 200 && ex <= 1800;
}

__device__ __forceinline__ Row scaled_row(const double* d, const double* e, int n, int i, double scale) {
  const double ei = i + 1 < n ? e[i] * scale : 0.0;
  return Row{d[i] * scale, fmax(ei * ei, 0x1p-130)};  // below 2^-65 ||T|| an entry is nothing
}

// Bisection of [lo, hi] for eigenvalue t down to its last bit.
__device__ __forceinline__ double bisect(const Row* T, int n, int t, double lo, double hi, unsigned* shm) {
  for (int round = 0; round < 64; ++round) {
    if (hi - lo <= fmax(2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)), 0x1p-58)) break;
    const double h = (hi - lo) * (1.0 / (NT + 1));
    const double x = fmin(lo + (threadIdx.x + 1) * h, hi);
    const int j = first_thread(count_below(T, n, x) > t, shm);
    const double old = lo;
    if (j > 0) lo = fmin(old + j * h, hi);
    if (j < NT) hi = fmin(old + (j + 1) * h, hi);
  }
  return 0.5 * (lo + hi);
}

size_t values_smem(int n) { return std::max((sizeof(Row) + sizeof(float2)) * (size_t)n, 2 * kPanel * kPanel * sizeof(double)); }

// CTA t < k: eigenvalue t of T.  CTA k + b: factor of reflector panel b.
__global__ void __launch_bounds__(NT) tri_values_kernel(const double* __restrict__ A, int n, int k,
                                                        const double* __restrict__ d, const double* __restrict__ e,
                                                        const double* __restrict__ beta, double* __restrict__ w,
                                                        double* __restrict__ Tf, EigControl* ctl) {
  extern __shared__ double smem_d[];
  __shared__ double sh[4];
  __shared__ unsigned shm[4];
  if (ctl->err) return;  // the reduction gave up
  if ((int)blockIdx.x >= k) {
    panel_factor(A, n, (int)blockIdx.x - k, beta, Tf, smem_d);
    return;
  }
  const int tid = threadIdx.x, t = (int)blockIdx.x;
  Row* T = (Row*)smem_d;
  float2* Tf32 = (float2*)(T + n);
  double lo, hi;
  int ex;
  if (!interval(d, e, n, sh, lo, hi, ex)) {  // not for this path
    if (tid == 0) ctl->bad = 1;
    return;
  }
  // scaled by a power of two so that ||T|| < 1
  const double scale = __hiloint2double((2045 - ex) << 20, 0), unscale = __hiloint2double((ex + 1) << 20, 0);
  for (int i = tid; i < n; i += NT) {
    const Row r = scaled_row(d, e, n, i, scale);
    T[i] = r;
    Tf32[i] = make_float2((float)r.d, (float)r.e2);
  }
  lo = lo * scale - 0x1p-50;
  hi = hi * scale + 0x1p-50;
  const double lo0 = lo, hi0 = hi;
  __syncthreads();
  for (int round = 0; round < 4 && hi - lo > 0x1p-20; ++round) {
    const double h = (hi - lo) * (1.0 / (NT + 1));
    const int j = first_thread(count_below_f(Tf32, n, (float)(lo + (tid + 1) * h)) > t, shm);
    hi = j < NT ? lo + (j + 1) * h : hi;
    lo = lo + j * h;
  }
  {
    // 128 points across the widened bracket, both ends among them
    const double a = fmax(lo0, lo - 0x1p-19), b = fmin(hi0, hi + 0x1p-19), h = (b - a) * (1.0 / (NT - 1));
    const double x = tid == NT - 1 ? b : a + tid * h;
    const int j = first_thread(count_below(T, n, x) > t, shm);
    if (j == 0 || j == NT) {  // FP32 went wrong
      lo = lo0;
      hi = hi0;
    } else {
      lo = a + (j - 1) * h;
      hi = j == NT - 1 ? b : a + j * h;
    }
  }
  const double l = bisect(T, n, t, lo, hi, shm);
  if (tid == 0) w[t] = l * unscale;
}

constexpr int kMembers = 4096;  // members of a cluster in one block times its rows, at most

// Dynamic shared memory of tri_vectors_kernel: Row [n], five arrays [n], the members of a cluster and
// the rescalings.
size_t vectors_smem(int n) {
  return (sizeof(Row) + 5 * sizeof(double)) * (size_t)n + kMembers * sizeof(double) + 2 * sizeof(int) * (size_t)(n / 8 + 1);
}

constexpr double kCluster = 0x1p-44;  // of ||T||: closer eigenvalues than that are one cluster
// Inside a cluster a subdiagonal entry up to 2^-52 sqrt(n) ||T|| separates blocks: twice what rounding
// makes of a zero in the reduction, and what dropping it adds to a residual.  Where that leaves a block
// with more members than inverse iteration has room for, entries up to 2^-46 ||T|| separate (a
// projector of 900 rows: 117 ms by Gram-Schmidt over the grid, with residuals of 6e-14).
__device__ __forceinline__ double split2_of(int n, int attempt) { return attempt ? 0x1p-92 : n * 0x1p-104; }

// Counts of eigenvalues below x block by block of T (ends of blocks: squared subdiagonal <= split2):
// out[i] for the last row i of each block, -1 elsewhere.  One thread.
__device__ void block_counts(const Row* __restrict__ T, int n, double x, double split2, int* __restrict__ out) {
  double p0 = 1.0, p1 = 1.0, e2 = 0.0;
  int c = 0;
  for (int i = 0; i < n; ++i) {
    const double p = fma(T[i].d - x, p1, -(e2 * p0));
    c += (unsigned)(__double2hiint(p) ^ __double2hiint(p1)) >> 31;
    e2 = T[i].e2;
    if (i == n - 1 || e2 <= split2) {
      out[i] = c;
      c = 0;
      p0 = p1 = 1.0;
      e2 = 0.0;
    } else {
      out[i] = -1;
      p0 = p1;
      p1 = p;
      const int k = rescale(p0, p1);
      if (k) {
        p0 = shifted(p0, k);
        p1 = shifted(p1, k);
      }
    }
  }
}

// Eigenvalues base .. base + j of the block T (nb rows) lie in one cluster: their vectors by inverse
// iteration, each made orthogonal to the ones before it after every solve, so that the next solve
// works in their complement (LAPACK's dstein).  Member q goes to members + q nb.  f: 5 arrays of
// stride fs for the factors of T - l = P L U with partial pivoting (multiplier and interchange, 1/U
// and its two superdiagonals) and the vector.
__device__ bool cluster_member(const Row* __restrict__ T, const double* __restrict__ e, double scale, int nb, int base,
                               int j, double lo, double hi, double* f, int fs, double* members, double* sh,
                               unsigned* shm) {
  double *L = f, *ru0 = f + fs, *u1 = f + 2 * (size_t)fs, *u2 = f + 3 * (size_t)fs, *x = f + 4 * (size_t)fs;
  const int tid = threadIdx.x;
  double last = 0.0;
  for (int q = 0; q <= j; ++q) {
    double l = bisect(T, nb, base + q, lo, hi, shm);
    if (q > 0 && l < last + 0x1p-50) l = last + 0x1p-50;  // distinct shifts
    last = l;
    __syncthreads();
    for (int i = tid; i < nb; i += NT) {
      unsigned h = (unsigned)i * 0x9E3779B1u ^ ((unsigned)q + 0x7F4A7C15u) * 0x85EBCA77u;
      h ^= h >> 15;
      h *= 0x2C1B3C6Du;
      h ^= h >> 12;
      x[i] = 1.0 + (double)(h >> 8) * (0.5 / 16777216.0);
    }
    if (tid == 0) {  // an interchange is marked by the multiplier's lowest bit
      double di = T[0].d - l, ui = nb > 1 ? e[0] * scale : 0.0;
      for (int i = 0; i < nb; ++i) {
        const bool end = i + 1 == nb;
        const double li = end ? 0.0 : e[i] * scale, dn = end ? 0.0 : T[i + 1].d - l, un = i + 2 < nb ? e[i + 1] * scale : 0.0;
        double piv, m;
        bool swap = false;
        if (fabs(di) >= fabs(li)) {
          m = di != 0.0 ? li / di : 0.0;
          piv = di;
          u1[i] = ui;
          u2[i] = 0.0;
          di = dn - m * ui;
          ui = un;
        } else {
          swap = true;
          m = di / li;
          piv = li;
          u1[i] = dn;
          u2[i] = un;
          di = ui - m * dn;
          ui = -m * un;
        }
        if (fabs(piv) < 0x1p-53) piv = copysign(0x1p-53, piv);
        ru0[i] = 1.0 / piv;
        L[i] = __longlong_as_double((__double_as_longlong(m) & ~1ll) | (swap ? 1ll : 0ll));
      }
    }
    for (int it = 0; it < 4; ++it) {
      __syncthreads();
      if (tid == 0) {
        double xi = x[0];
        for (int i = 0; i + 1 < nb; ++i) {
          const double m = L[i], xn = x[i + 1];
          const bool swap = __double_as_longlong(m) & 1ll;
          x[i] = swap ? xn : xi;
          xi = swap ? fma(-m, xn, xi) : fma(-m, xi, xn);
        }
        x[nb - 1] = xi;
        double x1 = 0.0, x2 = 0.0;
        for (int i = nb - 1; i >= 0; --i) {
          const double v = fma(-u2[i], x2, fma(-u1[i], x1, x[i])) * ru0[i];
          x[i] = v;
          x2 = x1;
          x1 = v;
        }
      }
      __syncthreads();
      // scaled to norm 1 before the projections, and after them
      for (int part = 0; part < 2; ++part) {
        double n2 = 0.0;
        for (int i = tid; i < nb; i += NT) n2 = fma(x[i], x[i], n2);
        n2 = sum4(n2, sh);
        if (!(n2 > 1e-280 && n2 < 1e300)) return false;
        const double inv = 1.0 / sqrt(n2);
        for (int i = tid; i < nb; i += NT) x[i] *= inv;
        if (part == 0)
          for (int r = 0; r < 2 * q; ++r) {  // all of them twice
            const double* y = members + (size_t)(r % q) * nb;
            double s = 0.0;
            for (int i = tid; i < nb; i += NT) s = fma(x[i], y[i], s);
            s = sum4(s, sh);
            for (int i = tid; i < nb; i += NT) x[i] = fma(-s, y[i], x[i]);
          }
      }
    }
    for (int i = tid; i < nb; i += NT) members[(size_t)q * nb + i] = x[i];
    __syncthreads();
  }
  return true;
}

// Integer with the order of the doubles (FP64 comparisons take 64 clocks a warp; no NaN, no -0 here).
__device__ __forceinline__ long long sortable(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// Bisection of [lo, hi] for eigenvalue t by one thread.
__device__ double bisect_thread(const Row* __restrict__ T, int n, int t, double lo, double hi) {
  if (n == 1) return T[0].d;
  for (int it = 0; it < 64; ++it) {
    if (hi - lo <= fmax(2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)), 0x1p-58)) break;
    const double x = 0.5 * (lo + hi);
    if (count_below(T, n, x) > t) hi = x;
    else lo = x;
  }
  return 0.5 * (lo + hi);
}

// Row i of (T - l) z to about twice the working precision.
__device__ __forceinline__ double residual_row(const Row* __restrict__ T, const double* __restrict__ e, double scale,
                                               int n, double l, const double* __restrict__ z, int i) {
  const double d = T[i].d, a = d - l, bb = a - d, al = (d - (a - bb)) + (-l - bb);  // a + al = d - l (Knuth)
  const double zi = z[i], em = i > 0 ? e[i - 1] * scale : 0.0, zm = i > 0 ? z[i - 1] : 0.0;
  const double ep = i + 1 < n ? e[i] * scale : 0.0, zp = i + 1 < n ? z[i + 1] : 0.0;
  const double h1 = a * zi, h2 = em * zm, h3 = ep * zp;
  const double l1 = fma(al, zi, fma(a, zi, -h1)), l2 = fma(em, zm, -h2), l3 = fma(ep, zp, -h3);
  const double s1 = h1 + h2, t1 = s1 - h1, r1 = (h1 - (s1 - t1)) + (h2 - t1);
  const double s2 = s1 + h3, t2 = s2 - s1, r2 = (s1 - (s2 - t2)) + (h3 - t2);
  return s2 + (((l1 + l2) + (l3 + r1)) + r2);
}

// s[at] += f[at + df] s[at - dir] along `count` entries from `at`, the first as it is; one thread,
// operands loaded eight ahead of the chain.
__device__ __forceinline__ void chain(double* __restrict__ s, const double* __restrict__ f, int at, int count, int dir,
                                      int df) {
  if (count < 2) return;
  double v = s[at];
  for (int q = 1; q < count; q += 8) {
    double c[8], x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = at + dir * min(q + u, count - 1);
      c[u] = f[i + df];
      x[u] = s[i];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (q + u < count) s[at + dir * (q + u)] = v = fma(c[u], v, x[u]);
  }
}

// CTA t: eigenvector t of T into row t of Y, and its eigenvalue into wv[t].  Eigenvalues closer than
// rounding come from different blocks of a T that falls apart (equal eigenvalues of A make it do
// so).  Every CTA of such a cluster forms the blocks' own eigenvalues there, the same bits in each,
// and takes the one of its rank: 25 halvings a member, one thread each (10 us for blocks of one row),
// or 3 rounds on the whole CTA for a few members of what may be large blocks.
__global__ void __launch_bounds__(NT) tri_vectors_kernel(int n, int k, const double* __restrict__ d,
                                                         const double* __restrict__ e, const double* __restrict__ w,
                                                         double* __restrict__ Y, double* __restrict__ wv,
                                                         bool exact, EigControl* ctl) {
  extern __shared__ double smem_d[];
  __shared__ double sh[4];
  __shared__ unsigned shm[4];
  __shared__ unsigned long long best;
  __shared__ int pick[5], leave, found;
  __shared__ double own;
  const int tid = threadIdx.x, t = (int)blockIdx.x;
  // Other CTAs of this grid may raise ctl->bad at any time: one thread reads it for all, or part of
  // the CTA would leave and the rest work on shared memory that was never written.
  if (tid == 0) leave = ctl->err | *(volatile int*)&ctl->bad;
  __syncthreads();
  if (leave) return;
  Row* T = (Row*)smem_d;
  double* p = smem_d + 2 * (size_t)n;
  double* s = p + n;
  double* fa = s + n;
  double* fb = fa + n;
  double* members = fb + 2 * (size_t)n;  // after the fifth array of cluster_member
  int* scp = (int*)(members + kMembers);
  int* scs = scp + n / 8 + 1;
  double lo, hi;
  int ex;
  if (!interval(d, e, n, sh, lo, hi, ex)) {
    if (tid == 0) ctl->bad = 1;
    return;
  }
  const double scale = __hiloint2double((2045 - ex) << 20, 0), unscale = __hiloint2double((ex + 1) << 20, 0);
  for (int i = tid; i < n; i += NT) T[i] = scaled_row(d, e, n, i, scale);
  if (tid == 0) best = ~0ull;
  double l = w[t] * scale;
  int i0 = 0, nb = n;  // the vector's block
  int ta = t, tb = t;
  while (ta > 0 && (w[ta] - w[ta - 1]) * scale <= kCluster) --ta;
  while (tb + 1 < k && (w[tb + 1] - w[tb]) * scale <= kCluster) ++tb;
  __syncthreads();
  if (ta < tb) {
    lo = w[ta] * scale - 0.5 * kCluster;
    hi = w[tb] * scale + 0.5 * kCluster;
    // the cluster's members in block order: last row of the block, number in it (arrays of n ints)
    int *cl = (int*)fa, *ch = (int*)fb, *first = cl + n, *last = (int*)s, *number = last + n;
    for (int attempt = 0; attempt < 2; ++attempt) {
      if (tid == 0) block_counts(T, n, lo, split2_of(n, attempt), cl);
      if (tid == 32) block_counts(T, n, hi, split2_of(n, attempt), ch);
      __syncthreads();
      if (tid == 0) {
        int count = 0, start = 0;
        bool large = false;
        for (int i = 0; i < n; ++i)
          if (cl[i] >= 0) {
            const int m = ch[i] - cl[i];
            large |= m > 1 && m * (i + 1 - start) > kMembers;
            for (int q = cl[i]; q < ch[i] && count < n; ++q) {
              last[count] = i;
              number[count++] = q;
            }
            first[i] = start;
            start = i + 1;
          }
        found = large ? 0 : count;
        pick[3] = 0;
      }
      __syncthreads();
      if (found) break;
    }
    double* value = p;
    const int members_in = found;
    if (members_in > 8) {
      for (int q = tid; q < members_in; q += NT) {
        const int i = first[last[q]];
        value[q] = bisect_thread(T + i, last[q] + 1 - i, number[q], lo, hi);
      }
    } else {
      for (int q = 0; q < members_in; ++q) {
        const int i = first[last[q]];
        const double v = bisect(T + i, last[q] + 1 - i, number[q], lo, hi, shm);
        if (tid == 0) value[q] = v;
      }
    }
    __syncthreads();
    for (int q = tid; q < members_in; q += NT) {
      const double v = value[q];
      const long long kv = sortable(v);
      int rank = 0;
      for (int r = 0; r < members_in; ++r) {
        const long long kr = sortable(value[r]);
        rank += kr < kv || (kr == kv && r < q);
      }
      if (rank == t - ta) {
        const int i = last[q];
        pick[0] = first[i];
        pick[1] = i + 1 - first[i];
        pick[2] = cl[i];
        pick[3] = ch[i] - cl[i];
        pick[4] = number[q] - cl[i];
        own = v;
      }
    }
    __syncthreads();
    const int m = pick[3];
    if (m == 0) {
      if (tid == 0) ctl->bad = 1;
      return;
    }
    i0 = pick[0];
    nb = pick[1];
    l = own;
    if (tid == 0) wv[t] = l * unscale;
    __syncthreads();  // before the arrays that the values came from are used again
    if (m > 1) {
      const bool ok = cluster_member(T + i0, e + i0, scale, nb, pick[2], pick[4], lo, hi, p, n, members, sh, shm);
      if (!ok) {
        if (tid == 0) ctl->bad = 1;
        return;
      }
      const double* z = members + (size_t)pick[4] * nb;
      for (int i = tid; i < n; i += NT) Y[(size_t)t * n + i] = i >= i0 && i < i0 + nb ? z[i - i0] : 0.0;
      return;
    }
  } else if (tid == 0) {
    wv[t] = w[t];
  }
  const Row* Tb = T + i0;
  double *qa = fb + n, *qz = members;  // pivots (n is below kMembers: vectors_smem)
  if (tid < 32) minors(Tb, nb, l, 1, p, scp);
  else if (tid < 64) minors(Tb, nb, l, -1, s, scs);
  __syncthreads();
  unsigned long long mine = ~0ull;
  int at = 0;
  for (int i = tid; i < nb; i += NT) {
    // the neighbour's minor as the recurrence used it, after its block's rescaling
    const double before = i > 0 ? (((i - 1) & 7) == 0 && i > 1 ? shifted(p[i - 1], scp[(i - 2) / 8]) : p[i - 1]) : 1.0;
    const int m = nb - 1 - i;  // position in the backward recurrence
    const double after = m > 0 ? (((m - 1) & 7) == 0 && m > 1 ? shifted(s[i + 1], scs[(m - 2) / 8]) : s[i + 1]) : 1.0;
    const double qf = p[i] / before, qb = s[i] / after;
    qa[i] = qf;
    qz[i] = qb;
    const double gamma = (qf + qb) - (Tb[i].d - l);
    const unsigned long long key = (unsigned long long)__double_as_longlong(fabs(gamma));
    if (key < mine) {
      mine = key;
      at = i;
    }
    fa[i] = i + 1 < nb ? -(e[i0 + i] * scale) / qf : 0.0;
    fb[i] = i > 0 ? -(e[i0 + i - 1] * scale) / qb : 0.0;
  }
  atomicMin(&best, mine);
  if (tid == 0) shm[0] = 0x7fffffffu;
  __syncthreads();
  if (mine == best && best != ~0ull) atomicMin(&shm[0], (unsigned)at);
  __syncthreads();
  const int r = (int)min(shm[0], (unsigned)(nb - 1));
  // outward from r, the factors loaded eight ahead of the chain of products
  if (tid == 0) {
    double z = 1.0;
    p[r] = 1.0;
    for (int i = r - 1; i >= 0; i -= 8) {
      double f[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) f[u] = fa[max(i - u, 0)];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i - u >= 0) p[i - u] = z *= f[u];
    }
  } else if (tid == 32) {
    double z = 1.0;
    for (int i = r + 1; i < nb; i += 8) {
      double f[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) f[u] = fb[min(i + u, nb - 1)];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i + u < nb) p[i + u] = z *= f[u];
    }
  } else if (tid >= 64) {
    for (int i = tid - 64; i < nb; i += NT - 64) qa[i] = 1.0 / (i < r ? qa[i] : qz[i]);
  }
  __syncthreads();
  double n2 = 0.0;
  for (int i = tid; i < nb; i += NT) n2 = fma(p[i], p[i], n2);
  n2 = sum4(n2, sh);
  if (!(n2 >= 0.5 && n2 < 1e300)) {
    if (tid == 0) ctl->bad = 1;
    return;
  }
  const double inv = 1.0 / sqrt(n2);
  for (int i = tid; i < nb; i += NT) p[i] *= inv;
  __syncthreads();
  if (!exact) {
    for (int i = tid; i < n; i += NT) Y[(size_t)t * n + i] = i >= i0 && i < i0 + nb ? p[i - i0] : 0.0;
    return;
  }
  // ---- correction: (T - l) y = (T - l) z - delta z without row r, y_r = 0, delta = z.(T - l) z ----------
  // z's components along its neighbours, 1.4e-14 for the 90 lowest of 900 rows where inverse iteration
  // left 4e-15, become negligible (the residual of a rounded z).
  double c = 0.0;
  for (int i = tid; i < nb; i += NT) {
    const double b = residual_row(Tb, e + i0, scale, nb, l, p, i);
    s[i] = b;
    c = fma(p[i], b, c);
  }
  c = sum4(c, sh);
  for (int i = tid; i < nb; i += NT) s[i] = i == r ? 0.0 : fma(-c, p[i], s[i]);
  __syncthreads();
  if (tid == 0) {
    chain(s, fa, 0, r, 1, -1);
  } else if (tid == 32) {
    chain(s, fb, nb - 1, nb - 1 - r, -1, 1);
  }
  __syncthreads();
  for (int i = tid; i < nb; i += NT) s[i] *= qa[i];  // s_r = 0
  __syncthreads();
  if (tid == 0) {
    chain(s, fa, r, r + 1, -1, 0);
  } else if (tid == 32) {
    chain(s, fb, r, nb - r, 1, 0);
  }
  __syncthreads();
  double y2 = 0.0, m2 = 0.0;
  for (int i = tid; i < nb; i += NT) {
    const double y = s[i], v = p[i] - y;
    y2 = fma(y, y, y2);
    m2 = fma(v, v, m2);
  }
  y2 = sum4(y2, sh);
  m2 = sum4(m2, sh);
  const bool take = y2 <= 1e-4;  // else the factors are too poor for it
  const double norm = take ? 1.0 / sqrt(m2) : 1.0;
  for (int i = tid; i < n; i += NT)
    Y[(size_t)t * n + i] = i >= i0 && i < i0 + nb ? (take ? p[i - i0] - s[i - i0] : p[i - i0]) * norm : 0.0;
}

// z <- H_0 .. H_{n-3} z for row blockIdx.x of Y, into Z; its eigenvalue from wv into w.  Dynamic shared
// memory: z [n].
__global__ void __launch_bounds__(NT) back_transform_kernel(const double* __restrict__ A, int n,
                                                            const double* __restrict__ Tf, const double* __restrict__ Y,
                                                            const double* __restrict__ wv, double* __restrict__ w,
                                                            double* __restrict__ Z, const EigControl* ctl) {
  extern __shared__ double z[];
  __shared__ double red[NT / 32][kPanel], cs[kPanel];
  if (ctl->err | ctl->bad) return;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const size_t row = (size_t)blockIdx.x * n;
  if (tid == 0) w[blockIdx.x] = wv[blockIdx.x];
  for (int i = tid; i < n; i += NT) z[i] = Y[row + i];
  __syncthreads();
  for (int b = (n - 2 + kPanel - 1) / kPanel - 1; b >= 0; --b) {
    const int r0 = b * kPanel, nr = min(kPanel, n - 2 - r0);
    const double* V = A + (size_t)r0 * n;
    const int j16 = lane & 15, h8 = (lane >> 4) * 8;
    double trow[8];  // half a row of the panel's factor, for the first warp
    if (wid == 0)
#pragma unroll
      for (int i = 0; i < 8; ++i) trow[i] = Tf[(size_t)b * kPanel * kPanel + j16 * kPanel + h8 + i];
    double acc[kPanel];
#pragma unroll
    for (int j = 0; j < kPanel; ++j) acc[j] = 0.0;
    for (int c = r0 + 1 + tid; c < n; c += NT) {
      double v[kPanel];
#pragma unroll
      for (int j = 0; j < kPanel; ++j) v[j] = j < nr ? V[(size_t)j * n + c] : 0.0;
      const double zc = z[c];
#pragma unroll
      for (int j = 0; j < kPanel; ++j) acc[j] = fma(c > r0 + j ? v[j] : 0.0, zc, acc[j]);
    }
    // sums over the lanes, 16 at a time: 16 additions instead of 80
#pragma unroll
    for (int h = kPanel / 2, o = 16; h >= 1; h /= 2, o /= 2) {
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const double send = up ? acc[i] : acc[i + h], keep = up ? acc[i + h] : acc[i];
        acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if ((lane & 1) == 0) red[wid][lane >> 1] = acc[0];
    __syncthreads();
    if (wid == 0) {
      const double dj = (red[0][j16] + red[1][j16]) + (red[2][j16] + red[3][j16]);
      double c = 0.0;
#pragma unroll
      for (int i = 0; i < 8; ++i) c = fma(trow[i], __shfl_sync(0xffffffffu, dj, h8 + i), c);
      c += __shfl_xor_sync(0xffffffffu, c, 16);
      if (lane < kPanel) cs[lane] = c;
    }
    __syncthreads();
    for (int c = r0 + 1 + tid; c < n; c += NT) {
      double v[kPanel];
#pragma unroll
      for (int j = 0; j < kPanel; ++j) v[j] = j < nr ? V[(size_t)j * n + c] : 0.0;
      double z0 = z[c], z1 = 0.0;
#pragma unroll
      for (int j = 0; j < kPanel; j += 2) {
        z0 = fma(-(c > r0 + j ? v[j] : 0.0), cs[j], z0);
        z1 = fma(-(c > r0 + j + 1 ? v[j + 1] : 0.0), cs[j + 1], z1);
      }
      z[c] = z0 + z1;
    }
    __syncthreads();
  }
  for (int i = tid; i < n; i += NT) Z[row + i] = z[i];
}

// The later passes have nothing to do when the first met vectors that one correction settles; else
// all three run, which also leaves the result where the first would.
__device__ __forceinline__ bool ortho_done(const EigControl* c, int k, int pass) {
  return c->err | c->bad || (pass > 0 && k * __longlong_as_double((long long)c->emax[0]) <= kOrthoDone);
}

constexpr int GT = 4;  // rows per tile of the Gram matrix and of the correction

// E = Z Z^T - 1 in tiles of 4 x 4 on and below the diagonal, and the largest |E|.
__global__ void __launch_bounds__(NT) gram_kernel(const double* __restrict__ Z, int n, int k, int pass,
                                                  double* __restrict__ E, EigControl* ctl) {
  __shared__ double red[NT / 32][GT * GT];
  if (ortho_done(ctl, k, pass)) return;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int bi = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while (bi * (bi + 1) / 2 > (int)blockIdx.x) --bi;
  while ((bi + 1) * (bi + 2) / 2 <= (int)blockIdx.x) ++bi;
  const int i0 = bi * GT, j0 = ((int)blockIdx.x - bi * (bi + 1) / 2) * GT;
  double acc[GT * GT];
#pragma unroll
  for (int q = 0; q < GT * GT; ++q) acc[q] = 0.0;
  for (int c = tid; c < n; c += NT) {
    double a[GT], b[GT];
#pragma unroll
    for (int u = 0; u < GT; ++u) {
      a[u] = Z[(size_t)min(i0 + u, k - 1) * n + c];
      b[u] = Z[(size_t)min(j0 + u, k - 1) * n + c];
    }
#pragma unroll
    for (int u = 0; u < GT; ++u)
#pragma unroll
      for (int v = 0; v < GT; ++v) acc[u * GT + v] = fma(a[u], b[v], acc[u * GT + v]);
  }
#pragma unroll
  for (int h = GT * GT / 2, o = 16; h >= 1; h /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = up ? acc[i] : acc[i + h], keep = up ? acc[i + h] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
  if ((lane & 1) == 0) red[wid][lane >> 1] = acc[0];
  __syncthreads();
  if (tid < GT * GT) {
    const int i = i0 + tid / GT, j = j0 + tid % GT;
    const double v = ((red[0][tid] + red[1][tid]) + (red[2][tid] + red[3][tid])) - (i == j ? 1.0 : 0.0);
    if (i < k && j < k) {
      E[(size_t)i * k + j] = v;
      E[(size_t)j * k + i] = v;
      // NaN has the larger bit pattern: it ends up above every bound
      atomicMax(&ctl->emax[pass], (unsigned long long)__double_as_longlong(fabs(v)));
    }
  }
}

// Zn = Z - E Z / 2: 4 rows and 128 columns per CTA.
__global__ void __launch_bounds__(NT) ortho_step_kernel(const double* __restrict__ Z, int n, int k, int pass,
                                                        const double* __restrict__ E, double* __restrict__ Zn,
                                                        const EigControl* ctl) {
  if (ortho_done(ctl, k, pass)) return;
  const int i0 = blockIdx.y * GT, c = blockIdx.x * NT + threadIdx.x;
  if (c >= n) return;
  double acc[GT];
#pragma unroll
  for (int u = 0; u < GT; ++u) acc[u] = 0.0;
#pragma unroll 4
  for (int j = 0; j < k; ++j) {
    const double z = Z[(size_t)j * n + c];
#pragma unroll
    for (int u = 0; u < GT; ++u) acc[u] = fma(E[(size_t)min(i0 + u, k - 1) * k + j], z, acc[u]);
  }
#pragma unroll
  for (int u = 0; u < GT; ++u)
    if (i0 + u < k) Zn[(size_t)(i0 + u) * n + c] = fma(-0.5, acc[u], Z[(size_t)(i0 + u) * n + c]);
}

size_t panels_of(int n) { return n > 2 ? (size_t)(n - 2 + kPanel - 1) / kPanel : 0; }
}  // namespace

size_t trivec_scratch_doubles(int n, int k) {
  return panels_of(n) * kPanel * kPanel + 2 * (size_t)n * k + (size_t)k * k;
}

bool trivec_fits(int n) { return vectors_smem(n) <= 220 * 1024 && values_smem(n) <= 220 * 1024; }

int trivec_launch(const double* A, int n, int k, const double* d, const double* e, const double* beta, double* w,
                  double* ZT, double* scratch, bool exact, EigControl* ctl, cudaStream_t s) {
  const int np = (int)panels_of(n);
  double* Tf = scratch;
  double* Y = Tf + (size_t)np * kPanel * kPanel;
  double* Q = Y + (size_t)n * k;
  double* E = Q + (size_t)n * k;
  double* wv = E;  // eigenvalues on their way to w, before the Gram matrix
  DF_CUDA(cudaFuncSetAttribute(tri_values_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  tri_values_kernel<<<k + np, NT, values_smem(n), s>>>(A, n, k, d, e, beta, w, Tf, ctl);
  DF_LAUNCHED("tri_values_kernel");
  DF_CUDA(cudaFuncSetAttribute(tri_vectors_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  tri_vectors_kernel<<<k, NT, vectors_smem(n), s>>>(n, k, d, e, w, Y, wv, exact, ctl);
  DF_LAUNCHED("tri_vectors_kernel");
  DF_CUDA(cudaFuncSetAttribute(back_transform_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  back_transform_kernel<<<k, NT, sizeof(double) * (size_t)n, s>>>(A, n, Tf, Y, wv, w, Q, ctl);
  DF_LAUNCHED("back_transform_kernel");
  const int kt = (k + GT - 1) / GT;
  const dim3 grid((n + NT - 1) / NT, kt);
  for (int pass = 0; pass < 3; ++pass) {
    const double* from = pass == 1 ? ZT : Q;
    double* to = pass == 1 ? Q : ZT;
    gram_kernel<<<kt * (kt + 1) / 2, NT, 0, s>>>(from, n, k, pass, E, ctl);
    DF_LAUNCHED("gram_kernel");
    ortho_step_kernel<<<grid, NT, 0, s>>>(from, n, k, pass, E, to, ctl);
    DF_LAUNCHED("ortho_step_kernel");
  }
  return DF_OK;
}

}  // namespace dfscf

DF_BOUNDS_READER(bounds_read_trivec)
