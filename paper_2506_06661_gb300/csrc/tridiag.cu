// Householder reduction of a symmetric matrix to tridiagonal form on many SMs.
//
// FP64 issues one warp instruction per 64 clocks on each of an SM's four partitions, latency and
// throughput alike: four warps fill an SM, and what counts is the number of FP64 warp instructions
// in sequence.  Row r of the trailing matrix lives in the shared memory of CTA r mod G, thread t
// of a CTA works on columns t, t + 128, ...  One step kk has one exchange between the CTAs and no
// barrier:
//   1. four warps apply the rank-2 update of the step before and form y = A x (x the current
//      column) in one pass over the owned rows; y and the entries c of the next column go out;
//   2. meanwhile four other warps form the reflector v = x - alpha e_0 of x;
//   3. with A v = y - alpha c every CTA forms w and from it the next column.
// All CTAs run the same instructions on the same numbers, so they hold the same bits.
//
// The exchange is a pair of buffers of self-validating words (32 bits of data, the step's number in
// the other 32), polled by the readers: one trip through L2 instead of a barrier's three.  A CTA
// overwrites a buffer two steps later, after every CTA that reads it has published again; a
// CTA leaves when it has no row left to publish, before it reads.  Waits are bounded.
//
// Device time against two block reductions, square root and division on every warp and a grid
// barrier per step: n = 100 1.66 (one CTA) -> 0.34 ms, n = 300 2.29 -> 1.54 ms, n = 900 9.47 -> 8.25 ms
// (6.9 without EXACT).  A step takes about 3 us at n = 100, of which 1.2
// are chains of FP64 additions across lanes; at n = 900 9.2 us, 4 of them the packets' way through
// L2 (152 CTAs read 900 each), the rest the FP64 pass over the rows.
#include <algorithm>

#include "fp64.cuh"
#include "kernels.cuh"
#include "tridiag.cuh"

namespace dfscf {

namespace {
constexpr int HALF = 128;  // threads that work on the rows, and as many on the reflector
constexpr size_t kSmemLimit = 227 * 1024 - 160;  // beside the kernel's static shared memory

constexpr unsigned kTopTag = 0x3fffffffu;  // tag of the exchange before the first step

// One FP64 number in transit: low half, high half, each with the step's number above it.
struct __align__(16) Word {
  unsigned long long lo, hi;
};
// What the owner of a row publishes: one 32-byte sector, which no other CTA writes.  (With the y and the
// c in arrays of their own two CTAs write each sector: 8.0 instead of 6.9 ms at n = 900.)
struct __align__(32) Packet {
  Word y, c;
};

__device__ __forceinline__ void ll_store(Word* p, double v, unsigned tag) {
  const unsigned long long t = (unsigned long long)tag << 32;
  const unsigned long long lo = t | (unsigned)__double2loint(v), hi = t | (unsigned)__double2hiint(v);
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ bool ll_load(const Word* p, unsigned tag, double& v) {
  unsigned long long lo, hi;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
  v = __hiloint2double((int)(unsigned)hi, (int)(unsigned)lo);
  return (unsigned)(lo >> 32) == tag && (unsigned)(hi >> 32) == tag;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier of one half of the CTA (1: the row warps, 2: the reflector warps) or of both (3).  The
// instruction counts whole warps and wants them converged, and the lanes of a warp leave a polling
// loop one by one: they meet first.
__device__ __forceinline__ void bar(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Two roundings of the same reduction.  EXACT (the eigensolver's own entry points): the update
// v_i w_j + w_i v_j is rounded before it is subtracted, w carries the factor b, and the reflector's
// norm and b are good to half an ulp.  Otherwise (the iterations of an SCF): the update is two FMAs into
// the element, which round it twice at its own size, v carries b, and norm and b are good to one or
// two ulps.  Space of the 90 lowest of 900 rows, with the vectors of trivec.cu, geometric mean over 20
// random matrices: 1.2e-14 off and 10.0 ms against 2.3e-14 and 9.0 (inverse iteration on one thread
// block: 1.3e-14).  An SCF's density is determined to 1e-10 by its thresholds, and it is 2 to 6%
// faster with the second.
__device__ __forceinline__ double rank2(double vi, double wj, double wi, double vj) { return fma(vi, wj, wi * vj); }

// One pass over S owned rows (slots s0 .. s0 + S - 1, global rows from r0 in steps of G): the
// pending update, y = row . x, and the entry of column kk + 1.  The S sums are
// reduced together: P - 1 + log2(32 / P) additions (P = S rounded up to a power of two) instead
// of 5 S.
template <int S, bool EXACT>
__device__ __forceinline__ void rows_pass(double* __restrict__ rows, int n, int s0, int r0, int G, int kk,
                                          const double* __restrict__ x, const double* __restrict__ vp,
                                          const double* __restrict__ wt, double* red, int R, double* cnew) {
  constexpr int P = S <= 1 ? 1 : S <= 2 ? 2 : S <= 4 ? 4 : 8;
  const int t = threadIdx.x & (HALF - 1), lane = t & 31, wid = t >> 5;
  double acc[P], vr[S], wr[S];
#pragma unroll
  for (int s = 0; s < P; ++s) acc[s] = 0.0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    vr[s] = vp[r0 + s * G];
    wr[s] = wt[r0 + s * G];
  }
  const int c0 = kk + 1;
  int col = (c0 & ~(HALF - 1)) + t;
  if (col < c0) col += HALF;
  double* row = rows + (size_t)s0 * n;
  double xc = 0.0, vc = 0.0, wc = 0.0, a[S];
  auto fetch = [&](int q, double& xq, double& vq, double& wq, double (&aq)[S]) {
    xq = x[q];
    vq = vp[q];
    wq = wt[q];
#pragma unroll
    for (int s = 0; s < S; ++s) aq[s] = row[(size_t)s * n + q];
  };
  if (col < n) fetch(col, xc, vc, wc, a);
  while (col < n) {
    const int next = col + HALF;
    double xn = 0.0, vn = 0.0, wn = 0.0, an[S];
    if (next < n) fetch(next, xn, vn, wn, an);
    if (!EXACT) {
#pragma unroll
      for (int s = 0; s < S; ++s) a[s] = fma(-vr[s], wc, a[s]);
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
      a[s] = EXACT ? a[s] - rank2(vr[s], wc, wr[s], vc) : fma(-wr[s], vc, a[s]);
      row[(size_t)s * n + col] = a[s];
    }
#pragma unroll
    for (int s = 0; s < S; ++s) acc[s] = fma(a[s], xc, acc[s]);
    if (col == c0) {
#pragma unroll
      for (int s = 0; s < S; ++s) cnew[s0 + s] = a[s];
    }
    xc = xn;
    vc = vn;
    wc = wn;
#pragma unroll
    for (int s = 0; s < S; ++s) a[s] = an[s];
    col = next;
  }
  int o = 16;
#pragma unroll
  for (int h = P / 2; h >= 1; h /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = up ? acc[i] : acc[i + h];
      const double keep = up ? acc[i + h] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (; o; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
  constexpr int W = 32 / P;  // lanes that hold the same sum
  if (lane % W == 0 && lane / W < S) red[wid * R + s0 + lane / W] = acc[0];
}

template <bool EXACT>
__device__ __forceinline__ void all_rows(double* rows, int n, int s0, int s1, int cta, int G, int kk, const double* x,
                                         const double* vp, const double* wt, double* red, int R, double* cnew) {
#define DF_PASS(S)                                                                          \
  case S:                                                                                   \
    rows_pass<S, EXACT>(rows, n, s0, s0 * G + cta, G, kk, x, vp, wt, red, R, cnew);         \
    break
  for (; s0 < s1; s0 += 8) switch (min(s1 - s0, 8)) {
      DF_PASS(1);
      DF_PASS(2);
      DF_PASS(3);
      DF_PASS(4);
      DF_PASS(5);
      DF_PASS(6);
      DF_PASS(7);
      DF_PASS(8);
    }
#undef DF_PASS
}

// Dynamic shared memory: x, vp (two), wt, cn [n], R rows of n, red [4][R], cnew [R].  With vps = 1
// there is one vp and red and cnew lie in cn: the reflector half then waits for the pass over the
// rows before it writes vp, and the row half for itself before it writes cn.  NC: columns per thread
// whose packets are in flight together.
template <int NC, bool EXACT>
__global__ void __launch_bounds__(2 * HALF, 1) tridiag_kernel(double* __restrict__ A, int n, double* __restrict__ d,
                                                             double* __restrict__ e, double* __restrict__ beta, int R,
                                                             int vps, Packet* ex, EigControl* ctl) {
  extern __shared__ double smem_d[];
  __shared__ double sh_sigma[4], sh_pv[4], sh_ref[5];
  __shared__ int give_up;
  __shared__ unsigned sh_top;
  if (NC < 8) vps = 2;  // the plan takes one vp for large n only
  const int G = (int)gridDim.x, cta = (int)blockIdx.x, tid = threadIdx.x;
  const int t = tid & (HALF - 1), lane = tid & 31, wid = t >> 5;
  const bool reflector_half = tid >= HALF;
  double* x = smem_d;         // current column, rows kk + 1 ..
  double* v2 = smem_d + n;    // the pending update is A -= v2 wt^T + wt v2^T; by parity
  double* wt = v2 + vps * (size_t)n;
  double* cn = wt + n;  // the next column before this step's update
  double* rows = cn + n;
  double* red = vps == 2 ? rows + (size_t)R * n : cn;
  double* cnew = red + 4 * R;
  const unsigned limit = ctl->limit, off_tag = ctl->extra ? 0x40000000u : 0u;
  const bool writer = cta == (n - 1) % G;  // the CTA that stays to the end writes the results
  const int nrows = (n - 1 - cta) / G + 1, last_row = (nrows - 1) * G + cta;
  bool lost = false;
  unsigned it = 0;
  // A wait ends after `limit` polls, or two seconds and 0.1 ms a row after the kernel's start: a poll
  // takes a microsecond, and several when every CTA of a full grid polls.
  const unsigned long long t0 = global_ns();
  auto tired = [&]() {
    const bool look = (++it & 255u) == 0u;
    if (it > limit || (look && global_ns() - t0 > 2000000000ull + 100000ull * (unsigned)n)) {
      atomicCAS(&ctl->err, 0, 1);
      return true;
    }
    return look && *(volatile int*)&ctl->err != 0;
  };
  unsigned top = 0;  // high word of the largest |element|
  for (int s = 0; s < nrows; ++s)
    for (int j = tid; j < n; j += 2 * HALF) {
      const double a = A[DF_IX((size_t)(s * G + cta) * n + j, (size_t)n * n)];
      rows[(size_t)s * n + j] = a;
      top = max(top, (unsigned)__double2hiint(a) & 0x7fffffffu);
    }
  // The matrix is scaled by a power of two to a largest element in [1, 2): products of three of its
  // elements stay in range.  One exchange, in the buffer of step 1.
  top = __reduce_max_sync(0xffffffffu, top);
  if (tid == 0) {
    give_up = 0;
    sh_top = 0;
  }
  __syncthreads();
  if (lane == 0) atomicMax(&sh_top, top);
  __syncthreads();
  if (tid == 0) ll_store(&ex[n + cta].y, __hiloint2double((int)sh_top, 0), kTopTag);
  if (last_row < 1) return;  // row 0 alone: nothing to publish
  for (int q = tid; q < G && !lost; q += 2 * HALF) {
    double v;
    while (!ll_load(&ex[n + q].y, kTopTag + off_tag, v) && !(lost = tired())) {
    }
    top = max(top, (unsigned)__double2hiint(v));
  }
  if (lost) give_up = 1;
  top = __reduce_max_sync(0xffffffffu, top);
  if (lane == 0) atomicMax(&sh_top, top);
  __syncthreads();
  if (give_up) return;
  const int tex = (int)(sh_top >> 20);
  const bool scaled = tex > 0 && tex < 2046;  // neither zero nor infinite
  const double down = scaled ? __hiloint2double((2046 - tex) << 20, 0) : 1.0;
  const double up = scaled ? __hiloint2double(tex << 20, 0) : 1.0;
  for (int s = 0; s < nrows; ++s)
    for (int j = tid; j < n; j += 2 * HALF) rows[(size_t)s * n + j] *= down;
  // Column 0 is never overwritten: reflector r goes to columns r + 1 .. of row r, after the owner
  // of that row, who has read it above, published from it (row 0 is not read again).
  for (int i = tid; i < n; i += 2 * HALF) {
    x[i] = A[(size_t)i * n] * down;
    v2[(vps - 1) * n + i] = 0.0;  // no update is pending
    wt[i] = 0.0;
  }
  if (writer && tid == 0) d[0] = A[0];
  __syncthreads();

  int s0 = 0;  // first slot with row > kk
  for (int kk = 0; kk + 2 < n; ++kk) {
    const int c1 = kk + 2, base = c1 & ~(HALF - 1);
    const double* vp = v2 + (vps == 2 ? (size_t)((kk & 1) ^ 1) * n : 0);  // of the step before
    double* vn = v2 + (vps == 2 ? (size_t)(kk & 1) * n : 0);
    if (reflector_half) {
      // ---- reflector of x, while the other half works on the rows: v = x but for v0,
      // H = 1 - b v v^T
      if (last_row <= kk + 1) return;
      double part = 0.0;
      for (int col = base + t; col < n; col += HALF)
        if (col >= c1) part = fma(x[col], x[col], part);
      part = warp_sum(part);
      if (lane == 0) sh_sigma[wid] = part;
      bar(2, HALF);
      if (wid == 0) {
        const double sigma = (sh_sigma[0] + sh_sigma[1]) + (sh_sigma[2] + sh_sigma[3]);
        const double x0 = x[kk + 1];
        double alpha = x0, b = 0.0, v0 = 0.0;
        if (__double_as_longlong(sigma) != 0) {
          const double n2 = fma(x0, x0, sigma);
          const bool fast = ordinary(n2);
          const double rs = fast ? rsqrt_ordinary(n2) : 0.0, nr = n2 * rs;
          const double nrm = !fast ? sqrt(n2) : EXACT ? fma(fma(-nr, nr, n2), 0.5 * rs, nr) : nr;
          alpha = __double2hiint(x0) >= 0 ? -nrm : nrm;
          v0 = x0 - alpha;
          const double vv = fma(v0, v0, sigma), rc = fast ? rcp_ordinary(vv) : 0.0;
          b = !fast ? 2.0 / vv : EXACT ? 2.0 * fma(fma(-vv, rc, 1.0), rc, rc) : 2.0 * rc;
        }
        if (lane == 0) {
          sh_ref[0] = alpha;
          sh_ref[1] = b;
          sh_ref[2] = v0;
          sh_ref[3] = 0.5 * b;
          sh_ref[4] = EXACT ? v0 : b * v0;
          if (writer) {
            A[(size_t)kk * n + kk + 1] = v0;
            e[kk] = alpha * up;
            beta[kk] = b;
          }
        }
      }
      bar(2, HALF);
      if (vps == 1) bar(3, 2 * HALF);  // the row half has read vp
      for (int col = base + t; col < n; col += HALF)
        if (col >= c1) {
          const double v = x[col];
          vn[col] = EXACT ? v : sh_ref[1] * v;
          if (writer) A[(size_t)kk * n + col] = v;
        }
      bar(3, 2 * HALF);
      bar(3, 2 * HALF);
      if (give_up) return;
      continue;
    }
    // ---- 1. pending update, y = A x ---------------------------------------------------------
    // a tag that no packet carries, in the test of the bounded wait
    const unsigned tag = (unsigned)(kk + 1), want = tag + off_tag;
    Packet* buf = ex + (size_t)(kk & 1) * n;
    if (s0 * G + cta <= kk) ++s0;
    all_rows<EXACT>(rows, n, s0, nrows, cta, G, kk, x, vp, wt, red, R, cnew);
    bar(1, HALF);
    for (int s = s0 + t; s < nrows; s += HALF) {
      const double y = (red[s] + red[R + s]) + (red[2 * R + s] + red[3 * R + s]);
      Packet* p = buf + DF_IX(s * G + cta, n);
      ll_store(&p->y, y, tag);
      ll_store(&p->c, cnew[s], tag);
    }
    if (last_row <= kk + 1) return;  // nothing to publish any more
    if (vps == 1) bar(3, 2 * HALF);
    // ---- 2. A v = y - alpha c for the own columns > kk + 1 ----------------------------------------
    it = 0;
    double y0 = 0.0, d0 = 0.0, alpha = 0.0, pv = 0.0;  // y0, d0: row kk + 1 itself
    for (int q0 = base; q0 < n; q0 += NC * HALF) {
      double y[NC], c[NC];
      bool ok;
      do {
        ok = true;
        if (q0 == base) {
          ok &= ll_load(&buf[kk + 1].y, want, y0);
          ok &= ll_load(&buf[kk + 1].c, want, d0);
        }
#pragma unroll
        for (int u = 0; u < NC; ++u) {
          const int q = q0 + t + u * HALF;
          if (q >= c1 && q < n) {
            ok &= ll_load(&buf[q].y, want, y[u]);
            ok &= ll_load(&buf[q].c, want, c[u]);
          }
        }
      } while (!ok && !lost && !(lost = tired()));
      if (q0 == base) {
        bar(3, 2 * HALF);  // the reflector is there
        alpha = sh_ref[0];
      }
#pragma unroll
      for (int u = 0; u < NC; ++u) {
        const int q = q0 + t + u * HALF;
        if (q >= c1 && q < n) {
          const double av = fma(-alpha, c[u], y[u]);
          wt[q] = av;
          cn[q] = c[u];
          pv = fma(av, x[q], pv);
        }
      }
    }
    pv = warp_sum(pv);
    if (lane == 0) sh_pv[wid] = pv;
    bar(1, HALF);
    pv = (sh_pv[0] + sh_pv[1]) + (sh_pv[2] + sh_pv[3]);
    // ---- 3. w = A v - (b/2)(v.Av) v and the next column -------------------------------------------
    const double b = sh_ref[1], v0 = sh_ref[2], u0 = sh_ref[4];
    const double av0 = fma(-alpha, d0, y0), kap = sh_ref[3] * fma(av0, v0, pv);
    const double w0 = EXACT ? b * fma(-kap, v0, av0) : fma(-kap, v0, av0);
    for (int col = base + t; col < n; col += HALF)
      if (col >= c1) {
        const double v = x[col], w1 = fma(-kap, v, wt[col]), w = EXACT ? b * w1 : w1;
        wt[col] = w;
        x[col] = EXACT ? cn[col] - rank2(v, w0, w, v0) : fma(-u0, w, fma(-vn[col], w0, cn[col]));
      }
    if (writer && tid == 0) d[kk + 1] = up * fma(-2.0 * u0, w0, d0);
    if (lost) give_up = 1;
    bar(3, 2 * HALF);
    if (give_up) return;
  }
  if (writer && tid == 0) {
    if (n >= 2) {
      const double* vp = v2 + (vps == 2 ? (size_t)((n - 3) & 1) * n : 0);  // of the last step
      const double a = rows[(size_t)(nrows - 1) * n + n - 1];
      d[n - 1] = up * (n >= 3 ? fma(-2.0 * vp[n - 1], wt[n - 1], a) : a);
      e[n - 2] = up * x[n - 1];
    }
    e[n - 1] = 0.0;
  }
}

size_t smem_of(int n, int R, int vps) {
  return sizeof(double) * (vps == 2 ? (size_t)n * (5 + R) + 5 * (size_t)R : std::max((size_t)n, 5 * (size_t)R) + (size_t)n * (3 + R));
}
}  // namespace

namespace {
using Kernel = void (*)(double*, int, double*, double*, double*, int, int, Packet*, EigControl*);
template <bool EXACT>
Kernel kernel_for(int n) {
  return n <= HALF ? tridiag_kernel<1, EXACT>
                   : n <= 2 * HALF ? tridiag_kernel<2, EXACT> : n <= 4 * HALF ? tridiag_kernel<4, EXACT> : tridiag_kernel<8, EXACT>;
}
Kernel kernel_of(int n, bool exact) { return exact ? kernel_for<true>(n) : kernel_for<false>(n); }
}  // namespace

size_t tridiag_exchange_bytes(int n) { return 2 * sizeof(Packet) * (size_t)n; }

TridiagPlan tridiag_plan(int n, int forced, bool exact) {
  TridiagPlan P;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return P;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // More CTAs shorten the pass over the rows and lengthen the exchange.  All of eigh_lowest, us:
  // n = 100: 8 CTAs 651, 16 592, 25 588, 50 596; 200: 16 1424, 32 1237, 50 1235, 100 1315;
  // 300: 25 2442, 50 2161, 100 2112, 152 2296; 450: 50 3879, 100 3535, 152 3440; 900: 100 10973,
  // 152 10051.
  int G = forced > 1 ? forced : std::min(sms, std::max(16, n / 5));
  G = std::min(G, n);
  const int R = (n + G - 1) / G;
  // Two vp until they are what keeps the rows out of shared memory (n from 1705 to 1814 on 152 SMs:
  // 1800 rows, 181 vectors take 33.9 ms here and 83.7 ms on the general path).
  const int vps = n <= 4 * HALF || smem_of(n, R, 2) <= kSmemLimit ? 2 : 1;
  const size_t smem = smem_of(n, R, vps);
  if (smem > kSmemLimit) return P;
  if (cudaFuncSetAttribute(kernel_of(n, exact), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel_of(n, exact), 2 * HALF, smem) != cudaSuccess)
    return P;
  if (G > sms * per_sm) return P;
  P.G = G;
  P.R = R;
  P.vps = vps;
  P.exact = exact;
  P.smem = smem;
  return P;
}

int tridiag_launch(double* A, int n, double* d, double* e, double* beta, const TridiagPlan& P, void* exchange,
                   EigControl* ctl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P.G);
  cfg.blockDim = dim3(2 * HALF);
  cfg.dynamicSmemBytes = P.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // the CTAs wait for one another
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  DF_CUDA(cudaLaunchKernelEx(&cfg, kernel_of(n, P.exact), A, n, d, e, beta, P.R, P.vps, (Packet*)exchange, ctl));
  return DF_OK;
}

}  // namespace dfscf

DF_BOUNDS_READER(bounds_read_tridiag)
