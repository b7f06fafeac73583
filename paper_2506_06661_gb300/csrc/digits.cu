// Digit products (digits.cuh): slicing kernels, the tcgen05 GEMM and its launchers.
//
// GEMM tile: 128 rows x 2 G columns (G = 16 or 32), as two column groups with accumulators of
// their own (NS orders x G columns of TMEM each).  The NS digit planes of a group's B rows lie
// stacked in shared memory, so one MMA of N = (NS - a) G multiplies digit plane a of A with
// planes 0 .. NS-1-a of B and adds straight into the accumulators of orders a .. NS-1: 7 MMAs
// per K step of 16 instead of 28, with A read 7 times instead of 28 (125 B/clk of shared memory
// at the full tensor rate).  While eight epilogue warps drain one group the tensor cores work
// on the other: the groups run 64-term chunks staggered by one 32-term stage, so each stage is
// used by both groups back to back and two 84 KB stages suffice.
// FP64 exchange at nao 1000, naux 3000, nocc 100: 914 ms with FP64 FMAs (0.99 TFLOP/s, 0.8 of the
// FP64 peak), 70 ms here: slicing 28 ms, the two contractions 42 ms.  At nao 1500, naux 4500, nocc
// 150 the half-transform issues 0.51 and the SYRK 0.53 of the sustained BF16 rate.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "digits.cuh"
#include "kernels.cuh"
#include "tcgen05.cuh"

namespace dfscf {
namespace digits {

using namespace umma;

constexpr int EPI_WARPS = 8;
constexpr int GEMM_THREADS = 64 + 32 * EPI_WARPS;
constexpr int MAX_RING = 4;

enum Mode { MATRIX = 0, HALF_TRANSFORM = 1 };

struct Params {
  int mode;
  int M, N;             // rows of A, rows of B
  int groups;           // column groups per tile (1 when N <= G)
  int ntn;              // column tiles
  int nst, nst_split;   // stages of the whole K range, per split
  int ring;             // shared-memory stages
  uint32_t stage_bytes, b_off, g_bytes;
  const unsigned *ka, *kb;
  double alpha, beta;
  double* C;
  long ldc, sC;
  int lower, trans;     // lower tiles only; C stored transposed (C[col ldc + row])
  // half-transform
  int nao, p0;
  double* X;
  long ldx, xcol0;
  unsigned* xkey;
  // FP64 originals (rows with non-finite elements)
  const double *A0, *B0;
  long sam, sak, sbn, sbk, K;
  int* err;
};

__device__ __forceinline__ void tmem_ld_x8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
          smem_u32(dst)),
      "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// (hi + lo 2^-15) 2^e rounded to FP64 once (0 <= lo < 2^15).
__device__ __forceinline__ double assemble(long long hi, int lo, int e) {
  unsigned long long tl = ((unsigned long long)hi << 15) | (unsigned long long)lo;
  long long th = hi >> 49;
  const bool neg = th < 0;
  if (neg) {
    tl = ~tl + 1ull;
    th = ~th + (tl == 0 ? 1 : 0);
  }
  if (th == 0 && tl == 0) return 0.0;
  unsigned long long m;
  bool sticky = false;
  int n;
  if (th) {
    const int sh = __clzll(th);
    m = sh ? ((unsigned long long)th << sh) | (tl >> (64 - sh)) : (unsigned long long)th;
    sticky = (tl << sh) != 0;
    n = 128 - sh;
  } else {
    const int sh = __clzll((long long)tl);
    m = tl << sh;
    n = 64 - sh;
  }
  const unsigned r = (unsigned)(m & 0x7ffull);
  m >>= 11;
  if (r > 0x400u || (r == 0x400u && (sticky || (m & 1)))) ++m;
  const int be = n - 1 + e - 15 + 1023;
  if (be >= 1 && be <= 2045) {
    const unsigned long long bits = ((unsigned long long)be << 52) + (m - (1ull << 52));
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0)));
  }
  const double v = scalbn((double)m, n - 53 + e - 15);
  return neg ? -v : v;
}

struct Maps {
  CUtensorMap a, b;
};

// Which group works first on stage s, and where its 64-term chunks begin and end.
__device__ __forceinline__ int group_of(int groups, int s, int o) {
  return groups == 1 ? 0 : ((s == 0 || (s & 1)) ? o : 1 - o);
}
__device__ __forceinline__ bool chunk_begins(int g, int s) { return g == 0 ? !(s & 1) : (s == 0 || (s & 1)); }
__device__ __forceinline__ bool chunk_ends(int g, int s, int last) { return s == last || (g == 0 ? (s & 1) : !(s & 1)); }
// Accumulator set of a group's chunk: the group's own, or alternating when there is one group.
__device__ __forceinline__ int acc_set(int groups, int g, int s) { return groups == 1 ? (s >> 1) & 1 : g; }

template <int G>
__global__ void __launch_bounds__(GEMM_THREADS, 1) digit_gemm_kernel(const __grid_constant__ Maps maps, const Params p) {
  constexpr int CW = G / 2;  // columns of a group per epilogue warp
  extern __shared__ uint8_t dyn_smem[];
  __shared__ uint64_t full_bar[MAX_RING], empty_bar[MAX_RING], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int mt, nt;
  if (p.lower) {  // row block mt has the column tiles that start at or left of its last row
    int t = (int)blockIdx.x, m = 0;
    const int w = G * p.groups;
    while (true) {
      const int c = min((min((m + 1) * BM, p.M) - 1) / w + 1, p.ntn);
      if (t < c) break;
      t -= c;
      ++m;
    }
    mt = m;
    nt = t;
  } else {  // column tiles of a row block side by side: they share its A tile in L2
    mt = (int)(blockIdx.x / (unsigned)p.ntn);
    nt = (int)(blockIdx.x % (unsigned)p.ntn);
  }
  const int row0 = mt * BM, col0 = nt * G * p.groups;
  const int s0 = (int)blockIdx.y * p.nst_split;
  int nst = min(p.nst_split, p.nst - s0);
  if (*(volatile const int*)p.err) nst = 0;  // a wait already gave up in another CTA
  const int last = nst - 1;

  const uint32_t base = smem_u32(dyn_smem);
  uint8_t* ring = dyn_smem + ((1024u - (base & 1023u)) & 1023u);
  constexpr uint32_t ncols = 2 * NS * G <= 256 ? 256 : 512;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.ring; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], EPI_WARPS);
    }
    abort_flag = 0;
    mbar_fence_init();
    tma_prefetch(&maps.a);
    tma_prefetch(&maps.b);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base, ncols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  int issued = 0;

  if (warp == 0 && lane == 0 && nst > 0) {
    // ---- TMA producer ----------------------------------------------------------------
    for (int i = 0; i < nst; ++i) {
      const int s = i % p.ring;
      const uint32_t ph = (uint32_t)(i / p.ring) & 1u;
      if (!mbar_wait(&empty_bar[s], ph ^ 1u, &abort_flag)) {
        abort_flag = 1;
        break;
      }
      uint8_t* st = ring + (size_t)s * p.stage_bytes;
      mbar_arrive_expect_tx(&full_bar[s], p.stage_bytes);
      const int kx = (s0 + i) * BK;
      tma_load_3d(st, &maps.a, &full_bar[s], kx, row0, 0);
      for (int g = 0; g < p.groups; ++g) tma_load_3d(st + p.b_off + g * p.g_bytes, &maps.b, &full_bar[s], kx, col0 + g * G, 0);
      issued = i + 1;
    }
  } else if (warp == 1 && lane == 0 && nst > 0) {
    // ---- MMA issuer ------------------------------------------------------------------
    uint32_t used[2] = {0, 0};
    bool ok = true;
    for (int i = 0; i < nst && ok; ++i) {
      const int s = i % p.ring;
      if (!mbar_wait(&full_bar[s], (uint32_t)(i / p.ring) & 1u, &abort_flag)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t st = smem_u32(ring + (size_t)s * p.stage_bytes);
      for (int o = 0; o < p.groups; ++o) {
        const int g = group_of(p.groups, i, o), b = acc_set(p.groups, g, i);
        const bool begin = chunk_begins(g, i);
        if (begin) {
          if (!mbar_wait(&acc_empty[b], (used[b] & 1u) ^ 1u, &abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
        }
        const uint64_t bd = desc_sw<BK>(st + p.b_off + (uint32_t)g * p.g_bytes);
        const uint64_t ad = desc_sw<BK>(st);
        const uint32_t acc = tmem + (uint32_t)(b * NS * G);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
#pragma unroll
          for (int a = 0; a < NS; ++a) {
            const uint64_t off = (uint64_t)(kk * 32) >> 4;
            umma_bf16(acc + (uint32_t)(a * G), ad + ((uint64_t)(a * BM * BK * 2) >> 4) + off, bd + off,
                      idesc_bf16(BM, (NS - a) * G), (begin && kk == 0 && a == 0) ? 0u : 1u);
          }
        if (chunk_ends(g, i, last)) {
          umma_commit(&acc_full[b]);
          ++used[b];
        }
      }
      if (ok && i + p.ring < nst) umma_commit(&empty_bar[s]);  // the slot has another stage to come
    }
    if (!ok) abort_flag = 1;
  } else if (warp >= 2 && nst > 0) {
    // ---- epilogue: drain chunks into a 64-bit integer (orders 0..3, carries) and the fixed-
    // point rest (orders 4..6 in units of 2^-15 of order 3, 0 <= lo < 2^15) ------------------
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int row = row0 + q * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * CW);
    long long hi[2][CW];
    int lo[2][CW];
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int j = 0; j < CW; ++j) {
        hi[g][j] = 0;
        lo[g][j] = 0;
      }
    auto drain = [&](int b, long long(&h)[CW], int(&l)[CW]) {
#pragma unroll
      for (int c = 0; c < CW; c += 8) {
        uint32_t v[NS][8];
#pragma unroll
        for (int t = 0; t < NS; ++t) tmem_ld_x8(taddr + (uint32_t)(b * NS * G + t * G + c), v[t]);
        tmem_wait_ld();
        if (c + 8 == CW) {  // the last read of this chunk: the accumulators may be overwritten
          tc_fence_before();
          if (lane == 0) mbar_arrive(&acc_empty[b]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int i0 = __float2int_rn(__uint_as_float(v[0][j])), i1 = __float2int_rn(__uint_as_float(v[1][j])),
                    i2 = __float2int_rn(__uint_as_float(v[2][j])), i3 = __float2int_rn(__uint_as_float(v[3][j]));
          // order 4 is at most 5 * 64 * 2^16 < 2^24.4; orders 5 and 6 over 8 stay below 2^22, where
          // adding 1.5 * 2^23 rounds to an integer
          const int i4 = __float2int_rn(__uint_as_float(v[4][j]));
          const float r = __uint_as_float(v[5][j]) + __uint_as_float(v[6][j]) * (1.0f / 512);
          const int x = l[c + j] + i4 * 64 + (__float_as_int(fmaf(r, 0.125f, 12582912.0f)) - 0x4B400000);
          l[c + j] = x & 0x7fff;
          h[c + j] += (long long)i0 * (1 << 27) + ((long long)i1 * (1 << 18) + ((long long)i2 * (1 << 9) + (i3 + (x >> 15))));
        }
      }
    };
    uint32_t done[2] = {0, 0};
    bool ok = true;
    for (int i = 0; i < nst && ok; ++i)
      for (int o = 0; o < p.groups; ++o) {
        const int g = group_of(p.groups, i, o);
        if (!chunk_ends(g, i, last)) continue;
        const int b = acc_set(p.groups, g, i);
        ok = mbar_wait(&acc_full[b], done[b] & 1u, &abort_flag);
        ok = __all_sync(0xffffffffu, ok);  // the TMEM loads are warp-collective
        if (!ok) break;
        ++done[b];
        tc_fence_after();
        if (g == 0) drain(b, hi[0], lo[0]);
        else drain(b, hi[1], lo[1]);
      }
    if (!ok) abort_flag = 1;
    if (ok && row < p.M) {
      const unsigned ka = p.ka[row];
      const int fa = key_field(ka);
      const bool bada = key_bad(ka);
      int P = 0, m = row;
      if (p.mode == HALF_TRANSFORM) {
        P = row / p.nao;
        m = row - P * p.nao;
      }
      unsigned big = 0;
      const long rstep = p.trans ? 1 : p.ldc, cstep = p.trans ? p.ldc : 1;
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        if (g >= p.groups) break;
#pragma unroll
        for (int j0 = 0; j0 < CW; j0 += 8) {
          const int colb = col0 + g * G + half * CW + j0;
          double old[8];  // what the outputs add to, loaded ahead of the stores
          double* cb = nullptr;
          if (p.mode == MATRIX) {
            cb = p.C + (size_t)blockIdx.y * p.sC +
                 DF_IX((size_t)row * rstep + (size_t)min(colb, p.N - 1) * cstep, p.trans ? (size_t)p.N * p.ldc : (size_t)p.M * p.ldc);
            if (p.beta != 0.0) {
#pragma unroll
              for (int j = 0; j < 8; ++j) old[j] = colb + j < p.N ? cb[j * cstep] : 0.0;
            }
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int col = colb + j;
            if (col >= p.N) break;
            const unsigned kb = p.kb[col];
            // digit d_a has the weight 2^(E - 8 - 9 a), E = field - 1022; hi counts order 3
            double v = assemble(hi[g][j0 + j], lo[g][j0 + j], fa + key_field(kb) - 2044 - 16 - 27);
            if (bada || key_bad(kb)) {
              v = 0.0;
              const long k0 = (long)s0 * BK, k1 = min(p.K, k0 + (long)nst * BK);
              for (long k = k0; k < k1; ++k) {
                double x;
                if (p.mode == HALF_TRANSFORM) {
                  const long a = max((long)m, k), c = min((long)m, k);
                  x = p.A0[(long)(p.p0 + P) * p.sam + a * (a + 1) / 2 + c];
                } else {
                  x = p.A0[row * p.sam + k * p.sak];
                }
                v = fma(x, p.B0[col * p.sbn + k * p.sbk], v);
              }
            }
            if (p.mode == HALF_TRANSFORM) {
              p.X[DF_IX((size_t)m * p.ldx + p.xcol0 + (size_t)P * p.N + col, (size_t)p.nao * p.ldx)] = v;
              big = max(big, high_key(v));
            } else {
              // FP64 instructions only where they are needed: +-1 factors flip a sign or add
              const double w = p.alpha == 1.0 ? v : (p.alpha == -1.0 ? -v : p.alpha * v);
              cb[j * cstep] = p.beta == 0.0 ? w : (p.beta == 1.0 ? old[j] + w : fma(p.beta, old[j], w));
            }
          }
        }
      }
      if (p.mode == HALF_TRANSFORM && big) atomicMax(p.xkey + m, big);
    }
  }
  __syncwarp();  // the one-lane roles above; TMEM is freed by a whole warp
  tc_fence_before();
  __syncthreads();
  if (abort_flag && warp == 0 && lane == 0) {
    atomicExch(p.err, 1);
    for (int s = 0; s < p.ring; ++s) {  // loads in flight land before the shared memory goes
      const int lst = issued - 1 - ((issued - 1 - s) % p.ring + p.ring) % p.ring;
      if (issued > 0 && lst >= 0 && lst % p.ring == s) mbar_wait(&full_bar[s], (uint32_t)(lst / p.ring) & 1u, nullptr);
    }
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, ncols);
  }
}

// ---- slicing ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned cta_max_key(unsigned v, unsigned* sh) {
  for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned t = 0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t = max(t, sh[i]);
  return t;
}

// Rows contiguous over k; one CTA per row (and per slice blockIdx.x of K when the keys are given).
template <bool KEYS>
__global__ void __launch_bounds__(128) slice_rows_kernel(const double* __restrict__ A, long lda, long rows, long K,
                                                         long ld, unsigned* __restrict__ key,
                                                         __nv_bfloat16* __restrict__ out) {
  __shared__ unsigned sh[4];
  const long r = blockIdx.y + (long)blockIdx.z * 32768;
  if (r >= rows) return;
  const double* a = A + (size_t)r * lda;
  unsigned k;
  if (KEYS) {
    k = key[r];
  } else {
    unsigned t = 0;
    for (long i = threadIdx.x; i < K; i += blockDim.x) t = max(t, high_key(a[i]));
    k = cta_max_key(t, sh);
    if (threadIdx.x == 0) key[r] = k;
  }
  const bool bad = key_bad(k);
  const int f = key_field(k);
  const size_t plane = (size_t)rows * ld;
  for (long c = ((long)blockIdx.x * blockDim.x + threadIdx.x) * 8; c < ld; c += (long)gridDim.x * blockDim.x * 8) {
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = (c + u < K && !bad) ? a[c + u] : 0.0;
    store_digits8(x, f, out + DF_IXW((size_t)r * ld + c, 8, plane), plane);
  }
}

// Rows strided: element (r, k) = A[k lda + r]; one CTA per 32 rows, lanes along the rows.
__global__ void __launch_bounds__(256) slice_cols_kernel(const double* __restrict__ A, long lda, long rows, long K,
                                                         long ld, unsigned* __restrict__ key,
                                                         __nv_bfloat16* __restrict__ out) {
  __shared__ unsigned sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long r = (long)blockIdx.x * 32 + lane;
  const bool live = r < rows;
  unsigned t = 0;
  if (live)
    for (long k = w; k < K; k += 8) t = max(t, high_key(A[(size_t)k * lda + r]));
  sh[w][lane] = t;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) t = max(t, sh[i][lane]);
  if (!live) return;
  if (w == 0) key[r] = t;
  const bool bad = key_bad(t);
  const int f = key_field(t);
  const size_t plane = (size_t)rows * ld;
  for (long c = 8L * w; c < ld; c += 64) {
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = (c + u < K && !bad) ? A[(size_t)(c + u) * lda + r] : 0.0;
    store_digits8(x, f, out + DF_IXW((size_t)r * ld + c, 8, plane), plane);
  }
}

// Symmetric matrices from packed rows: rows (P, m) over n.  One CTA per P and 32 rows m; tiles of
// 32 x 64 go through shared memory, read along rows left of the diagonal and along columns
// right of it, once for the row keys and (from L2) once for the digits.
constexpr int PT = 32, PN = 64;
__global__ void __launch_bounds__(256) slice_packed_kernel(const double* __restrict__ B, long ldb, int nao, int p0,
                                                           int np, long ld, unsigned* __restrict__ key,
                                                           __nv_bfloat16* __restrict__ out) {
  __shared__ double T[PT][PN + 1];
  __shared__ unsigned keys[PT];
  const int m0 = blockIdx.x * PT;
  const int P = blockIdx.y;
  const double* b = B + (size_t)(p0 + P) * ldb;
  const int tid = threadIdx.x;
  auto load = [&](int n0) {
    __syncthreads();
    // left of the diagonal (n <= m): consecutive threads along n
    if (n0 <= m0 + PT - 1) {
#pragma unroll
      for (int e = tid; e < PT * PN; e += 256) {
        const int i = e / PN, j = e % PN, m = m0 + i, n = n0 + j;
        if (n <= m && m < nao) T[i][j] = b[DF_IX((size_t)m * (m + 1) / 2 + n, ldb)];
      }
    }
    // right of it (n > m): consecutive threads along m
    if (n0 + PN - 1 > m0) {
#pragma unroll
      for (int e = tid; e < PT * PN; e += 256) {
        const int j = e / PT, i = e % PT, m = m0 + i, n = n0 + j;
        if (n > m && n < nao) T[i][j] = b[DF_IX((size_t)n * (n + 1) / 2 + m, ldb)];
      }
    }
    __syncthreads();
  };
  const int r = tid >> 3, u = tid & 7;  // 8 threads per row, 8 elements each
  const int m = m0 + r;
  unsigned t = 0;
  for (int n0 = 0; n0 < nao; n0 += PN) {
    load(n0);
    if (m < nao)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = u + 8 * j;
        if (n0 + c < nao) t = max(t, high_key(T[r][c]));
      }
  }
  for (int o = 4; o; o >>= 1) t = max(t, __shfl_xor_sync(0xffffffffu, t, o));
  const long row = (long)P * nao + m;
  if (m < nao && u == 0) key[row] = t;
  const bool bad = key_bad(t);
  const int f = key_field(t);
  const size_t plane = (size_t)np * nao * ld;
  for (int n0 = 0; n0 < nao; n0 += PN) {
    load(n0);
    const int c0 = n0 + 8 * u;
    if (m < nao && c0 < ld) {
      double x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = (c0 + j < nao && !bad) ? T[r][8 * u + j] : 0.0;
      store_digits8(x, f, out + DF_IXW((size_t)row * ld + c0, 8, plane), plane);
    }
  }
}

// 3-D map of digit planes: K (contiguous) x rows x planes, box 32 x box_rows x NS.
static int make_planes_map(CUtensorMap* map, const DigitOperand& o, int box_rows) {
  auto enc = get_encode();
  DF_REQUIRE(enc, DF_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  const uint64_t ld = (uint64_t)plane_ld(o.K);
  cuuint64_t dims[3] = {(cuuint64_t)o.K, (cuuint64_t)o.rows, (cuuint64_t)NS};
  cuuint64_t strides[2] = {ld * 2, ld * 2 * (uint64_t)o.rows};
  cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, (cuuint32_t)NS};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, o.p, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  DF_REQUIRE(r == CUDA_SUCCESS, DF_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d) for %ld x %ld digit planes", (int)r,
             o.rows, o.K);
  return DF_OK;
}

template <int G>
static int launch(const DigitOperand& A, const DigitOperand& B, Params p, int splits, cudaStream_t s) {
  Maps maps;
  DF_TRY(make_planes_map(&maps.a, A, BM));
  DF_TRY(make_planes_map(&maps.b, B, G));
  p.groups = p.N > G ? 2 : 1;
  p.ntn = (p.N + G * p.groups - 1) / (G * p.groups);
  p.nst = (int)((A.K + BK - 1) / BK);
  p.nst_split = (p.nst + splits - 1) / splits;
  p.nst_split += p.nst_split & 1;  // whole 64-term chunks
  const int ns = (p.nst + p.nst_split - 1) / p.nst_split;
  p.g_bytes = NS * G * BK * 2;
  p.b_off = NS * BM * BK * 2;
  p.stage_bytes = p.b_off + p.groups * p.g_bytes;
  p.ring = std::min<int>(MAX_RING, (220 * 1024) / (int)p.stage_bytes);
  p.K = A.K;
  long tiles = 0;
  const int mts = (p.M + BM - 1) / BM;
  if (p.lower) {
    for (int m = 0; m < mts; ++m) tiles += std::min((std::min((m + 1) * BM, p.M) - 1) / (G * p.groups) + 1, p.ntn);
  } else {
    tiles = (long)mts * p.ntn;
  }
  DF_REQUIRE(tiles < (1L << 31) && ns <= 65535, DF_ERR_ARG, "digit GEMM: too many tiles");
  // an int64 holds 2^11 drained chunks of the largest possible sums (2^52 each)
  DF_REQUIRE(p.nst_split <= 4096, DF_ERR_ARG, "digit GEMM: K range of %d stages in one split", p.nst_split);
  // splits the rounding left without work: their output slices are zeroed
  if (p.mode == MATRIX && p.beta == 0.0)
    for (int z = ns; z < splits; ++z)
      DF_CUDA(cudaMemsetAsync(p.C + (size_t)z * p.sC, 0, sizeof(double) * (size_t)p.M * p.ldc, s));
  DF_TRY(digits_prepare());
  const size_t smem = (size_t)p.ring * p.stage_bytes + 1024;
  digit_gemm_kernel<G><<<dim3((unsigned)tiles, (unsigned)ns), GEMM_THREADS, smem, s>>>(maps, p);
  DF_LAUNCHED("digit_gemm_kernel");
  return DF_OK;
}

// Columns per group: 16 for up to 32 columns (a 64-column tile would be half empty), else 32, whose
// tile reads half as many A bytes per product.
static int launch_any(const DigitOperand& A, const DigitOperand& B, const Params& p, int splits, int width,
                      cudaStream_t s) {
  return (width ? width == 16 : p.N <= 32) ? launch<16>(A, B, p, splits, s) : launch<32>(A, B, p, splits, s);
}

}  // namespace digits

using namespace digits;

int digits_prepare() {
  static bool done = false;
  if (!done) {
    const int lim = 220 * 1024 + 1024;
    DF_CUDA(cudaFuncSetAttribute(digit_gemm_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    DF_CUDA(cudaFuncSetAttribute(digit_gemm_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    done = true;
  }
  return DF_OK;
}

size_t digit_operand_bytes(long rows, long K) {
  return align_up(plane_bytes(rows, K), 256) + align_up(sizeof(unsigned) * (size_t)rows, 256);
}

DigitOperand digit_operand(void* mem, long rows, long K) {
  DigitOperand o;
  o.p = (__nv_bfloat16*)mem;
  o.key = (unsigned*)((char*)mem + align_up(plane_bytes(rows, K), 256));
  o.rows = rows;
  o.K = K;
  return o;
}

int slice_matrix(const double* A, long lda, bool trans, const DigitOperand& o, cudaStream_t s) {
  const long ld = plane_ld(o.K);
  if (trans) {
    slice_cols_kernel<<<(unsigned)((o.rows + 31) / 32), 256, 0, s>>>(A, lda, o.rows, o.K, ld, o.key, o.p);
    DF_LAUNCHED("slice_cols_kernel");
  } else {
    const dim3 grid(1, (unsigned)std::min<long>(o.rows, 32768), (unsigned)((o.rows + 32767) / 32768));
    slice_rows_kernel<false><<<grid, 128, 0, s>>>(A, lda, o.rows, o.K, ld, o.key, o.p);
    DF_LAUNCHED("slice_rows_kernel");
  }
  return DF_OK;
}

int slice_with_keys(const double* A, long lda, const DigitOperand& o, cudaStream_t s) {
  const long ld = plane_ld(o.K);
  const dim3 grid((unsigned)std::min<long>((ld / 8 + 127) / 128, 256L), (unsigned)std::min<long>(o.rows, 32768),
                  (unsigned)((o.rows + 32767) / 32768));
  slice_rows_kernel<true><<<grid, 128, 0, s>>>(A, lda, o.rows, o.K, ld, o.key, o.p);
  DF_LAUNCHED("slice_rows_kernel");
  return DF_OK;
}

int slice_packed(const double* B, long ldb, int nao, int p0, int np, const DigitOperand& o, cudaStream_t s) {
  slice_packed_kernel<<<dim3((unsigned)((nao + PT - 1) / PT), (unsigned)np), 256, 0, s>>>(B, ldb, nao, p0, np,
                                                                                      plane_ld(nao), o.key, o.p);
  DF_LAUNCHED("slice_packed_kernel");
  return DF_OK;
}

int digit_gemm(const DigitOperand& A, const DigitOperand& B, DigitSource A0, DigitSource B0, double alpha, double beta,
               double* C, long ldc, long sC, int splits, int shape, int* err, cudaStream_t s) {
  DF_REQUIRE(A.rows < INT_MAX && B.rows < INT_MAX && A.K == B.K, DF_ERR_ARG, "digit GEMM: bad operand sizes");
  Params p{};
  p.mode = MATRIX;
  p.M = (int)A.rows;
  p.N = (int)B.rows;
  p.ka = A.key;
  p.kb = B.key;
  p.alpha = alpha;
  p.beta = beta;
  p.C = C;
  p.ldc = ldc;
  p.sC = sC;
  p.lower = shape == DIGIT_LOWER;
  p.trans = shape == DIGIT_TRANSPOSED;
  p.A0 = A0.p;
  p.sam = A0.sr;
  p.sak = A0.sk;
  p.B0 = B0.p;
  p.sbn = B0.sr;
  p.sbk = B0.sk;
  p.err = err;
  return launch_any(A, B, p, std::max(1, splits), 0, s);
}

int digit_half_transform(const DigitOperand& A, const DigitOperand& Ct, const double* B, long ldb, int nao, int p0,
                         const double* C, int nocc, double* X, long ldx, long xcol0, unsigned* xkey, int* err,
                         cudaStream_t s) {
  DF_REQUIRE(A.rows < INT_MAX, DF_ERR_ARG, "half-transform: too many rows");
  Params p{};
  p.mode = HALF_TRANSFORM;
  p.M = (int)A.rows;
  p.N = nocc;
  p.ka = A.key;
  p.kb = Ct.key;
  p.nao = nao;
  p.p0 = p0;
  p.X = X;
  p.ldx = ldx;
  p.xcol0 = xcol0;
  p.xkey = xkey;
  p.A0 = B;
  p.sam = ldb;
  p.B0 = C;
  p.sbn = 1;
  p.sbk = nocc;
  p.err = err;
  return launch_any(A, Ct, p, 1, knob("fp64_ht_cols"), s);
}

}  // namespace dfscf

DF_BOUNDS_READER(bounds_read_digits)
