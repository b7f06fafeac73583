// s-type Gaussian integrals: Boys entry point, one-electron S/T/V, the two-centre
// Coulomb metric and the three-centre tensor (Q|mn) of the density-fitting equations
// (arXiv 2506.06661, Section "Density fitting").  Products of two primitives use the
// Gaussian product theorem of the paper's overlap example: p = a + b, mu = ab/p,
// P = (aA + bB)/p.
#include "common.cuh"
#include "boys.cuh"
#include "kernels.cuh"

namespace dfscf {

__device__ __forceinline__ double norm_s(double a) {
  // (2a/pi)^(3/4)
  double x = 2.0 * a / kPi;
  return sqrt(x * sqrt(x));
}

__global__ void boys_kernel(const double* __restrict__ t, long n, double* __restrict__ out) {
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = boys_f0(t[i]);
}

// S_ab = N_a N_b (pi/p)^(3/2) e^{-mu R^2};  T_ab = mu (3 - 2 mu R^2) S_ab;
// V_ab = -sum_C Z_C N_a N_b (2pi/p) e^{-mu R^2} F0(p |P - C|^2).
__global__ void int1e_kernel(const double* __restrict__ xyz, const double* __restrict__ ex, int nao,
                             const double* __restrict__ nxyz, const double* __restrict__ nz, int natm,
                             double* __restrict__ S, double* __restrict__ T, double* __restrict__ V) {
  __shared__ double sn[4 * 128];
  int a = blockIdx.y;
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  bool ok = b < nao;
  int bb = ok ? b : 0;
  double ea = ex[a], eb = ex[bb];
  double p = ea + eb, mu = ea * eb / p;
  double dx = xyz[3 * a] - xyz[3 * bb], dy = xyz[3 * a + 1] - xyz[3 * bb + 1], dz = xyz[3 * a + 2] - xyz[3 * bb + 2];
  double r2 = dx * dx + dy * dy + dz * dz;
  double kab = norm_s(ea) * norm_s(eb) * exp(-mu * r2);
  double px = (ea * xyz[3 * a] + eb * xyz[3 * bb]) / p;
  double py = (ea * xyz[3 * a + 1] + eb * xyz[3 * bb + 1]) / p;
  double pz = (ea * xyz[3 * a + 2] + eb * xyz[3 * bb + 2]) / p;
  double v = 0.0;
  if (V) {
    for (int c0 = 0; c0 < natm; c0 += 128) {
      __syncthreads();
      for (int c = threadIdx.x; c < 128 && c0 + c < natm; c += blockDim.x) {
        sn[4 * c] = nxyz[3 * (c0 + c)];
        sn[4 * c + 1] = nxyz[3 * (c0 + c) + 1];
        sn[4 * c + 2] = nxyz[3 * (c0 + c) + 2];
        sn[4 * c + 3] = nz[c0 + c];
      }
      __syncthreads();
      int cn = min(128, natm - c0);
      for (int c = 0; c < cn; ++c) {
        double qx = px - sn[4 * c], qy = py - sn[4 * c + 1], qz = pz - sn[4 * c + 2];
        v -= sn[4 * c + 3] * boys_f0(p * (qx * qx + qy * qy + qz * qz));
      }
    }
    v *= kab * 2.0 * kPi / p;
  }
  if (!ok) return;
  double s = kab * (kPi / p) * sqrt(kPi / p);
  size_t o = (size_t)a * nao + b;
  if (S) S[o] = s;
  if (T) T[o] = mu * (3.0 - 2.0 * mu * r2) * s;
  if (V) V[o] = v;
}

// (c|d) = N_c N_d 2 pi^{5/2} / (c d sqrt(c + d)) F0(cd/(c+d) R^2).  With omega > 0 the
// long-range operator erf(omega r)/r of the paper's LRDF split: the reduced exponent
// rho = cd/(c+d) becomes rho f in the Boys argument and the prefactor gains sqrt(f),
// f = omega^2 / (rho + omega^2).
// One lane per column d and 16 rows c, whose factors N_c / c are formed once per CTA.
constexpr int I2C_ROWS = 16;
__global__ void __launch_bounds__(128) int2c_kernel(const double* __restrict__ xyz, const double* __restrict__ ex,
                                                    int naux, double omega, const double* __restrict__ table,
                                                    double* __restrict__ M) {
  __shared__ double sc[I2C_ROWS][5];  // exponent, centre, N_c / c
  const int c0 = blockIdx.y * I2C_ROWS, nc = min(I2C_ROWS, naux - c0);
  if ((int)threadIdx.x < nc) {
    const int c = c0 + threadIdx.x;
    const double e = ex[c];
    sc[threadIdx.x][0] = e;
    sc[threadIdx.x][1] = xyz[3 * c];
    sc[threadIdx.x][2] = xyz[3 * c + 1];
    sc[threadIdx.x][3] = xyz[3 * c + 2];
    sc[threadIdx.x][4] = norm_s(e) / e;
  }
  __syncthreads();
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= naux) return;
  const double ed = ex[d], x = xyz[3 * d], y = xyz[3 * d + 1], z = xyz[3 * d + 2];
  const double nd = norm_s(ed) / ed, k = 2.0 * kPi * kPi * sqrt(kPi);
  for (int i = 0; i < nc; ++i) {
    const double ec = sc[i][0], dx = sc[i][1] - x, dy = sc[i][2] - y, dz = sc[i][3] - z;
    const double r2 = dx * dx + dy * dy + dz * dz;
    const double q = rsqrt_fast(ec + ed);
    double pre = (sc[i][4] * nd) * (k * q), rho = ec * ed * (q * q);  // the same bits for (c, d) and (d, c)
    if (omega > 0.0) {
      const double f = omega * omega / (rho + omega * omega);
      pre *= sqrt(f);
      rho *= f;
    }
    M[DF_IX((size_t)(c0 + i) * naux + d, (size_t)naux * naux)] = pre * boys_f0_table(rho * r2, table);
  }
}

// Row k of the Boys table: (-1)^j F_j(t) / j!, j = 0..6, at t = k / 32.  Below t = 10, F_6 from its
// series e^-t sum_i (2t)^i / (13 15 .. (13 + 2i)) (all terms positive) and downward recursion
// F_{j-1} = (2t F_j + e^-t) / (2j - 1); above, upward from F_0.
__global__ void boys_table_kernel(double* __restrict__ table) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= BOYS_ROWS) return;
  const double t = k * 0.03125, et = exp(-t);
  double F[7];
  if (t < 10.0) {
    double r = 1.0;
#pragma unroll
    for (int i = 47; i >= 1; --i) r = fma(2.0 * t * (1.0 / (13 + 2 * i)), r, 1.0);
    F[6] = et * r * (1.0 / 13.0);
#pragma unroll
    for (int j = 6; j >= 1; --j) F[j - 1] = fma(2.0 * t, F[j], et) * (1.0 / (2 * j - 1));
  } else {
    F[0] = boys_f0(t);
    const double h = 0.5 / t;
#pragma unroll
    for (int j = 0; j < 6; ++j) F[j + 1] = ((2 * j + 1) * F[j] - et) * h;
  }
  double f = 1.0;
#pragma unroll
  for (int j = 0; j < 7; ++j) {
    table[(size_t)k * BOYS_STRIDE + j] = F[j] * f;
    f *= -1.0 / (j + 1);
  }
  table[(size_t)k * BOYS_STRIDE + 7] = 0.0;
}

static int launch_boys_table(double* table, cudaStream_t s) {
  boys_table_kernel<<<(BOYS_ROWS + 31) / 32, 32, 0, s>>>(table);
  DF_LAUNCHED("boys_table_kernel");
  return DF_OK;
}

size_t boys_table_doubles() { return BOYS_TABLE; }

// Per packed pair mn: product exponent p, centre P and K_mn = N_m N_n e^{-mu R^2} 2 pi^{5/2} / p.
__global__ void pair_table_kernel(const double* __restrict__ xyz, const double* __restrict__ ex, long npair,
                                  double* __restrict__ pp, double* __restrict__ px, double* __restrict__ py,
                                  double* __restrict__ pz, double* __restrict__ pk) {
  long ij = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (ij >= npair) return;
  int a, b;
  unpack_pair(ij, a, b);
  double ea = ex[a], eb = ex[b];
  double p = ea + eb, mu = ea * eb / p;
  double dx = xyz[3 * a] - xyz[3 * b], dy = xyz[3 * a + 1] - xyz[3 * b + 1], dz = xyz[3 * a + 2] - xyz[3 * b + 2];
  pp[ij] = p;
  px[ij] = (ea * xyz[3 * a] + eb * xyz[3 * b]) / p;
  py[ij] = (ea * xyz[3 * a + 1] + eb * xyz[3 * b + 1]) / p;
  pz[ij] = (ea * xyz[3 * a + 2] + eb * xyz[3 * b + 2]) / p;
  pk[ij] = norm_s(ea) * norm_s(eb) * exp(-mu * (dx * dx + dy * dy + dz * dz)) * 2.0 * kPi * kPi * sqrt(kPi) / p;
}

// (Q|mn) = K_mn N_Q / (c sqrt(p + c)) F0(p c / (p + c) |P - C|^2), written row Q of R
// (row stride ld, padding columns [npair, ld) set to zero).  One lane per pair mn and 8 rows Q:
// the pair is loaded once, and FP64 work is about 28 instructions per integral.
constexpr int I3C_ROWS = 8;
__global__ void __launch_bounds__(256) int3c_kernel(const double* __restrict__ pp, const double* __restrict__ px,
                                                    const double* __restrict__ py, const double* __restrict__ pz,
                                                    const double* __restrict__ pk, long npair, long ld,
                                                    const double* __restrict__ axyz, const double* __restrict__ aex,
                                                    int naux, int q0, double omega, const double* __restrict__ table,
                                                    double* __restrict__ R) {
  __shared__ double sq[I3C_ROWS][5];
  q0 += blockIdx.y * I3C_ROWS;
  const int nq = min(I3C_ROWS, naux - q0);
  if ((int)threadIdx.x < nq) {
    const int q = q0 + threadIdx.x;
    const double c = aex[q];
    sq[threadIdx.x][0] = c;
    sq[threadIdx.x][1] = axyz[3 * q];
    sq[threadIdx.x][2] = axyz[3 * q + 1];
    sq[threadIdx.x][3] = axyz[3 * q + 2];
    sq[threadIdx.x][4] = norm_s(c) / c;
  }
  __syncthreads();
  const long ij = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (ij >= ld) return;
  double* row = R + (size_t)q0 * ld + ij;
  if (ij >= npair) {
    for (int i = 0; i < nq; ++i) row[(size_t)i * ld] = 0.0;
    return;
  }
  const double p = pp[ij], x = px[ij], y = py[ij], z = pz[ij], k = pk[ij];
  for (int i = 0; i < nq; ++i) {
    const double c = sq[i][0], dx = x - sq[i][1], dy = y - sq[i][2], dz = z - sq[i][3];
    const double v = rsqrt_fast(p + c);
    double rho = p * c * (v * v), pre = k * sq[i][4] * v;
    if (omega > 0.0) {  // long-range operator, as in int2c_kernel
      const double f = omega * omega / (rho + omega * omega);
      pre *= sqrt(f);
      rho *= f;
    }
    row[DF_IX((size_t)i * ld, (size_t)(naux - q0) * ld)] =
        pre * boys_f0_table(rho * (dx * dx + dy * dy + dz * dz), table);
  }
}

__global__ void enuc_kernel(const double* __restrict__ xyz, const double* __restrict__ z, int natm,
                            double* __restrict__ out) {
  __shared__ double sh[32];
  double e = 0.0;
  for (long k = threadIdx.x; k < (long)natm * natm; k += blockDim.x) {
    int a = (int)(k / natm), b = (int)(k % natm);
    if (b < a) {
      double dx = xyz[3 * a] - xyz[3 * b], dy = xyz[3 * a + 1] - xyz[3 * b + 1], dz = xyz[3 * a + 2] - xyz[3 * b + 2];
      e += z[a] * z[b] / sqrt(dx * dx + dy * dy + dz * dz);
    }
  }
  e = block_sum(e, sh);
  if (threadIdx.x == 0) *out = e;
}

int launch_int1e(const double* ao_xyz, const double* ao_exp, int nao, const double* nuc_xyz, const double* nuc_z,
                 int natm, double* S, double* T, double* V, cudaStream_t s) {
  dim3 grid((nao + 127) / 128, nao);
  int1e_kernel<<<grid, 128, 0, s>>>(ao_xyz, ao_exp, nao, nuc_xyz, nuc_z, natm, S, T, V);
  DF_LAUNCHED("int1e_kernel");
  return DF_OK;
}

int launch_int2c(const double* xyz, const double* ex, int naux, double* M, double* table, cudaStream_t s,
                 double omega) {
  DF_TRY(launch_boys_table(table, s));
  dim3 grid((naux + 127) / 128, (naux + I2C_ROWS - 1) / I2C_ROWS);
  int2c_kernel<<<grid, 128, 0, s>>>(xyz, ex, naux, omega, table, M);
  DF_LAUNCHED("int2c_kernel");
  return DF_OK;
}

int launch_pair_table(const double* ao_xyz, const double* ao_exp, int nao, double* pair_tab, cudaStream_t s) {
  long npair = npair_of(nao);
  double* pp = pair_tab;
  pair_table_kernel<<<(unsigned)((npair + 255) / 256), 256, 0, s>>>(ao_xyz, ao_exp, npair, pp, pp + npair,
                                                                    pp + 2 * npair, pp + 3 * npair, pp + 4 * npair);
  DF_LAUNCHED("pair_table_kernel");
  return DF_OK;
}

int launch_int3c(const double* ao_xyz, const double* ao_exp, int nao, const double* aux_xyz, const double* aux_exp,
                 int naux, double* R, long ld, double* pair_tab, cudaStream_t s, double omega) {
  long npair = npair_of(nao);
  double* pp = pair_tab;
  double* px = pp + npair;
  double* py = px + npair;
  double* pz = py + npair;
  double* pk = pz + npair;
  DF_TRY(launch_pair_table(ao_xyz, ao_exp, nao, pair_tab, s));
  double* table = pair_tab_boys(pair_tab, nao);
  DF_TRY(launch_boys_table(table, s));
  for (int q0 = 0; q0 < naux; q0 += 32768 * I3C_ROWS) {
    dim3 grid((unsigned)((ld + 255) / 256), (unsigned)((min(32768 * I3C_ROWS, naux - q0) + I3C_ROWS - 1) / I3C_ROWS));
    int3c_kernel<<<grid, 256, 0, s>>>(pp, px, py, pz, pk, npair, ld, aux_xyz, aux_exp, naux, q0, omega, table, R);
    DF_LAUNCHED("int3c_kernel");
  }
  return DF_OK;
}

int launch_enuc(const double* xyz, const double* z, int natm, double* out, cudaStream_t s) {
  enuc_kernel<<<1, 256, 0, s>>>(xyz, z, natm, out);
  DF_LAUNCHED("enuc_kernel");
  return DF_OK;
}

}  // namespace dfscf

using namespace dfscf;

extern "C" int df_boys_f0(const double* t, long n, double* out, cudaStream_t s) {
  clear_error();
  DF_REQUIRE(n >= 0, DF_ERR_ARG, "df_boys_f0: n < 0");
  if (n == 0) return DF_OK;
  DF_REQUIRE(t && out, DF_ERR_ARG, "df_boys_f0: null pointer");
  boys_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(t, n, out);
  DF_LAUNCHED("boys_kernel");
  return DF_OK;
}

extern "C" int df_int1e(const double* ao_xyz, const double* ao_exp, int nao, const double* nuc_xyz,
                        const double* nuc_z, int natm, double* S, double* T, double* V, cudaStream_t s) {
  clear_error();
  DF_REQUIRE(nao > 0 && natm >= 0, DF_ERR_ARG, "df_int1e: bad sizes nao=%d natm=%d", nao, natm);
  DF_REQUIRE(ao_xyz && ao_exp, DF_ERR_ARG, "df_int1e: null basis arrays");
  DF_REQUIRE(!V || natm == 0 || (nuc_xyz && nuc_z), DF_ERR_ARG, "df_int1e: V requested without nuclei");
  return launch_int1e(ao_xyz, ao_exp, nao, nuc_xyz, nuc_z, natm, S, T, V, s);
}

extern "C" int df_nuclear_repulsion(const double* nuc_xyz, const double* nuc_z, int natm, double* e_nuc,
                                    cudaStream_t s) {
  clear_error();
  DF_REQUIRE(natm >= 0 && e_nuc, DF_ERR_ARG, "df_nuclear_repulsion: bad arguments");
  DF_REQUIRE(natm == 0 || (nuc_xyz && nuc_z), DF_ERR_ARG, "df_nuclear_repulsion: null pointer");
  return launch_enuc(nuc_xyz, nuc_z, natm, e_nuc, s);
}

DF_BOUNDS_READER(bounds_read_integrals)
