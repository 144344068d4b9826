// rt_dust.cu -- equilibrium dust temperatures and dust emission (Sects. 3.2
// and 4: a single dust component in equilibrium with the local radiation
// field; the emission of every cell is recomputed from its temperature in
// each Lambda-iteration step, Eq. 2).
//
// Per leaf the solve finds T with rho V E(T) = A, where
//   E(T) = 4 pi sum_i kappa_abs,i B_nu(nu_i, T) dnu_i     (erg/s/g)
// is the same for every cell.  It is tabulated once per call (log E and its
// slope on a uniform log-T grid, FP64) and each leaf inverts the cubic
// Hermite interpolant, so no leaf evaluates the Planck sum (GB300's FP64
// pipe is narrow); where E underflows at the cold end the exact sum is
// solved by safeguarded Newton instead.  Planck terms themselves are
// evaluated in 64-bit integer arithmetic (rt_planck.cuh).
#include <math_constants.h>

#include "philox.cuh"
#include "rt_internal.cuh"
#include "rt_planck.cuh"

namespace rtk {

#define C_CGS 2.99792458e10
#define H_CGS 6.62607015e-27
#define K_CGS 1.380649e-16
#define FOUR_PI 12.566370614359172

// B_nu(T) and its temperature derivative
__device__ __forceinline__ void planck_and_deriv(double nu, double T, double* B, double* dB) {
  const double x = H_CGS * nu / (K_CGS * T);
  const double em1 = expm1(x);
  if (!(em1 < HUGE_VAL)) {  // Wien tail below the double range
    *B = 0.0;
    *dB = 0.0;
    return;
  }
  const double b = 2.0 * H_CGS * nu * nu * nu / (C_CGS * C_CGS) / em1;
  *B = b;
  *dB = b * x * (1.0 + 1.0 / em1) / T;
}

__device__ __forceinline__ double emission_per_mass(const double* lam, const double* kabs, const double* dnu, int nl,
                                                    double T, double* dEdT) {
  double s = 0.0, ds = 0.0;
  for (int i = 0; i < nl; ++i) {
    const double nu = C_CGS / (lam[i] * 1e-4);
    double B, dB;
    planck_and_deriv(nu, T, &B, &dB);
    s += kabs[i] * B * dnu[i];
    ds += kabs[i] * dB * dnu[i];
  }
  if (dEdT) *dEdT = FOUR_PI * ds;
  return FOUR_PI * s;
}

// rho h^3 of a level-l cell, h = h0 2^-l; v0 = h0^3 (its exponent moved by
// 3 l, or the product itself where that leaves the normal range)
__device__ __forceinline__ double leaf_mass(double rho, double h0, double v0, int lev) {
  const uint64_t b = bits_of(v0);
  const int ex = (int)(b >> 52);
  if (ex > 3 * lev && ex < 2047) return rho * of_bits(b - ((uint64_t)(3 * lev) << 52));
  const double h = ldexp(h0, -lev);
  return rho * h * h * h;
}

// One bin of the emission as the kernels keep it in shared memory: the
// integer form, what the FP64 form needs where the integer one does not
// apply, and what the temperature derivative needs.
struct EmitBin {
  PlanckBin p;
  double hnu, inv_c;  // h nu; 1 / C_b
  double nu, kabs, dnu;
};

// dynamic shared memory of a kernel with nl bins: [2^-f table | bins]
static size_t emit_smem(int nl) { return sizeof(uint64_t) * RT_EXP2_TABLE + sizeof(EmitBin) * (size_t)nl; }

__device__ __forceinline__ void emit_setup(unsigned char* smem, const double* __restrict__ lam,
                                           const double* __restrict__ kabs, const double* __restrict__ dnu, int nl,
                                           const uint64_t*& tab, const EmitBin*& bins) {
  uint64_t* t = reinterpret_cast<uint64_t*>(smem);
  EmitBin* eb = reinterpret_cast<EmitBin*>(t + RT_EXP2_TABLE);
  for (int i = threadIdx.x; i < RT_EXP2_TABLE; i += blockDim.x) t[i] = exp2_table[i];
  for (int b = threadIdx.x; b < nl; b += blockDim.x) {
    EmitBin B;
    B.nu = C_CGS / (lam[b] * 1e-4);
    B.kabs = kabs[b];
    B.dnu = dnu[b];
    B.hnu = H_CGS * B.nu;
    const double c = FOUR_PI * B.kabs * B.dnu * (2.0 * H_CGS * B.nu * B.nu * B.nu / (C_CGS * C_CGS));
    B.p = planck_bin(B.hnu, c);
    B.inv_c = 1.0 / c;
    eb[b] = B;
  }
  __syncthreads();
  tab = t;
  bins = eb;
}

// mass * 4 pi kappa B_nu(T) dnu of one bin
__device__ __forceinline__ double emit_term(const EmitBin& B, const Norm64& inv, const Norm64& mass_n, double mass,
                                            double T, const uint64_t* tab) {
  bool ok;
  double v = planck_term(B.p, inv, mass_n, tab, ok);
  if (!ok) {
    double pl, dpl;
    planck_and_deriv(B.nu, T, &pl, &dpl);
    v = FOUR_PI * mass * B.kabs * pl * B.dnu;
  }
  return v;
}

// Tables for the temperature solve, on a uniform grid in log T (n nodes):
//   tab[3i] = log T_i, tab[3i+1] = log E(T_i), tab[3i+2] = d log E / d log T;
//   node[i]: what the inversion of the cubic Hermite interpolant of log E
//   between nodes i and i + 1 needs;
//   lg[i] = log2 E_i (f32), to find i.
// log E(log T) is smooth, so cubic Hermite interpolation between nodes
// (spacing ~1e-3 in log T for 8192 nodes) inverts it to ~1e-13 in T.
// Eight lanes share a node's bins (35 us with 12 to 30 bins; a thread per
// node, 64 blocks: 43 to 96 us).
struct InvNode {
  double inv_e;         // 1 / E_i; 0 where E_i is below the normal range: no shortcut
  double c1, c2, c3;    // log E = log E_i + t (c1 + t (c2 + t c3)), t = (log T - log T_i) / hx
  double T, hx;         // T_i, the grid's spacing
  double pad0, pad1;
};
static_assert(sizeof(InvNode) == 8 * sizeof(double), "table layout");
static constexpr int TABLE_NODES = 32;  // nodes per block; one more is evaluated for the intervals
__global__ void __launch_bounds__(8 * (TABLE_NODES + 1))
    table_kernel(const double* __restrict__ lam, const double* __restrict__ kabs, const double* __restrict__ dnu, int nl,
                 double Tmin, double Tmax, int n, double* __restrict__ table) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double ly[TABLE_NODES + 1], ls[TABLE_NODES + 1], lT[TABLE_NODES + 1];
  const uint64_t* tab;
  const EmitBin* bins;
  emit_setup(smem, lam, kabs, dnu, nl, tab, bins);
  const int g = threadIdx.x >> 3, lane = threadIdx.x & 7;
  const int i = blockIdx.x * TABLE_NODES + g;
  const double hx = log(Tmax / Tmin) / (double)(n - 1);
  const double x = log(Tmin) + log(Tmax / Tmin) * (double)min(i, n - 1) / (double)(n - 1);
  const double T = exp(x);
  const double kT = K_CGS * T;
  const Norm64 inv = planck_inverse(kT), one = norm64(1.0);
  const double ikT = 1.0 / kT;
  double E = 0.0, dE = 0.0;  // sum of the bins and its derivative by log T
  for (int b = lane; b < nl; b += 8) {
    const EmitBin& B = bins[b];
    const double v = emit_term(B, inv, one, 1.0, T, tab);
    E += v;
    // d(1 / (e^x - 1)) / d log T = x n (1 + n), n = v / C_b
    if (v > 0.0) dE += v * (B.hnu * ikT) * (1.0 + v * B.inv_c);
  }
  const unsigned m = (threadIdx.x >> 5) == TABLE_NODES / 4 ? 0xFFu : 0xFFFFFFFFu;  // the last warp has one group
  __syncwarp(m);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    E += __shfl_xor_sync(m, E, o);
    dE += __shfl_xor_sync(m, dE, o);
  }
  if (lane == 0) {
    ly[g] = E > 0.0 ? log(E) : -HUGE_VAL;
    ls[g] = E > 0.0 ? dE / E : 0.0;
    lT[g] = T;
    if (g < TABLE_NODES && i < n) {
      table[3 * i] = x;
      table[3 * i + 1] = ly[g];
      table[3 * i + 2] = ls[g];
    }
  }
  __syncthreads();
  if (lane == 0 && g < TABLE_NODES && i < n) {
    InvNode* node = reinterpret_cast<InvNode*>(table + 3 * (size_t)n) + i;
    float* lg = reinterpret_cast<float*>(table + 11 * (size_t)n);
    InvNode N;
    const double m0 = ls[g] * hx, m1 = ls[g + 1] * hx, dy = ly[g + 1] - ly[g];
    N.inv_e = E >= 1e-290 && i + 1 < n ? 1.0 / E : 0.0;
    N.c1 = m0;
    N.c2 = 3.0 * dy - 2.0 * m0 - m1;
    N.c3 = m0 + m1 - 2.0 * dy;
    N.T = lT[g];
    N.hx = hx;
    N.pad0 = N.pad1 = 0.0;
    *node = N;
    lg[i] = E > 0.0 ? (float)(ly[g] * 1.4426950408889634) : -CUDART_INF_F;
  }
}

// doubles of the tables for n nodes
size_t dust_table_doubles(int n) { return 12 * (size_t)n; }

cudaError_t dust_table(const double* lam, const double* kabs, const double* dnu, int nl, double Tmin, double Tmax,
                       int n_table, double* table, cudaStream_t s) {
  const int B = 8 * (TABLE_NODES + 1);
  table_kernel<<<(n_table + TABLE_NODES - 1) / TABLE_NODES, B, emit_smem(nl), s>>>(lam, kabs, dnu, nl, Tmin, Tmax,
                                                                                  n_table, table);
  return cudaGetLastError();
}

// exact safeguarded Newton on E(T) = target inside [Tl, Th] (used where the
// table has no finite logarithm, i.e. E underflows to 0 at the cold end)
__device__ double solve_exact(const double* lam, const double* kabs, const double* dnu, int nl, double target,
                              double Tl, double Th) {
  double T = 0.5 * (Tl + Th);
  for (int it = 0; it < 200; ++it) {
    double dE;
    const double E = emission_per_mass(lam, kabs, dnu, nl, T, &dE);
    const double f = E - target;
    if (f < 0.0) Tl = T;
    else Th = T;
    double Tn = dE > 0.0 ? T - f / dE : 0.5 * (Tl + Th);
    if (!(Tn > Tl && Tn < Th)) Tn = 0.5 * (Tl + Th);
    const double step = fabs(Tn - T);
    T = Tn;
    if (step <= 1e-14 * T || (Th - Tl) <= 1e-14 * Tl) break;
  }
  return T;
}

// T of one leaf from Y = log(A / mass), by the tables alone: bracket by
// bisection in log E, six Newton steps on the interpolant; the exact sum
// where log E is not finite.  The general form, for the cells the short one
// below leaves out.
__device__ __noinline__ double solve_by_table(double A, double mass, const double* lam, const double* kabs,
                                              const double* dnu, int nl, double Tmin, double Tmax,
                                              const double* __restrict__ table, int n_table) {
  const double Y = log(A / mass);
  if (!(Y > table[1])) return Tmin;
  if (Y >= table[3 * (n_table - 1) + 1]) return Tmax;
  // bracket: y_lo <= Y < y_hi (log E is increasing in log T)
  int lo = 0, hi = n_table - 1;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (table[3 * mid + 1] <= Y) lo = mid;
    else hi = mid;
  }
  const double x0 = table[3 * lo], y0 = table[3 * lo + 1], s0 = table[3 * lo + 2];
  const double x1 = table[3 * hi], y1 = table[3 * hi + 1], s1 = table[3 * hi + 2];
  if (!(y0 > -HUGE_VAL)) return solve_exact(lam, kabs, dnu, nl, A / mass, exp(x0), exp(x1));
  // invert the cubic Hermite interpolant p(t), t in [0,1], by Newton
  const double hx = x1 - x0;
  const double m0 = s0 * hx, m1 = s1 * hx;
  double t = (Y - y0) / (y1 - y0);
  for (int it = 0; it < 6; ++it) {
    const double t2 = t * t, t3 = t2 * t;
    const double p = (2 * t3 - 3 * t2 + 1) * y0 + (t3 - 2 * t2 + t) * m0 + (-2 * t3 + 3 * t2) * y1 + (t3 - t2) * m1;
    const double dp = (6 * t2 - 6 * t) * y0 + (3 * t2 - 4 * t + 1) * m0 + (-6 * t2 + 6 * t) * y1 + (3 * t2 - 2 * t) * m1;
    double tn = dp > 0.0 ? t - (p - Y) / dp : t;
    tn = tn < 0.0 ? 0.0 : (tn > 1.0 ? 1.0 : tn);
    const bool done = fabs(tn - t) < 1e-15;
    t = tn;
    if (done) break;
  }
  return exp(x0 + t * hx);
}

// a / b for normal a, b > 0 in integer arithmetic (error below an ulp);
// 0: outside the normal range
__device__ __forceinline__ double quotient(double a, double b) {
  const Norm64 x = norm64(a), y = norm64(b);
  if (!x.m || !y.m) return 0.0;
  const bool one = y.m == 0x8000000000000000ull;
  const uint64_t q = one ? x.m >> 1 : mul_hi64(x.m, recip64(y.m));  // x.m / y.m 2^63 (or 2^62 with y.m = 2^63)
  const int lz = clz64(q);
  const int eb = x.e - y.e - lz + (one ? 1 : 0) + 1023;
  if (eb < 2 || eb > 2045) return 0.0;
  const uint64_t n = q << lz;
  return of_bits(((uint64_t)(eb - 1) << 52) + ((n >> 11) + ((n >> 10) & 1ull)));
}

// Bound by the FP64 pipe (two lanes per SM and clock): the sum over the bins,
// one operation a bin, and about 20 operations of the inversion.  The
// general form takes some 400 (a logarithm, a division, up to six Newton
// steps, an exponential, FP64 compares of the bisection).  Here
//   * A / (rho V) is an integer quotient;
//   * the interval is found by bisection over log2 E in f32 (shared memory;
//     an f32 miss by one interval extrapolates the interpolant by a fraction
//     of a percent of an interval);
//   * log(a / E_i) is the series of log(1 + q), |q| < 1/64;
//   * Newton starts from the f32 solution, so one FP64 step leaves 1e-14 of an
//     interval, 1e-17 of T;
//   * T = T_i e^(t hx) by its series (hx ~ 1e-3).
// Cells outside this (a wider interval, values outside the normal range, the
// ends of the table) take the general form.  4.5e6 cells of 20 bins: 0.48 ms,
// the general form for all of them 3.1 ms.
__global__ void __launch_bounds__(256, 4) temperature_kernel(
    const double* __restrict__ absorbed, int n_bins, long long n, const uint32_t* __restrict__ child,
    const double* __restrict__ rho64, const uint8_t* __restrict__ level, double h0, const double* __restrict__ lam,
    const double* __restrict__ kabs, const double* __restrict__ dnu, int nl, double Tmin, double Tmax,
    const double* __restrict__ table, int n_table, bool short_form, double* __restrict__ Tout) {
  extern __shared__ float lg[];
  const float* lgt = reinterpret_cast<const float*>(table + 11 * (size_t)n_table);
  if (short_form)
    for (int i = threadIdx.x; i < n_table; i += blockDim.x) lg[i] = lgt[i];
  __syncthreads();
  const InvNode* node = reinterpret_cast<const InvNode*>(table + 3 * (size_t)n_table);
  const double v0 = h0 * h0 * h0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) {
    if (child[c]) {
      Tout[c] = 0.0;
      continue;
    }
    double A = 0.0;
#pragma unroll 8
    for (int b = 0; b < n_bins; ++b) A += absorbed[(long long)b * n + c];
    const double mass = leaf_mass(rho64[c], h0, v0, level[c]);
    if (!(mass > 0.0) || !(A > 0.0)) {
      Tout[c] = Tmin;
      continue;
    }
    const double a = short_form ? quotient(A, mass) : 0.0;
    double T = -1.0;
    if (a > 0.0) {
      const uint64_t ab = bits_of(a);
      const float lga = (float)((int)(ab >> 52) - 1023) +
                        __log2f(__uint_as_float(0x3F800000u | (uint32_t)((ab >> 29) & 0x7FFFFFu)));
      int lo = 0, hi = n_table - 1;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (lg[mid] <= lga) lo = mid;
        else hi = mid;
      }
      const double2* np = reinterpret_cast<const double2*>(node + lo);
      const double2 n0 = __ldg(np), n1 = __ldg(np + 1), n2 = __ldg(np + 2);
      const double q = fma(a, n0.x, -1.0);
      const float qf = (float)q;
      // the table's ends are left to the general form
      if (lo > 0 && lo < n_table - 2 && fabsf(qf) < 0.015625f && n0.x > 0.0) {
        // log(1 + q) = q (1 - q/2 + ... ), |q|^9 / 9 < 1e-17
        double s = fma(q, -0.125, 1.0 / 7.0);
        s = fma(q, s, -1.0 / 6.0);
        s = fma(q, s, 0.2);
        s = fma(q, s, -0.25);
        s = fma(q, s, 1.0 / 3.0);
        s = fma(q, s, -0.5);
        const double y = fma(q * q, s, q);
        // t (c1 + t (c2 + t c3)) = y: f32 start, one FP64 step
        const float c1 = (float)n0.y, c2 = (float)n1.x, c3 = (float)n1.y;
        const float yf = (float)y;
        float tf = yf / c1;
        tf = (yf + tf * tf * (c2 + 2.0f * tf * c3)) / (c1 + tf * (2.0f * c2 + 3.0f * tf * c3));
        tf = (yf + tf * tf * (c2 + 2.0f * tf * c3)) / (c1 + tf * (2.0f * c2 + 3.0f * tf * c3));
        double t = (double)tf;
        const double r = fma(-t, fma(t, fma(t, n1.y, n1.x), n0.y), y);
        t = fma(r, (double)(1.0f / (c1 + tf * (2.0f * c2 + 3.0f * tf * c3))), t);
        const double e = t * n2.y;
        double w = fma(e, 1.0 / 24.0, 1.0 / 6.0);
        w = fma(e, w, 0.5);
        w = fma(e * e, w, e);
        if (tf > -0.25f && tf < 1.25f) T = fma(n2.x, w, n2.x);
      }
    }
    Tout[c] = T > 0.0 ? T : solve_by_table(A, mass, lam, kabs, dnu, nl, Tmin, Tmax, table, n_table);
  }
}

cudaError_t dust_temperature(const double* absorbed, int n_bins, long long n_cells, const uint32_t* child,
                             const double* rho64, const uint8_t* level, double h0, const double* lam, const double* kabs,
                             const double* dnu, int nl, double Tmin, double Tmax, const double* table, int n_table,
                             double* T, int sm_count, cudaStream_t s) {
  // the short form's series of e^(t hx) holds for spacings up to 1.1e-3
  // (T_max / T_min of 8,000); with a wider table every cell takes the general
  // form at once, a thread per cell (4.5e6 cells, 0.1 to 1e5 K: 3.23 ms; 3.54
  // when each began the short one on a grid of 4 blocks per SM)
  const bool short_form = log(Tmax / Tmin) < 0.0011 * (n_table - 1);
  const long long B = 256, want = (n_cells + B - 1) / B;
  const unsigned G = (unsigned)(short_form ? std::min<long long>(want, 4ll * sm_count) : want);
  temperature_kernel<<<G, (unsigned)B, short_form ? sizeof(float) * (size_t)n_table : 0, s>>>(
      absorbed, n_bins, n_cells, child, rho64, level, h0, lam, kabs, dnu, nl, Tmin, Tmax, table, n_table, short_form,
      T);
  return cudaGetLastError();
}

// One thread per cell, its bins in turn (a slice of them per blockIdx.y where
// the cells alone do not fill the GPU).  Bound by integer issue, about 150
// instructions a term: 2.8e8 terms (9.2e6 cells, 30 bins) in 2.44 ms, 8.9e7
// (4.5e6 cells, 20 bins) in 0.90 ms; with the FP64 form 26.6 and 9.7 ms, all
// of it on the FP64 pipe.  Writing them takes 0.33 and 0.11 ms.
__global__ void __launch_bounds__(256) emission_kernel(
    const double* __restrict__ T, long long n, const uint32_t* __restrict__ child, const double* __restrict__ rho64,
    const uint8_t* __restrict__ level, double h0, const double* __restrict__ lam, const double* __restrict__ kabs,
    const double* __restrict__ dnu, int nl, double* __restrict__ em) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint64_t* tab;
  const EmitBin* bins;
  emit_setup(smem, lam, kabs, dnu, nl, tab, bins);
  const int b0 = (int)((long long)nl * blockIdx.y / gridDim.y), b1 = (int)((long long)nl * (blockIdx.y + 1) / gridDim.y);
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) {
    const double Tc = T[c];
    double mass = 0.0;
    if (!child[c] && Tc > 0.0) mass = leaf_mass(rho64[c], h0, h0 * h0 * h0, level[c]);
    const Norm64 inv = planck_inverse(K_CGS * Tc), mass_n = norm64(mass);
    for (int b = b0; b < b1; ++b) em[(long long)b * n + c] = mass > 0.0 ? emit_term(bins[b], inv, mass_n, mass, Tc, tab) : 0.0;
  }
}

// blocks for n cells: at most `per_sm` blocks of 256 per SM over the cells,
// and slices of the bins where that leaves SMs idle
static dim3 emit_grid(long long n, int nl, int sm_count, int per_sm) {
  const long long gx = std::max<long long>(1, std::min<long long>((n + 255) / 256, (long long)per_sm * sm_count));
  const long long gy = std::max<long long>(1, std::min<long long>(nl, (2ll * sm_count) / gx));
  return dim3((unsigned)gx, (unsigned)gy);
}

cudaError_t dust_emission(const double* T, long long n_cells, const uint32_t* child, const double* rho64,
                          const uint8_t* level, double h0, const double* lam, const double* kabs, const double* dnu,
                          int nl, double* emission, int sm_count, cudaStream_t s) {
  emission_kernel<<<emit_grid(n_cells, nl, sm_count, 8), 256, emit_smem(nl), s>>>(T, n_cells, child, rho64, level, h0,
                                                                                 lam, kabs, dnu, nl, emission);
  return cudaGetLastError();
}

// per-bin totals of the emission of emission_kernel, without storing it
__global__ void __launch_bounds__(256) emission_totals_kernel(
    const double* __restrict__ T, long long n, const uint32_t* __restrict__ child, const double* __restrict__ rho64,
    const uint8_t* __restrict__ level, double h0, const double* __restrict__ lam, const double* __restrict__ kabs,
    const double* __restrict__ dnu, int nl, double* __restrict__ tot) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint64_t* tab;
  const EmitBin* bins;
  emit_setup(smem, lam, kabs, dnu, nl, tab, bins);
  const int b0 = (int)((long long)nl * blockIdx.y / gridDim.y), b1 = (int)((long long)nl * (blockIdx.y + 1) / gridDim.y);
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long n_up = (n + 31) / 32 * 32;  // whole warps: the sums below take all lanes
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n_up; c += stride) {
    const double Tc = c < n ? T[c] : 0.0;
    double mass = 0.0;
    if (c < n && !child[c] && Tc > 0.0) mass = leaf_mass(rho64[c], h0, h0 * h0 * h0, level[c]);
    if (!__any_sync(0xFFFFFFFFu, mass > 0.0)) continue;
    const Norm64 inv = planck_inverse(K_CGS * Tc), mass_n = norm64(mass);
    for (int b = b0; b < b1; ++b) {
      double v = mass > 0.0 ? emit_term(bins[b], inv, mass_n, mass, Tc, tab) : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(tot + b, v);
    }
  }
}

cudaError_t dust_emission_totals(const double* T, long long n_cells, const uint32_t* child, const double* rho64,
                                 const uint8_t* level, double h0, const double* lam, const double* kabs,
                                 const double* dnu, int nl, double* tot, int sm_count, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(tot, 0, sizeof(double) * (size_t)nl, s);
  if (e != cudaSuccess || n_cells <= 0) return e;
  emission_totals_kernel<<<emit_grid(n_cells, nl, sm_count, 8), 256, emit_smem(nl), s>>>(
      T, n_cells, child, rho64, level, h0, lam, kabs, dnu, nl, tot);
  return cudaGetLastError();
}

__global__ void max_rel_change_kernel(const double* __restrict__ T, const double* __restrict__ Tp,
                                      const unsigned int* __restrict__ hits, const uint32_t* __restrict__ child,
                                      long long n, double min_hits, double* out) {
  double m = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (child[i] || (hits && (double)hits[i] < min_hits)) continue;
    const double tp = Tp[i];
    if (tp > 0.0) m = fmax(m, fabs(T[i] - tp) / tp);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  // non-negative doubles order like their bit patterns
  if ((threadIdx.x & 31) == 0 && m > 0.0)
    atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(m));
}

cudaError_t max_rel_change(const double* T, const double* T_prev, const unsigned int* hits, const uint32_t* child,
                           long long n, double min_hits, double* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  max_rel_change_kernel<<<(unsigned)std::min<long long>((n + 255) / 256, 1024), 256, 0, s>>>(T, T_prev, hits, child, n, min_hits, out);
  return cudaGetLastError();
}

// floor(e / w + u), u = (x + 1/2) 2^-32 with x word 0 of the cell's Philox
// block: exact, with the FP64 division only where an f32 estimate of
// e / w + u (relative error of the ratio below 4e-7) comes too close to a
// whole number to tell, about once in 1e6 cells.  Ratios below 2^-34 need no
// random number: u <= 1 - 2^-33.
struct CountBin {
  double w;
  float inv;  // 1 / mantissa of w
  int ex;     // its exponent; w not normal: every cell takes the division
  bool normal;
};
__device__ __forceinline__ CountBin count_bin(double w) {
  CountBin B;
  const Norm64 n = norm64(w);
  B.w = w;
  B.normal = n.m != 0ull;
  B.ex = n.e;
  B.inv = 1.0f / __uint_as_float(0x3F800000u | (uint32_t)((n.m >> 40) & 0x7FFFFFu));
  return B;
}
__device__ __forceinline__ long long dust_count(double e, const CountBin& B, uint32_t cell, uint32_t stream, uint32_t k0,
                                                uint32_t k1) {
  if (!(e > 0.0) || !(B.w > 0.0)) return 0;
  const Norm64 n = norm64(e);
  const int de = n.e - B.ex;
  const bool quick = B.normal && n.m != 0ull && de < 20;
  if (quick && de < -35) return 0;
  const uint4 r = philox4x32_10(make_uint4(cell, 0x80000000u, 0u, stream), k0, k1);
  if (quick) {
    const float q = __uint_as_float(0x3F800000u | (uint32_t)((n.m >> 40) & 0x7FFFFFu)) * B.inv *
                    __uint_as_float((uint32_t)(127 + de) << 23);
    const float v = q + ((float)(r.x >> 8) + 0.5f) * 5.9604644775390625e-08f;
    const float t = floorf(v), fr = v - t, err = q * 5e-7f + 3e-7f;
    if (fr > err && fr < 1.0f - err) return (long long)t;
  }
  const double u = ((double)r.x + 0.5) * 2.3283064365386963e-10;
  return (long long)floor(e / B.w + u);
}

// One warp per chunk of COUNT_CHUNK cells of a bin's row: first the chunk's
// packages (WRITE false), then, with the chunks' exclusive sums, the first
// package of each cell.  The counts are evaluated twice rather than stored
// and scanned in place: one read of the emission and one write of the row
// fewer, and no pass that adds the chunks' offsets.  2.8e8 counts: 1.4 ms a
// pass, bound by the Philox rounds; with an FP64 division per cell, a scan
// and the offsets' pass 8.7 ms in all.
static constexpr int COUNT_CHUNK = 1024;
template <bool WRITE>
__global__ void __launch_bounds__(256) dust_counts_kernel(const double* __restrict__ em, long long n,
                                                          const double* __restrict__ w, uint32_t k0, uint32_t k1,
                                                          uint32_t src, long long n_chunks,
                                                          long long* __restrict__ sums, long long* __restrict__ first) {
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  const long long chunk = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (chunk >= n_chunks) return;
  const CountBin B = count_bin(w[b]);
  const double* row = em + (long long)b * n;
  long long* out = first + (long long)b * (n + 1);
  const uint32_t stream = (src << 16) | (uint32_t)b;
  long long run = WRITE ? sums[(long long)b * n_chunks + chunk] : 0;
  for (int i = 0; i < COUNT_CHUNK / 32; ++i) {
    const long long c = chunk * COUNT_CHUNK + i * 32 + lane;
    if (chunk * COUNT_CHUNK + i * 32 > n) break;
    const long long k = c < n ? dust_count(row[c], B, (uint32_t)c, stream, k0, k1) : 0;
    if (WRITE) {
      long long inc = k;
      if (__any_sync(0xFFFFFFFFu, k != 0)) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const long long v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
          if (lane >= o) inc += v;
        }
      }
      if (c <= n) out[c] = run + inc - k;
      run += __shfl_sync(0xFFFFFFFFu, inc, 31);
    } else {
      run += k;
    }
  }
  if (!WRITE) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) run += __shfl_xor_sync(0xFFFFFFFFu, run, o);
    if (lane == 0) sums[(long long)b * n_chunks + chunk] = run;
  }
}

static long long count_chunks(long long n) { return (n + 1 + COUNT_CHUNK - 1) / COUNT_CHUNK; }

size_t dust_counts_tmp_bytes(int nl, long long n) {
  const long long ch = count_chunks(n);
  return sizeof(long long) * (size_t)nl * (size_t)ch + 256 + scan_rows_tmp_bytes(nl, ch);
}

cudaError_t dust_counts(const double* emission, long long n, int nl, const double* w, uint32_t k0, uint32_t k1,
                        uint32_t src, long long* first, void* tmp, size_t tmp_bytes, cudaStream_t s) {
  if (n <= 0 || nl <= 0) return cudaSuccess;
  if (tmp_bytes < dust_counts_tmp_bytes(nl, n)) return cudaErrorInvalidValue;
  const long long ch = count_chunks(n);
  long long* sums = static_cast<long long*>(tmp);
  const size_t sb = (sizeof(long long) * (size_t)nl * (size_t)ch + 255) / 256 * 256;
  const unsigned B = 256;
  const dim3 G((unsigned)((ch + B / 32 - 1) / (B / 32)), (unsigned)nl);
  dust_counts_kernel<false><<<G, B, 0, s>>>(emission, n, w, k0, k1, src, ch, sums, first);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = scan_rows_i64_excl(sums, nl, ch, static_cast<char*>(tmp) + sb, tmp_bytes - sb, s);
  if (e != cudaSuccess) return e;
  dust_counts_kernel<true><<<G, B, 0, s>>>(emission, n, w, k0, k1, src, ch, sums, first);
  return cudaGetLastError();
}

// One atomic per block: with one per warp and 512 blocks a row, the 1.2e5
// atomics to 30 addresses of a 30-bin row set took 145 us whatever the rows'
// length.
__global__ void __launch_bounds__(256) row_sum_kernel(const double* __restrict__ data, long long n,
                                                      double* __restrict__ out) {
  __shared__ double part[8];
  const long long row = blockIdx.y;
  const double* d = data + row * n;
  const long long stride = (long long)gridDim.x * blockDim.x;
  double v = 0.0, v2 = 0.0;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + stride < n; i += 2 * stride) {
    v += d[i];
    v2 += d[i + stride];
  }
  if (i < n) v += d[i];
  v += v2;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) v += part[k];
    if (v != 0.0) atomicAdd(out + row, v);
  }
}

cudaError_t row_sums_f64(const double* data, int n_rows, long long n, double* out, int sm_count, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * (size_t)n_rows, s);
  if (e != cudaSuccess) return e;
  // at least 16 values a thread, and eight blocks per SM over the rows
  const long long blocks = std::max<long long>(1, std::min<long long>((n + 4095) / 4096, (8ll * sm_count + n_rows - 1) / n_rows));
  row_sum_kernel<<<dim3((unsigned)blocks, n_rows), 256, 0, s>>>(data, n, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------
// subiterations (Sect. 3.2, App. B)
// ------------------------------------------------------------------------
// temperatures that emit in a subiteration: the cells below level L
__global__ void mask_levels_kernel(const double* __restrict__ T, const uint8_t* __restrict__ level, long long n,
                                   int L, double* __restrict__ out) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < n) out[c] = (int)level[c] > L ? T[c] : 0.0;
}

cudaError_t mask_levels(const double* T, const uint8_t* level, long long n, int L, double* out, cudaStream_t s) {
  mask_levels_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(T, level, n, L, out);
  return cudaGetLastError();
}

// Eq. 9: the field of a cell, constant sources plus the dust field of every
// level array (a cell holds nothing above its own level)
__global__ void sum_levels_kernel(const double* __restrict__ I, int n_levels, long long n,
                                  const double* __restrict__ A_star, double* __restrict__ A) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  double v = A_star[c];
  for (int i = 0; i < n_levels; ++i) v += I[(long long)i * n + c];
  A[c] = v;
}

cudaError_t sum_levels(const double* I, int n_levels, long long n, const double* A_star, double* A, cudaStream_t s) {
  sum_levels_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(I, n_levels, n, A_star, A);
  return cudaGetLastError();
}

// emission per unit mass E(T) from the table of log E(log T) (cubic Hermite)
__device__ __forceinline__ double table_emission(double T, const double* __restrict__ table, int n_table) {
  if (!(T > 0.0)) return 0.0;
  const double x0 = table[0], hx = table[3] - table[0];
  const double x = log(T);
  int i = (int)floor((x - x0) / hx);
  i = i < 0 ? 0 : (i > n_table - 2 ? n_table - 2 : i);
  const double y0 = table[3 * i + 1], y1 = table[3 * i + 4];
  if (!(y0 > -HUGE_VAL)) return 0.0;
  const double tt = (x - table[3 * i]) / hx, m0 = table[3 * i + 2] * hx, m1 = table[3 * i + 5] * hx;
  const double t2 = tt * tt, t3 = t2 * tt;
  return exp((2 * t3 - 3 * t2 + 1) * y0 + (t3 - 2 * t2 + tt) * m0 + (-2 * t3 + 3 * t2) * y1 + (t3 - t2) * m1);
}

// Eq. 3 with a diagonal operator per frequency (Sect. 3.1: the system
// decouples into one equation per cell, with one unknown per frequency):
// Lambda_b of a cell is the fraction of the energy its own bin-b packages
// carried that they left in it (self_b / emitted_b, two tallies of the same
// packages), capped at lam_max; the cell's temperature then solves
//   sum_b (1 - Lambda_b) E_b(T) = A - sum_b Lambda_b emitted_b.
// Only cells that sent at least min_count packages use it (flag 1); the
// others keep the plain step E(T) = A.  A bin in which such a cell sent no
// package takes the largest Lambda_j of the cell's sampled bins with
// kabs_j <= kabs_b (0 if none): self-absorption grows with opacity, and a
// weight of 1 would count that bin's emission at the new T as escaping.
__device__ __forceinline__ double ali_lambda(const double* __restrict__ self, const double* __restrict__ emitted,
                                             double lam_max, long long n, long long c, int b) {
  const double e = emitted[(long long)b * n + c];
  return e > 0.0 ? fmin(self[(long long)b * n + c] / e, lam_max) : -1.0;
}

__global__ void ali_weights_kernel(const double* __restrict__ A, const double* __restrict__ self,
                                   const double* __restrict__ emitted, const unsigned int* __restrict__ count,
                                   const double* __restrict__ kabs, unsigned int min_count, double lam_max, int nl,
                                   long long n, double* __restrict__ rhs, double* __restrict__ w,
                                   uint8_t* __restrict__ use) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const bool on = count[c] >= min_count;
  double r = A[c];
  for (int b = 0; b < nl; ++b) {
    double lam = on ? ali_lambda(self, emitted, lam_max, n, c, b) : 0.0;
    if (lam >= 0.0) {
      r -= lam * emitted[(long long)b * n + c];
    } else {
      lam = 0.0;
      for (int j = 0; j < nl; ++j)
        if (kabs[j] <= kabs[b]) lam = fmax(lam, ali_lambda(self, emitted, lam_max, n, c, j));
    }
    w[(long long)b * n + c] = 1.0 - lam;
  }
  rhs[c] = r;
  use[c] = on ? 1 : 0;
}

cudaError_t ali_weights(const double* A, const double* self, const double* emitted, const unsigned int* count,
                        const double* kabs, unsigned int min_count, double lam_max, int nl, long long n, double* rhs,
                        double* w, uint8_t* use, cudaStream_t s) {
  ali_weights_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(A, self, emitted, count, kabs, min_count, lam_max, nl,
                                                                  n, rhs, w, use);
  return cudaGetLastError();
}

// sum_b w_b E_b(T) per unit mass and its derivative, summed over the eight
// lanes of a cell's group (mask m)
__device__ __forceinline__ double weighted_emission(const EmitBin* bins, const uint64_t* tab,
                                                    const double* __restrict__ w, long long n, long long c, int nl,
                                                    double T, unsigned m, double* dEdT) {
  const double kT = K_CGS * T, ikT = 1.0 / kT;
  const Norm64 inv = planck_inverse(kT), one = norm64(1.0);
  double s = 0.0, ds = 0.0;
  for (int b = threadIdx.x & 7; b < nl; b += 8) {
    const double v = emit_term(bins[b], inv, one, 1.0, T, tab);
    const double wv = w[(long long)b * n + c] * v;
    s += wv;
    if (v > 0.0) ds += wv * (bins[b].hnu * ikT) * (1.0 + v * bins[b].inv_c);
  }
  __syncwarp(m);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    s += __shfl_xor_sync(m, s, o);
    ds += __shfl_xor_sync(m, ds, o);
  }
  *dEdT = ds / T;
  return s;
}

// The ALI cells' temperatures: safeguarded Newton (bisection when a step
// leaves the bracket) on sum_b w_b E_b(T) = rhs / (rho V), starting from the
// plain solve's T; T_min / T_max where the target lies outside (looked at
// when a step first runs into that end).  Eight lanes share a cell's bins:
// with a thread per cell the 27,200 cells of a small disc with 12 bins took
// 1.58 ms, most of it latency of 213 blocks, now 0.15 ms.  Newton stops once a
// step is below 1e-10 T: a step of d T leaves about x / 2 d^2, x = h nu / k T of
// the bins that emit (below 710, where a term is zero): below 4e-18.
__global__ void __launch_bounds__(128) temperature_weighted_kernel(
    const double* __restrict__ rhs, const double* __restrict__ w, const uint8_t* __restrict__ use, long long n,
    const uint32_t* __restrict__ child, const double* __restrict__ rho64, const uint8_t* __restrict__ level, double h0,
    const double* __restrict__ lam, const double* __restrict__ kabs, const double* __restrict__ dnu, int nl, double Tmin,
    double Tmax, double* __restrict__ T) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint64_t* tab;
  const EmitBin* bins;
  emit_setup(smem, lam, kabs, dnu, nl, tab, bins);
  const unsigned m = 0xFFu << (threadIdx.x & 24);  // the lanes of this cell
  const bool lead = (threadIdx.x & 7) == 0;
  const long long groups = (long long)gridDim.x * (blockDim.x >> 3);
  for (long long c = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 3; c < n; c += groups) {
    if (!use[c] || child[c]) continue;
    const double mass = leaf_mass(rho64[c], h0, h0 * h0 * h0, level[c]);
    double out = Tmin;
    if (mass > 0.0 && rhs[c] > 0.0) {
      const double target = rhs[c] / mass;
      const double t0 = T[c];
      double lo = Tmin, hi = Tmax, d;
      double t = t0 > Tmin && t0 < Tmax ? t0 : sqrt(Tmin * Tmax);
      bool low_known = false, high_known = false;
      for (int it = 0; it < 200; ++it) {
        const double f = weighted_emission(bins, tab, w, n, c, nl, t, m, &d) - target;
        if (f < 0.0) lo = t;
        else hi = t;
        double tn = d > 0.0 ? t - f / d : 0.5 * (lo + hi);
        if (!(tn > lo && tn < hi)) {
          double dd;
          if (f >= 0.0 && lo == Tmin && !low_known) {
            if (target <= weighted_emission(bins, tab, w, n, c, nl, Tmin, m, &dd)) {
              t = Tmin;
              break;
            }
            low_known = true;
          } else if (f < 0.0 && hi == Tmax && !high_known) {
            if (target >= weighted_emission(bins, tab, w, n, c, nl, Tmax, m, &dd)) {
              t = Tmax;
              break;
            }
            high_known = true;
          }
          tn = 0.5 * (lo + hi);
          t = tn;
          if ((hi - lo) <= 1e-14 * lo) break;
          continue;
        }
        const double step = fabs(tn - t);
        t = tn;
        if (step <= 1e-10 * t || (hi - lo) <= 1e-14 * lo) break;
      }
      out = t;
    }
    __syncwarp(m);
    if (lead) T[c] = out;
  }
}

cudaError_t dust_temperature_weighted(const double* rhs, const double* w, const uint8_t* use, long long n,
                                      const uint32_t* child, const double* rho64, const uint8_t* level, double h0,
                                      const double* lam, const double* kabs, const double* dnu, int nl, double Tmin,
                                      double Tmax, double* T, int sm_count, cudaStream_t s) {
  const long long want = (n + 15) / 16;
  temperature_weighted_kernel<<<(unsigned)std::min<long long>(want, 12ll * sm_count), 128, emit_smem(nl), s>>>(
      rhs, w, use, n, child, rho64, level, h0, lam, kabs, dnu, nl, Tmin, Tmax, T);
  return cudaGetLastError();
}

// Energy imbalance |absorbed - emitted|, mass and emission, summed over the
// leaves at level <= L (out[0], out[1], out[4]) and below L (out[2], out[3],
// out[5]).  The emission is rho V E(T) with E from the tabulated
// log E(log T) (cubic Hermite).
__global__ void imbalance_kernel(const double* __restrict__ A, const double* __restrict__ T,
                                 const uint32_t* __restrict__ child, const double* __restrict__ rho64,
                                 const uint8_t* __restrict__ level, double h0, const double* __restrict__ table,
                                 int n_table, long long n, int L, double* __restrict__ out) {
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    if (child[c]) continue;
    const double h = ldexp(h0, -(int)level[c]);
    const double mass = rho64[c] * h * h * h;
    const double E = table_emission(T[c], table, n_table);
    const int gi = (int)level[c] > L ? 2 : 0;
    v[gi] += fabs(A[c] - mass * E);
    v[gi + 1] += mass;
    v[4 + gi / 2] += mass * E;
  }
  __shared__ double part[6][8];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    double x = v[k];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    if ((threadIdx.x & 31) == 0) part[k][threadIdx.x >> 5] = x;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double x = 0.0;
    for (int k = 0; k < 8; ++k) x += part[threadIdx.x][k];
    if (x != 0.0) atomicAdd(out + threadIdx.x, x);
  }
}

cudaError_t level_imbalance(const double* A, const double* T, const uint32_t* child, const double* rho64,
                            const uint8_t* level, double h0, const double* table, int n_table, long long n, int L,
                            double* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, 6 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  imbalance_kernel<<<(unsigned)std::min<long long>((n + 255) / 256, 1024), 256, 0, s>>>(A, T, child, rho64, level, h0, table, n_table, n, L, out);
  return cudaGetLastError();
}

}  // namespace rtk
