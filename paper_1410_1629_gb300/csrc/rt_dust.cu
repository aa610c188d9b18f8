// Panchromatic mode (SKIRT paper, Sect. 2.1 and 2.2): the equilibrium
// temperature of the dust in every cell from the luminosity it absorbed over
// the wavelength grid, the dust's thermal emission per cell and wavelength,
// and the running sums over the cells from which the transport kernel draws
// the emitting cell of a dust-emission packet.
//
//   emission of cell c at temperature T: S m_c sum_l w_l beta_l(T), with
//   m_c = rho_c V_c, w_l = kappa_l (1 - albedo_l) dlambda_l (the host's
//   per-wavelength weights, S folded in), beta_l(T) = lambda_l^-5 /
//   (exp(C2 / (lambda_l T)) - 1), lambda in um, C2 = hc/k in um K.
//   The temperature solves emission = absorbed luminosity in ln T between
//   ln t_min and ln t_max (Newton steps kept in a bisection bracket: a
//   single-precision estimate, then double precision to 1e-15); no absorption or
//   no dust: 0; short of the absorption at t_max: t_max, beyond it at t_min:
//   t_min (both counted).
// All of it is FP64, whose pipe bounds it (88 % busy, memory at 3 % of its
// rate, when every cell was solved by itself): so E(T), the emission per unit
// mass, is one function for all cells of a launch and its inverse is tabulated
// once per call and looked up per cell, and the thermal emission uses the
// library's own a / (exp(x) - 1) (rt_math.cuh).  192 x 192 x 128 cells, 24
// wavelengths: temperatures 44.9 ms, emission and running sums 10.3 ms; now 7.0
// ms together with the read-out (56.0 before).
#include <algorithm>
#include <cmath>

#include "rt_internal.h"
#include "rt_math.cuh"

namespace rtk {

namespace {

constexpr double kC2 = 14387.768775039337;  // hc / k in um K

struct DustArgs {
  int n_lambda, nx, ny, nz;
  long long n_cells;
  int stride[3];          // storage strides of the absorption tallies
  const double* planes;   // FP64 cell planes: x [nx + 1], y [ny + 1], z [nz + 1]
  const float* density;   // row-major
  double a[kMaxLambda];   // S kabs_l dlambda_l / lambda_l^5
  double b[kMaxLambda];   // C2 / lambda_l
  float af[kMaxLambda];   // a_l / max a_l
  float bf[kMaxLambda];   // b_l
  double ln_a_max;
};

__device__ __forceinline__ double cell_mass(const DustArgs& A, long long c, int& ix, int& iy, int& iz) {
  ix = (int)(c % A.nx);
  iy = (int)((c / A.nx) % A.ny);
  iz = (int)(c / ((long long)A.nx * A.ny));
  const double* px = A.planes;
  const double* py = A.planes + A.nx + 1;
  const double* pz = py + A.ny + 1;
  const double V = (px[ix + 1] - px[ix]) * (py[iy + 1] - py[iy]) * (pz[iz + 1] - pz[iz]);
  return (double)A.density[c] * V;
}

// Emission per unit mass at T, sum_l a_l / (exp(b_l / T) - 1), and its
// derivative with respect to ln T; Real is double, or float with the a_l
// scaled by 1 / max a_l (a first estimate of the root only).
template <class Real>
__device__ __forceinline__ Real emission(int n, const Real* a, const Real* b, Real T, Real* d_dlnT = nullptr) {
  Real sum = 0, der = 0;
  for (int l = 0; l < n; ++l) {
    const Real x = b[l] / T;
    const Real em1 = expm1(x);
    const Real t = a[l] / em1;
    sum += t;
    if (d_dlnT) der += t * x * (Real(1) + Real(1) / em1);
  }
  if (d_dlnT) *d_dlnT = der;
  return sum;
}

// Root of ln E(exp(u)) = target in u within [lo, hi]: Newton steps, replaced by
// the bracket's midpoint where they leave it, until a step (or the bracket)
// is below tol relative to max(1, |u|).
template <class Real>
__device__ __forceinline__ Real solve_ln_t(int n, const Real* a, const Real* b, Real target, Real lo, Real hi,
                                           Real u, Real tol, int max_it) {
  for (int it = 0; it < max_it; ++it) {
    Real der;
    const Real e = emission(n, a, b, exp(u), &der);
    const Real f = log(e) - target;
    if (f < Real(0)) lo = u; else hi = u;
    const Real un = u - f * e / der;
    const Real scale = fmax(Real(1), fabs(u));
    if (fabs(un - u) <= tol * scale) return un;
    u = un >= lo && un <= hi ? un : Real(0.5) * (lo + hi);
    if (hi - lo <= tol * scale) break;
  }
  return u;
}

// The temperature at which the emission per unit mass is x, within [t_min,
// t_max]: the root of ln E(T) = ln x in ln T, a single-precision estimate to
// 1e-6, then double-precision steps to 1e-15 (the root the oracle's bisection
// converges to).
__device__ __forceinline__ double solve_temperature(const DustArgs& A, double x, double t_min, double t_max) {
  const double lo = log(t_min), hi = log(t_max);
  const double target = log(x);
  const float u32 = solve_ln_t<float>(A.n_lambda, A.af, A.bf, (float)(target - A.ln_a_max), (float)lo, (float)hi,
                                      (float)(0.5 * (lo + hi)), 1e-6f, 60);
  const double u0 = (double)u32 > lo && (double)u32 < hi ? (double)u32 : 0.5 * (lo + hi);
  return exp(solve_ln_t<double>(A.n_lambda, A.a, A.b, target, lo, hi, u0, 1e-15, 200));
}

// ---- the tabulated inverse
//
// T(x) for x = E(T) on intervals of 1/16 of a binary octave: x in 2^e [1 + j/16, 1
// + (j + 1)/16), found from the bits of x.  On each, T - T_mid as a Chebyshev
// series of degree 8 in s in [-1, 1]: the half width is at most 1/32 of x, T(x)
// is analytic well beyond it where the wavelengths are dense (its nearest
// singularities lie a distance of order 1 away in ln x), so the coefficients fall
// by about 60 per degree and the series ends below 1e-16 of T.  Where they fall
// more slowly (two wavelengths far apart) the row is marked by a negative T_mid
// and its values take one Newton step on E itself, or it is not used: a row
// that does not fall fast enough for the step, on which a node had no root, or an
// x beyond the table (E(t_min) to E(t_max), at most kTableOctaves down from the
// top) is solved by itself.  How far the series has fallen is judged by its last
// three coefficients, those before the last at 64 and 64^2 of it (kTableFall):
// where two terms of E meet, the coefficients change sign from degree to degree
// and the last alone can vanish while the series is far from its end (by the last
// alone 2e-7 of T on such a row).
constexpr int kTableNodes = 9, kTableRow = 10;  // T_mid and nine coefficients
constexpr double kTableFall = 1.0 / 64.0;

// Row i of the table from its nodes' roots (one thread per node, solved as a
// cell would be over a wider range, then one Newton step in T itself, whose
// error is E's rounding over the slope); first: (e << 4 | j) of row 0.
constexpr int kRowsPerBlock = 28;
__global__ void __launch_bounds__(kRowsPerBlock * kTableNodes) k_dust_table(const DustArgs A, double t_min, double t_max,
                                                                            int first, int rows,
                                                                            double* __restrict__ table,
                                                                            double* __restrict__ limits) {
  __shared__ double T[kRowsPerBlock][kTableNodes], C[kRowsPerBlock][kTableNodes];
  const int r = threadIdx.x / kTableNodes, j = threadIdx.x % kTableNodes;
  const int row = blockIdx.x * kRowsPerBlock + r;
  if (row < rows) {
    const int key = first + row;
    const double half = ldexp(1.0, (key >> 4) - 5);
    const double x = ldexp(1.0 + ((key & 15) + 0.5) / 16.0, key >> 4) + half * cospi((j + 0.5) / kTableNodes);
    double t = solve_temperature(A, x, 0.25 * t_min, 4.0 * t_max);
    double der;
    const double e = emission(A.n_lambda, A.a, A.b, t, &der);
    t -= t * ((e - x) / der);
    T[r][j] = t > 0.3 * t_min && t < 3.5 * t_max ? t : nan("");
  }
  __syncthreads();
  if (row < rows) {
    const double mid = T[r][kTableNodes / 2];
    double c = 0.0;
    for (int i = 0; i < kTableNodes; ++i) c += (T[r][i] - mid) * cospi(j * (i + 0.5) / kTableNodes);
    double* out = table + (size_t)row * kTableRow;
    c *= (j ? 2.0 : 1.0) / kTableNodes;
    out[1 + j] = c;
    C[r][j] = fabs(c);  // not a number on all degrees if a node had no root
  }
  __syncthreads();
  if (row < rows && j == 0) {
    const double mid = T[r][kTableNodes / 2];
    const double* c = &C[r][kTableNodes - 3];
    const double left = fmax(fmax(c[0] * kTableFall, c[1]) * kTableFall, c[2]);
    table[(size_t)row * kTableRow] = left <= 4e-16 * mid ? mid : (left <= 1e-9 * mid ? -mid : nan(""));
  }
  if (blockIdx.x == 0 && threadIdx.x < 2) limits[threadIdx.x] = emission(A.n_lambda, A.a, A.b, threadIdx.x ? t_max : t_min);
}

// T(x) from the table; refine: the value needs a Newton step.
__device__ __forceinline__ double look_up(const double* __restrict__ table, int first, int rows, double x,
                                          bool& refine) {
  refine = false;
  const long long b = bits_of(x);
  const int row = (int)(b >> 48) - (1023 << 4) - first;
  if ((unsigned)row >= (unsigned)rows) return nan("");
  const double2* c = reinterpret_cast<const double2*>(table + (size_t)row * kTableRow);
  const double2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2), c3 = __ldg(c + 3), c4 = __ldg(c + 4);
  // s: the lower 48 bits of x as a number in [1, 2), less 3/2, doubled
  const double s2 = 4.0 * double_of((b << 4 & 0xfffffffffffffll) | 0x3ff0000000000000ll) - 6.0;  // 2 s
  // Clenshaw's recurrence; c0.x is T_mid, c0.y the constant term
  double p = c4.y, q = fma(s2, p, c4.x), t;
  t = fma(s2, q, c3.y) - p; p = q; q = t;
  t = fma(s2, q, c3.x) - p; p = q; q = t;
  t = fma(s2, q, c2.y) - p; p = q; q = t;
  t = fma(s2, q, c2.x) - p; p = q; q = t;
  t = fma(s2, q, c1.y) - p; p = q; q = t;
  t = fma(s2, q, c1.x) - p; p = q; q = t;
  refine = c0.x < 0.0;
  return fabs(c0.x) + (fma(0.5 * s2, q, c0.y) - p);
}

// absorbed: row-major [n_lambda][n_cells] (a caller's field) or, when
// stored is set, the context's tallies in storage order.  table: the inverse
// (limits: E at t_min and t_max), or null: every cell is solved by itself.
__global__ void k_dust_temperature(const DustArgs A, const double* __restrict__ absorbed, int stored,
                                   double t_min, double t_max, const double* __restrict__ table, int first, int rows,
                                   const double* __restrict__ limits, double* __restrict__ T, unsigned* clamped) {
  const double e_max = table ? limits[1] : emission(A.n_lambda, A.a, A.b, t_max);
  const double e_min = table ? limits[0] : emission(A.n_lambda, A.a, A.b, t_min);
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < A.n_cells;
       c += (long long)gridDim.x * blockDim.x) {
    int ix, iy, iz;
    const double m = cell_mass(A, c, ix, iy, iz);
    const long long slot = stored ? (long long)ix * A.stride[0] + (long long)iy * A.stride[1] +
                                        (long long)iz * A.stride[2]
                                  : c;
    double ab = 0.0;
    // eight loads in flight; summed in wavelength order
    int l = 0;
    for (; l + 8 <= A.n_lambda; l += 8) {
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = absorbed[(size_t)(l + i) * A.n_cells + slot];
#pragma unroll
      for (int i = 0; i < 8; ++i) ab += v[i];
    }
    for (; l < A.n_lambda; ++l) ab += absorbed[(size_t)l * A.n_cells + slot];
    const double top = m * e_max;
    if (!(ab > 0.0) || !(m > 0.0) || !(top > 0.0)) {
      T[c] = 0.0;
      continue;
    }
    if (top < ab) {
      T[c] = t_max;
      atomicAdd(clamped, 1u);
      continue;
    }
    if (m * e_min >= ab) {
      T[c] = t_min;
      atomicAdd(clamped, 1u);
      continue;
    }
    const double x = ab / m;
    bool refine = false;
    double t = table ? look_up(table, first, rows, x, refine) : nan("");
    if (!(t > 0.0)) {
      t = solve_temperature(A, x, t_min, t_max);
    } else if (refine) {
      double der;
      const double e = emission(A.n_lambda, A.a, A.b, t, &der);
      t -= t * ((e - x) / der);
    }
    T[c] = fmin(fmax(t, t_min), t_max);
  }
}

// lum[l][c] = m_c w_l beta_l(T_c) (T = 0: none), row-major cells; a thread takes
// a cell through all wavelengths (its mass and 1 / T once).
__global__ void k_dust_luminosity(const DustArgs A, const double* __restrict__ T, double* __restrict__ lum) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < A.n_cells;
       c += (long long)gridDim.x * blockDim.x) {
    int ix, iy, iz;
    const double m = cell_mass(A, c, ix, iy, iz);
    const double t = T[c];
    const bool warm = t > 0.0;
    const double inv = warm ? 1.0 / t : 0.0;
    for (int l = 0; l < A.n_lambda; ++l) {
      // b / t to its last bit: the product with 1 / t and its remainder (not
      // a number where x or t is infinite: x is then 0 or infinite already)
      const double b = A.b[l];
      double x = b * inv;
      const double rem = fma(-x, t, b);
      if ((bits_of(rem) >> 52 & 0x7ff) != 0x7ff) x = fma(rem, inv, x);
      lum[(size_t)l * A.n_cells + c] = warm ? m * bose(x, A.a[l]) : 0.0;
    }
  }
}

// ---- inclusive running sums over the cells, per wavelength (blockIdx.y):
// tile totals, their exclusive scan, then each tile's scan plus its offset.
constexpr int kTile = 4096;  // 256 threads x 16 values

__device__ __forceinline__ double block_exclusive(double v, double* warp_tot, double& total) {
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  double incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (unsigned)o) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const double w = lane < (blockDim.x >> 5) ? warp_tot[lane] : 0.0;
    double wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= (unsigned)o) wi += t;
    }
    if (lane < (blockDim.x >> 5)) warp_tot[lane] = wi - w;
    if (lane == (blockDim.x >> 5) - 1) warp_tot[32] = wi;
  }
  __syncthreads();
  total = warp_tot[32];
  const double ex = warp_tot[warp] + incl - v;
  __syncthreads();
  return ex;
}

__global__ void __launch_bounds__(256) k_tile_sums(const double* __restrict__ x, long long n, double* tile_sum,
                                                   long long n_tiles) {
  __shared__ double warp_tot[33];
  const double* row = x + (size_t)blockIdx.y * n;
  const long long base = (long long)blockIdx.x * kTile + threadIdx.x * 16ll;
  double s = 0.0;
  for (int j = 0; j < 16; ++j)
    if (base + j < n) s += row[base + j];
  double total;
  block_exclusive(s, warp_tot, total);
  if (threadIdx.x == 0) tile_sum[(size_t)blockIdx.y * n_tiles + blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_scan_tile_sums(double* ts, long long n_tiles) {
  __shared__ double warp_tot[33];
  __shared__ double carry;
  double* row = ts + (size_t)blockIdx.x * n_tiles;
  if (threadIdx.x == 0) carry = 0.0;
  __syncthreads();
  for (long long b = 0; b < n_tiles; b += blockDim.x) {
    const long long i = b + threadIdx.x;
    const double v = i < n_tiles ? row[i] : 0.0;
    double total;
    const double ex = block_exclusive(v, warp_tot, total);
    const double c0 = carry;
    if (i < n_tiles) row[i] = c0 + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry = c0 + total;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(256) k_tile_scan(const double* __restrict__ x, double* __restrict__ sums, long long n,
                                                   const double* tile_off, long long n_tiles) {
  __shared__ double warp_tot[33];
  const double* row = x + (size_t)blockIdx.y * n;
  double* out = sums + (size_t)blockIdx.y * n;
  const long long base = (long long)blockIdx.x * kTile + threadIdx.x * 16ll;
  double v[16];
  double s = 0.0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    v[j] = base + j < n ? row[base + j] : 0.0;
    s += v[j];
  }
  double total;
  double run = tile_off[(size_t)blockIdx.y * n_tiles + blockIdx.x] + block_exclusive(s, warp_tot, total);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    run += v[j];
    if (base + j < n) out[base + j] = run;
  }
}

DustArgs make_args(int n_lambda, int nx, int ny, int nz, const int stride[3], const double* planes,
                   const float* density, const double* w, const double* lambda) {
  DustArgs A;
  A.n_lambda = n_lambda;
  A.nx = nx; A.ny = ny; A.nz = nz;
  A.n_cells = (long long)nx * ny * nz;
  for (int a = 0; a < 3; ++a) A.stride[a] = stride[a];
  A.planes = planes;
  A.density = density;
  double a_max = 0.0;
  for (int l = 0; l < kMaxLambda; ++l) {
    const double lam = l < n_lambda ? lambda[l] : 1.0;
    A.a[l] = l < n_lambda ? w[l] / (lam * lam * lam * lam * lam) : 0.0;
    A.b[l] = kC2 / lam;
    a_max = A.a[l] > a_max ? A.a[l] : a_max;
  }
  if (!(a_max > 0.0)) a_max = 1.0;
  A.ln_a_max = std::log(a_max);
  for (int l = 0; l < kMaxLambda; ++l) {
    A.af[l] = (float)(A.a[l] / a_max);
    A.bf[l] = (float)A.b[l];
  }
  return A;
}

unsigned cell_blocks(long long n) { return (unsigned)((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192); }

// Emission per unit mass on the host (the table's extent only).
double host_emission(const DustArgs& A, double T) {
  double sum = 0.0;
  for (int l = 0; l < A.n_lambda; ++l) sum += A.a[l] / std::expm1(A.b[l] / T);
  return sum;
}

constexpr int kTableOctaves = 192;
// Cells from which the table pays: those of one wave of direct solves (a block of
// 256 on each of 152 SMs, the FP64 pipe's share of each).  Up to there both take
// the time of one root (484 us for 32768 cells by the table, 487 us solved by
// themselves; 24 wavelengths, 4 to 60 K), and from there on the direct solves
// take a second wave (46656 cells 495 against 868 us, 64000 cells 497 against 872
// us).
constexpr long long kTableCells = 152 * 256;

}  // namespace

size_t dust_table_bytes() { return ((size_t)(kTableOctaves + 1) * 16 * kTableRow + 2) * sizeof(double); }

cudaError_t launch_dust_temperature(int n_lambda, int nx, int ny, int nz, const int stride[3], const double* planes,
                                    const float* density, const double* w, const double* lambda,
                                    const double* absorbed, int stored, double t_min, double t_max, double* table,
                                    double* T, unsigned* clamped, cudaStream_t s) {
  const DustArgs A = make_args(n_lambda, nx, ny, nz, stride, planes, density, w, lambda);
  const double top = host_emission(A, t_max), bottom = host_emission(A, t_min);
  int first = 0, rows = 0;
  if (A.n_cells >= kTableCells && std::isnormal(top)) {
    const int e1 = std::ilogb(top);
    const int e0 = std::isnormal(bottom) ? std::max(std::ilogb(bottom), e1 - kTableOctaves + 1) : e1 - kTableOctaves + 1;
    first = std::max(e0, -1000) * 16;
    rows = (e1 + 1) * 16 - first;
  }
  double* limits = table;
  double* const body = rows > 0 ? table + 2 : nullptr;
  if (rows > 0) {
    k_dust_table<<<(unsigned)((rows + kRowsPerBlock - 1) / kRowsPerBlock), kRowsPerBlock * kTableNodes, 0, s>>>(
        A, t_min, t_max, first, rows, body, limits);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  k_dust_temperature<<<cell_blocks(A.n_cells), 256, 0, s>>>(A, absorbed, stored, t_min, t_max, body, first, rows, limits,
                                                            T, clamped);
  return cudaGetLastError();
}

cudaError_t launch_dust_emission(int n_lambda, int nx, int ny, int nz, const int stride[3], const double* planes,
                                 const float* density, const double* w, const double* lambda, const double* T,
                                 double* lum, double* cum, double* tile_sum, cudaStream_t s) {
  const DustArgs A = make_args(n_lambda, nx, ny, nz, stride, planes, density, w, lambda);
  const long long n = A.n_cells;
  k_dust_luminosity<<<cell_blocks(n), 256, 0, s>>>(A, T, lum);
  const long long n_tiles = (n + kTile - 1) / kTile;
  k_tile_sums<<<dim3((unsigned)n_tiles, (unsigned)n_lambda), 256, 0, s>>>(lum, n, tile_sum, n_tiles);
  k_scan_tile_sums<<<(unsigned)n_lambda, 1024, 0, s>>>(tile_sum, n_tiles);
  k_tile_scan<<<dim3((unsigned)n_tiles, (unsigned)n_lambda), 256, 0, s>>>(lum, cum, n, tile_sum, n_tiles);
  return cudaGetLastError();
}

long long dust_tiles(long long n_cells) { return (n_cells + kTile - 1) / kTile; }

}  // namespace rtk
