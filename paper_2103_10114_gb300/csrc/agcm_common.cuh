// agcm_common.cuh — device-side geometry and indexing shared by the kernels.
//
// Grid conventions (pole-free C grid): scalar/U rows j = 0..J-1 at colatitude
// (j+1/2) dth, V rows j = 0..J-2 at (j+1) dth, U index i at longitude
// (i+1/2) dlam.  Storage [k][j][i], longitude contiguous.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace agcm {

// Stride classes of single rows (all strides 1, 3, 5, 7; any): the order of a
// small grid's items and its launches.
constexpr int kRowCls = 5;

// Per-grid tables on the device, in the arithmetic type T of the kernels.
// Built once per (grid, precision) by the host from the FP64 geometry.
template <class T>
struct Geom {
  int I, J, K;
  // scalar / U rows (J)
  const int* Mu;    // leap stride M_j (odd), Eq. 6 / Eq. 7
  const T* rdx;     // 1 / (a sin(theta_j) M_j dlam): leap zonal difference
  const T* rdy;     // 1 / (a sin(theta_j) dth): meridional divergence
  const T* zf;      // a dth / M_j: zonal face length over the leap stride
  const T* r2A;     // 1 / (2 A_j)
  const T* f0;      // 2 Omega cos(theta_j)
  const T* cota;    // cot(theta_j) / a
  // V rows (J-1)
  const int* Mv;    // leap stride of the V rows
  const T* sv;      // sin(theta^v_j)
  const T* yv;      // a dlam sin(theta^v_j): meridional face length
  const T* zfv;     // a dth / Mv_j
  const T* r2Av;    // 1 / (2 Av_j)
  const T* cn;      // A_j / (4 Av_j)   Coriolis weight of the northern U row
  const T* cs;      // A_{j+1} / (4 Av_j) Coriolis weight of the southern U row
  // levels
  const T* ds;      // dsigma_k (K)
  const T* r2ds;    // 1 / (2 dsigma_k) (K)
  // hydrostatic weights times the level coefficient beta_k = (1 - delta_p)
  // (1 + delta_c) b_k of Eq. 1 (b_k = sqrt(kappa R T~(sigma_k))):
  const T* hk;      // beta_k ln(sh_{k+1}/sh_k), the off-diagonal weight; hk[0] = 0 (K)
  const T* Hkk;     // beta_k ln(sh_{k+1}/sigma_k), the diagonal (K)
  const T* hk_rds;  // hk / dsigma_k (K)
  const T* rho;     // beta2 / beta_k: the delta kappa Phi/P part of the coefficient (K)
  const T* oms;     // 1 - sigma_hat_k (K): W_k = SD_k - (1 - sigma_hat_k) C
  // the row-segment kernel's tables: kLevN values a level (kLev...), kRowTabN
  // values a row (kRt...); in FP64 z_j / A_j and edge_units of V edge j-1 (J x 2)
  const T* lev;
  const T* rowtab;
  const double* rAz;
  // rows the low-latitude filter changes, entry 4 j + band (1 two-grid, 2 3-point)
  const int* filtU; // scalar / U rows
  const int* filtV; // V rows
  int nfU, nfV;
  const double* dsd;  // dsigma_k in FP64 (column integral of the divergence)
  const float4* ds3;  // dsigma_k as the sum of three FP32 parts x + y + z (K)
  const double* Ad;   // A_j in FP64 (J)     (diagnostics)
  const double* Avd;  // Av_j in FP64 (J-1)  (diagnostics)
  // columns (J*I)
  const T* rt0pit;  // R T~_s / pi~
  const T* pit;     // pi~: standard surface pressure / p0 under phi_s
  int nl;           // 1: the delta kappa Phi/P term is on (beta2 != 0)
  int l1lo, l1hi;   // rows [l1lo, l1hi): interior rows whose strides Mu_j, Mv_j, Mu_{j+1} are all 1
  T rady;           // 1 / (a dth)
  // work items of the row-segment stage kernel (agcm_row.cuh), longest first:
  // chunks of the rows left to the column body, pairs of rows of equal strides,
  // single rows; kind q's items are items[off[q]] .. items[off[q] + cnt[q]],
  // the single rows' stride classes start at cls[c]
  const int4* items;
  int off[3], cnt[3], cls[kRowCls + 1], nitems;
  int rowT;  // threads of a CTA that holds every item
  int column;  // 1: the column kernel unless the row kernel is asked for
};

// Values per level of Geom::lev: dsigma, 4 beta Hkk, 4 beta hk, 2 beta hk /
// dsigma, 1 / dsigma, sigma_hat (the level's upper half level), rho, 2 beta Hkk.
enum { kLevDs, kLevH4, kLevh4, kLevhr2, kLevRds, kLevSh, kLevRho, kLevH2, kLevN };

// Values per row of Geom::rowtab, lengths in units of the row's z = a dth / Mu_j,
// each formed in FP64 and rounded once: z / (2 A_j), z / (2 Av_j); the V edges'
// lengths a dlam sin(theta^v) of V rows j, j-1; A_j f0, A_j cot(theta) / a; Av_j /
// A_j, Av_j / A_{j+1}.  Then, for a row of any strides, of its southern neighbour
// in the same units: V row j+1's length, z of row j+1, A_{j+1} f0, A_{j+1}
// cot(theta) / a.  Zero where there is no such row.
enum { kRtPh, kRtV, kRtYv, kRtYn, kRtAf, kRtAc, kRtRvn, kRtRvs, kRtOwn, kRtYs = kRtOwn, kRtZs, kRtAfs, kRtAcs, kRowTabN };
struct RowTab {
  double v[kRowTabN];
};
// Row j's values from FP64 tables: A and Av, sv = sin(theta^v), c = cos(theta), cot
// = cot(theta); adlam, adth = a dlam, a dth; om2 = 2 Omega; ra = 1 / a.
__host__ __device__ inline RowTab row_tab(int j, int J, double adlam, double adth, double om2, double ra, const double* A,
                                          const double* sv, const double* Av, const double* c, const double* cot,
                                          const int* Mu) {
  RowTab t{};
  const double z = adth / Mu[j];
  t.v[kRtPh] = 0.5 * z / A[j];
  t.v[kRtAf] = A[j] * (om2 * c[j]) / z;
  t.v[kRtAc] = A[j] * (cot[j] * ra) / z;
  if (j > 0) t.v[kRtYn] = adlam * sv[j - 1] / z;
  if (j < J - 1) {
    t.v[kRtV] = 0.5 * z / Av[j];
    t.v[kRtYv] = adlam * sv[j] / z;
    t.v[kRtRvn] = Av[j] / A[j];
    t.v[kRtRvs] = Av[j] / A[j + 1];
    t.v[kRtZs] = (double)Mu[j] / Mu[j + 1];
    t.v[kRtAfs] = A[j + 1] * (om2 * c[j + 1]) / z;
    t.v[kRtAcs] = A[j + 1] * (cot[j + 1] * ra) / z;
  }
  if (j < J - 2) t.v[kRtYs] = adlam * sv[j + 1] / z;
  return t;
}

__device__ __forceinline__ int wrapi(int i, int I) {
  return i < 0 ? i + I : (i >= I ? i - I : i);
}

template <class T>
__device__ __forceinline__ T ldg(const T* p) {
  return __ldg(p);
}

// sqrt in the kernel's type
__device__ __forceinline__ double sqrt_t(double x) { return sqrt(x); }
__device__ __forceinline__ float sqrt_t(float x) { return sqrtf(x); }

// The length of V edge e = j or j - 1 as row j's column integrals take it: a
// dlam sin(theta^v) in units of the row's z = a dth / Mu_j, rounded to T; on a row
// left to the column body (cols), sin(theta^v) and 1 / (a sin(theta) dth) rounded
// to T, times the cell's area.
template <class T>
__host__ __device__ inline double edge_length(bool cols, double sv, double A, double s, double z, double a, double dlam,
                                              double dth) {
  return cols ? A * ((double)(T)sv * (double)(T)(1.0 / (a * s * dth))) : z * (double)(T)(a * dlam * sv / z);
}
// What the row above makes of an edge over what the row below does, less 1.
// Without it the mass that crosses an edge between rows of different strides
// changes by some 3e-8 of itself: 1.4e-10 of the total in 500 steps of
// 1440x720x30 FP32, 4e-12 with it.
__host__ __device__ inline double edge_units(double above, double below) { return above / below - 1.0; }

// a + b = s + e exactly (TwoSum, Knuth), and a sum of FP32 numbers in three
// FP32 terms.  Products that go in are formed by __fmul_rn: a multiply-add
// made of one of these additions would not be exact.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
struct Sum3 {
  float s = 0.f, c = 0.f, d = 0.f;
  __device__ __forceinline__ void add(float x) {
    float e, f;
    two_sum(s, x, s, e);
    two_sum(c, e, c, f);
    d += f;
  }
  __device__ __forceinline__ void add_low(float x) {  // x below 2^-20 of the sum
    float f;
    two_sum(c, x, c, f);
    d += f;
  }
  __device__ __forceinline__ double total() const { return (double)s + ((double)c + (double)d); }
};

}  // namespace agcm
