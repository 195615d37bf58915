// agcm_diag.cuh — FP64 global sums (a11): mass, kinetic, available potential
// and available surface potential energy, max |U|, max |V|, non-finite count.
// Deterministic: fixed grid, rows of a warp in a fixed order, fixed-order tree
// reductions, one final block.
#pragma once
#include "agcm_common.cuh"

namespace agcm {

constexpr int kDiagPartials = 608;  // four blocks per SM on a 152-SM part
constexpr int kDiagThreads = 256;

__device__ __forceinline__ void diag_reduce_block(double v[7], double* part) {
  __shared__ double red[7][kDiagThreads];
  for (int q = 0; q < 7; ++q) red[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = kDiagThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int q = 0; q < 7; ++q) {
        const double a = red[q][threadIdx.x], b = red[q][threadIdx.x + w];
        red[q][threadIdx.x] = (q == 4 || q == 5) ? fmax(a, b) : a + b;
      }
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 7; ++q) part[q] = red[q][0];
}

// Sum of squares, largest magnitude and count of non-finite values of a row
// (a lane's share).  FP32: GB300 issues FP64 at 1/64 of the FP32 rate (the
// sums alone took 1.26 ms at 1440x720x30, where reading the state takes 55
// us), so squares are split exactly by a multiply-add and added in three FP32
// terms (Sum3), which drops nothing above 2^-60 of the sum; a row whose
// largest magnitude lets squares or their parts leave the FP32 range is done
// in FP64.
template <class T>
struct RowSums {
  double sq;
  T big;
  int bad;
};
__device__ __forceinline__ RowSums<double> diag_row(const double* __restrict__ x, int I, int lane) {
  RowSums<double> r{0.0, 0.0, 0};
  for (int i = lane; i < I; i += 32) {
    const double v = x[i];
    r.sq += v * v;
    // magnitudes of numbers order as their bits
    const long long b = __double_as_longlong(v) & 0x7fffffffffffffffLL;
    if (b <= 0x7ff0000000000000LL && b > __double_as_longlong(r.big)) r.big = __longlong_as_double(b);
    r.bad += b >= 0x7ff0000000000000LL;
  }
  return r;
}
__device__ __forceinline__ RowSums<float> diag_row(const float* __restrict__ x, int I, int lane) {
  RowSums<float> r{0.0, 0.f, 0};
  Sum3 a;
  auto one = [&](float v) {
    const float p = __fmul_rn(v, v);
    a.add(p);
    a.add_low(fmaf(v, v, -p));
    r.big = fmaxf(r.big, fabsf(v));
    r.bad += !(fabsf(v) < __int_as_float(0x7f800000));
  };
  if (I % 4 == 0 && ((uintptr_t)x & 15) == 0) {
    const float4* __restrict__ q = reinterpret_cast<const float4*>(x);
#pragma unroll 4
    for (int i = lane; i < I / 4; i += 32) {
      const float4 v = q[i];
      one(v.x);
      one(v.y);
      one(v.z);
      one(v.w);
    }
  } else {
#pragma unroll 4
    for (int i = lane; i < I; i += 32) one(x[i]);
  }
  r.sq = a.total();
  float m = r.big;
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const bool out = (m != 0.f && !(m > 2e-12f && m < 1e15f)) || __any_sync(0xffffffffu, r.bad);
  if (out) {
    r.sq = 0.0;
    for (int i = lane; i < I; i += 32) r.sq += (double)x[i] * (double)x[i];
  }
  return r;
}

// A warp takes rows in a fixed order (fields U, Phi, V, then pi), so the sums
// do not depend on the order in which warps run.  197 us at 1440x720x30 FP32.
template <class T>
__global__ void __launch_bounds__(kDiagThreads) k_diag(Geom<double> g, const T* __restrict__ U,
                                                       const T* __restrict__ V, const T* __restrict__ Phi,
                                                       const T* __restrict__ pi, double* __restrict__ part) {
  const int I = g.I, J = g.J, K = g.K;
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long nU = (long long)K * J, nV = (long long)K * (J - 1);
  double v[7] = {0, 0, 0, 0, 0, 0, 0};  // mass, ek, ep, eps, max|U|, max|V|, nonfinite
  T maxU = 0, maxV = 0;
  int bad = 0;
  for (long long it = warp; it < 2 * nU + nV; it += nwarps) {
    const bool isV = it >= 2 * nU;
    const int row = (int)(isV ? it - 2 * nU : (it >= nU ? it - nU : it));
    const int JJ = isV ? J - 1 : J, k = row / JJ, j = row - k * JJ;
    const T* const F = isV ? V : (it >= nU ? Phi : U);
    const RowSums<T> r = diag_row(F + (size_t)row * I, I, lane);
    v[it >= nU && !isV ? 2 : 1] += 0.5 * g.dsd[k] * (isV ? g.Avd[j] : g.Ad[j]) * r.sq;
    if (isV)
      maxV = r.big > maxV ? r.big : maxV;
    else if (it < nU)
      maxU = r.big > maxU ? r.big : maxU;
    bad += r.bad;
  }
  for (long long j = warp; j < J; j += nwarps) {
    const double A = g.Ad[j];
    for (int i = lane; i < I; i += 32) {
      const size_t n = (size_t)j * I + i;
      const double p = (double)pi[n];
      v[0] += A * (g.pit[n] + p);
      v[3] += 0.5 * A * g.rt0pit[n] * p * p;
      bad += !isfinite(pi[n]);
    }
  }
  v[4] = (double)maxU;
  v[5] = (double)maxV;
  v[6] = (double)bad;
  diag_reduce_block(v, part + 8 * blockIdx.x);
}

__global__ void __launch_bounds__(kDiagThreads) k_diag_final(const double* __restrict__ part, int nb,
                                                             double* __restrict__ out) {
  double v[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
    for (int q = 0; q < 7; ++q) v[q] = (q == 4 || q == 5) ? fmax(v[q], part[8 * b + q]) : v[q] + part[8 * b + q];
  diag_reduce_block(v, out);
}

}  // namespace agcm
