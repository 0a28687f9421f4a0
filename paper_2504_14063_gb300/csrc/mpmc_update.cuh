// Divergence of the face fluxes (Eq. DiscreteGoverningEquations) and the
// SSP-RK combination (Eq. SSPRK3) of one cell, from face fluxes F_d[v][face]
// of type FT: double, or float on the mixed path (every flux enters its two
// cells with the same value, and its cells' sums are FP64's, so that the sum
// over cells telescopes to FP64 rounding).
#pragma once
#include "mpmc_device.cuh"

namespace mpmc {

// fs[v] = sum_d (F_d[m_d] - F_d[p_d]) of every component
template <int NV, int D>
__device__ __forceinline__ void flux_sums(const double* const* Fd, const long long* nf, const long long* fm,
                                          const long long* fp, double* fs) {
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    fs[v] = Fd[0][(long long)v * nf[0] + fm[0]] - Fd[0][(long long)v * nf[0] + fp[0]];
#pragma unroll
    for (int d = 1; d < D; ++d) fs[v] += Fd[d][(long long)v * nf[d] + fm[d]] - Fd[d][(long long)v * nf[d] + fp[d]];
  }
}

// the same of FP32 fluxes: the differences and all but the last two additions
// on the FP32 pipe (ff_diff_sum).  (FP64 differences and sums, on fluxes widened
// by the face pass, were 5 of the update's 8 FP64 operations per component in
// 3D, and twice the flux traffic.  With one FP64 addition, of a pair that holds
// the sum to 2^-47 of the largest difference, a 256^3 step takes 46.2 ms for
// 47.0, but its cells no longer telescope to FP64 rounding.)  Sums beyond FP32's
// normal range take FP64, once all are formed: a branch per component would
// keep the next one's loads back.
template <int NV, int D>
__device__ __forceinline__ void flux_sums(const float* const* Fd, const long long* nf, const long long* fm,
                                          const long long* fp, double* fs) {
  float a[NV][D], b[NV][D];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int d = 0; d < D; ++d) {
      a[v][d] = Fd[d][(long long)v * nf[d] + fm[d]];
      b[v][d] = Fd[d][(long long)v * nf[d] + fp[d]];
    }
  bool ok = true;
#pragma unroll
  for (int v = 0; v < NV; ++v) fs[v] = ff_diff_sum<D>(a[v], b[v], ok);
  if (!ok) {
#pragma unroll 1
    for (int v = 0; v < NV; ++v) {
      double f = (double)Fd[0][(long long)v * nf[0] + fm[0]] - (double)Fd[0][(long long)v * nf[0] + fp[0]];
      for (int d = 1; d < D; ++d)
        f += (double)Fd[d][(long long)v * nf[d] + fm[d]] - (double)Fd[d][(long long)v * nf[d] + fp[d]];
#pragma unroll
      for (int w = 0; w < NV; ++w)
        if (w == v) fs[w] = f;
    }
  }
}

template <int NS, int D, typename FT>
__device__ __forceinline__ void update_cell(const KParams& P, const long long c, const double* __restrict__ Un,
                                            const double* __restrict__ Uk, const FT* __restrict__ F0,
                                            const FT* __restrict__ F1, const FT* __restrict__ F2,
                                            const double* __restrict__ scal, const double rk0, const double rk1,
                                            const double rk2, double* __restrict__ Uout, double* __restrict__ dUdt,
                                            int* __restrict__ status) {
  constexpr int NV = NS + D + 1;
  const int n0 = P.n[0], n1 = P.n[1];
  int ijk[3];
  unflatten(c, n0, n1, ijk);
  const int i = ijk[0], j = ijk[1], k = ijk[2];
  const FT* Fd[3] = {F0, F1, F2};
  long long fm[3], fp[3], nf[3];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int f0 = n0 + (d == 0), f1 = n1 + (d == 1), f2 = P.n[2] + (d == 2);
    nf[d] = (long long)f0 * f1 * f2;
    fm[d] = ((long long)k * f1 + j) * f0 + i;
    fp[d] = fm[d] + (d == 0 ? 1 : (d == 1 ? f0 : (long long)f0 * f1));
  }
  const double dt = scal[0];
  // U = rk0 U^n + rk1 U^(k) + rk2 dt L, L = sum_d (F_{-1/2} - F_{+1/2}) / dx:
  // the flux differences are summed first and scaled once (the FP64 pipe
  // binds this kernel on GB300); a zero coefficient skips its state's load
  const double sdx = (rk2 * dt) * P.inv_dx;
  // the coefficient tests, once per thread as integers (FP64 comparisons
  // issue on the FP64 pipe, and would otherwise be repeated per variable)
  const int keep = dt == 0.0, use_k = rk1 != 0.0, use_n = rk0 != 0.0;
  // (all loads before the first use: a conditional load per component would
  // wait for the one before)
  double Uo[NV], fs[NV], un[NV], uk[NV];
  if (use_n) {
#pragma unroll
    for (int v = 0; v < NV; ++v) un[v] = Un[(long long)v * P.ncell + c];
  }
  if (use_k | keep) {
#pragma unroll
    for (int v = 0; v < NV; ++v) uk[v] = Uk[(long long)v * P.ncell + c];
  }
  flux_sums<NV, D>(Fd, nf, fm, fp, fs);
  if (dUdt) {
#pragma unroll
    for (int v = 0; v < NV; ++v) dUdt[(long long)v * P.ncell + c] = fs[v] * P.inv_dx;
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    double t = sdx * fs[v];
    if (use_k) t = fma(rk1, uk[v], t);
    if (use_n) t = fma(rk0, un[v], t);
    // a zero-length step (a run past its end time) leaves the state as it is
    Uo[v] = keep ? uk[v] : t;
  }
  if (Uout) {
#pragma unroll
    for (int v = 0; v < NV; ++v) Uout[(long long)v * P.ncell + c] = Uo[v];
    if (!admissible_cell<NS, D>(P, Uo)) atomicMax(status, (int)ST_INADMISSIBLE);
  }
}

}  // namespace mpmc
