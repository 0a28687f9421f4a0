// Device probes of the kernels' own arithmetic for tests/test_gpu_arith.py: the
// two forms of the mixed path's cell inversion side by side, and the short
// reciprocals, roots and quotients beside CUDA's.
#include "mpmc_mixed.cuh"
#include "mpmc_params.h"

using namespace mpmc;

// out: [0] cells that the float-float form takes; [1..6] of these the cells whose
// T, p, rho, Y, u, status differ in a bit from the FP64 form's.  p is that of the
// converged FP64 solve (the FP64 form's stops short with several liquids), T is
// compared where the FP64 form has that p.
template <int NS, int D>
__global__ void k_cells(const __grid_constant__ KParams P, const double* __restrict__ U, long long n,
                        unsigned long long* out) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  constexpr int NV = NS + D + 1;
  ff Uc[NV];
  bool range = true, neg = false;
  for (int v = 0; v < NV; ++v) {
    const double x = U[v * n + c];
    range = range && mx::in_f32(x);
    neg = neg || (v < NS && x < 0.0);
    Uc[v] = ff_of(x);
  }
  mx::CellF<NS> a, b;
  if (!range || neg || !mx::cell_ff<NS, D>(P, Uc, a)) return;
  mx::cell_fp64<NS, D>(P, U + c, n, b);
  double Ud[NV], rho, Y[NS], u[3], e, v, p, T;
  for (int q = 0; q < NV; ++q) Ud[q] = U[q * n + c];
  decode<NS, D>(Ud, rho, Y, u, e, v);
  pt_equilibrium<NS>(P, Y, e, v, p, T);
  auto differ = [](float x, float y) { return __float_as_uint(x) != __float_as_uint(y); };
  bool dY = false, du = false;
  for (int k = 0; k < NS; ++k) dY = dY || differ(a.Y[k], b.Y[k]);
  for (int d = 0; d < D; ++d) du = du || differ(a.u[d], b.u[d]);
  atomicAdd(out, 1ull);
  if (differ(a.T, b.T) && !differ(a.p, b.p)) atomicAdd(out + 1, 1ull);
  if (differ(a.p, narrow(p))) atomicAdd(out + 2, 1ull);
  if (differ(a.rho, b.rho)) atomicAdd(out + 3, 1ull);
  if (dY) atomicAdd(out + 4, 1ull);
  if (du) atomicAdd(out + 5, 1ull);
  if (a.st != b.st) atomicAdd(out + 6, 1ull);
}

extern "C" int probe_cells(const mpmc_grid* g, const mpmc_eos* e, const mpmc_model* m, const double* U, long long n,
                           unsigned long long* out) {
  KParams P;
  if (build_params(g, e, m, P) || n <= 0) return 1;
  const unsigned nb = (unsigned)((n + 127) / 128);
  switch (P.ns * 4 + P.dim) {
    case 2 * 4 + 1: k_cells<2, 1><<<nb, 128>>>(P, U, n, out); break;
    case 3 * 4 + 2: k_cells<3, 2><<<nb, 128>>>(P, U, n, out); break;
    case 4 * 4 + 3: k_cells<4, 3><<<nb, 128>>>(P, U, n, out); break;
    default: return 1;
  }
  return cudaDeviceSynchronize() != cudaSuccess;
}

// |x - y| in units of the last place (same sign, finite)
__device__ unsigned long long ulps(double x, double y) {
  const long long d = __double_as_longlong(x) - __double_as_longlong(y);
  return (unsigned long long)(d < 0 ? -d : d);
}
// out: largest errors of [0] drcp, [1] qdiv against CUDA's division, in ulps;
// [2] drsqrt's in 2^-60 of its value; differences from CUDA's division of ddiv
// [3] with drcp's reciprocal, [4] with a refined one
__global__ void k_div(const double* __restrict__ a, const double* __restrict__ b, long long n,
                      unsigned long long* out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x = a[i], y = b[i], r = drcp(y);
  atomicMax(out, ulps(r, 1.0 / y));
  atomicMax(out + 1, ulps(qdiv(x, y), x / y));
  // z = 1 / sqrt(w) (1 + d): w z^2 - 1 = 2 d + d^2, w z^2 as p z + q z exactly
  const double w = fabs(y), z = drsqrt(w), p = __dmul_rn(w, z), q = __fma_rn(w, z, -p);
  const double d = 0.5 * __fma_rn(q, z, __fma_rn(p, z, -1.0));
  atomicMax(out + 2, (unsigned long long)ceil(fabs(d) * 0x1p60));
  if (ulps(ddiv(x, y, r), x / y)) atomicAdd(out + 3, 1ull);
  const double r2 = fma(fma(-y, r, 1.0), r, r);
  if (ulps(ddiv(x, y, r2), x / y)) atomicAdd(out + 4, 1ull);
}

extern "C" int probe_div(const double* a, const double* b, long long n, unsigned long long* out) {
  if (n <= 0) return 1;
  k_div<<<(unsigned)((n + 255) / 256), 256>>>(a, b, n, out);
  return cudaDeviceSynchronize() != cudaSuccess;
}
