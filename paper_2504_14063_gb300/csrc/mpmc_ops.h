// Internal launch table of the MPMC kernels: one entry per (species count,
// dimension) instantiation.  Not part of the public C ABI.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mpmc {

struct KParams;

// Threads per block of a pass over n cells or faces that takes `most` on large
// grids.  Blocks of one warp spread a small grid over more SMs, each with an
// FP64 pipe of its own, and leave a smaller last wave: slab of 400 cells, 20
// steps 2.24 -> 2.03 ms, reverse step of a 201 x 103 box 3.30 -> 2.38 ms,
// 301 x 203 right-hand side 240 -> 219 us.  Beyond eight full blocks per SM the
// waves are many and full blocks share more of their stencils in L1: 512 x 512
// adjoint faces 9.1 ms (9.9 with one warp), 256^3 mixed faces 36.7 (38.5).
inline int block_threads(long long n, int most) { return n < 152ll * 8 * most ? 32 : most; }
inline unsigned nblocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

struct Ops {
  void (*init)(const KParams&, cudaStream_t, const double* prim, double* U, long long n);
  void (*prim)(const KParams&, cudaStream_t, const double* U, const double* Uin, double* Wc,
               unsigned long long* red, int* status);
  void (*face)(const KParams&, cudaStream_t, int d, const double* Wc, const double* Un, const double* Uk,
               const double* Uin, const double* scal, double rk0, double rk1, double rk2, double* F,
               uint32_t* flags, unsigned long long* stats);
  void (*update)(const KParams&, cudaStream_t, const double* Un, const double* Uk, double* const* F,
                 const double* scal, double rk0, double rk1, double rk2, double* Uout, double* dUdt, int* status);
  // ghost states of the characteristic boundaries of U into its ghost buffer
  // G (FP64 on both paths; nothing to do without such boundaries)
  void (*ghost)(const KParams&, cudaStream_t, const double* U, double* G);
};

// discrete adjoint (FP64): per-face contributions of one direction into a
// slot buffer, their per-cell gather, the per-cell primitive-recovery VJP
// fused with the reverse RK combination, and the VJP of the initialisation
struct AdjOps {
  int (*slots)(const KParams&);
  void (*face)(const KParams&, cudaStream_t, int d, const double* Wc, const double* Uk, const double* Uin,
               const double* scal, const uint32_t* tape, const double* lamL, double coef, int mul_dt, double* C);
  // the viscous stress and conduction flux of the same faces, reversed (adds
  // to the slots the face pass wrote)
  void (*face_visc)(const KParams&, cudaStream_t, int d, const double* Wc, const double* scal,
                    const uint32_t* tape, const double* lamL, double coef, int mul_dt, double* C);
  void (*gather)(const KParams&, cudaStream_t, int d, const double* C, int first, double* gW, double* gU);
  // Wc (nullable): U's primitive cache, whose T and P the reverse takes
  // instead of solving the p-T equilibrium again
  void (*cell)(const KParams&, cudaStream_t, const double* U, const double* Wc, const double* gW, const double* gU,
               double* out, double a, const double* x, double b, const double* y, double cz, const double* z);
  void (*init)(const KParams&, cudaStream_t, const double* prim, const double* lamU, double* lprim, long long n);
};

using FaceFn = decltype(Ops::face);
using PrimFn = decltype(Ops::prim);
// FP64 face passes with Sec. 4.1's other ENO-type interpolations, for
// (dimension, species count), null if none: defined in
// mpmc_recon_{weno5js,teno5,teno6}.cu
FaceFn face_fp64_weno5js(int dim, int ns);
FaceFn face_fp64_teno5(int dim, int ns);
FaceFn face_fp64_teno6(int dim, int ns);
// forward FP64 primitive and face passes (parts in float-float), the ones that
// steps and right-hand sides run: mpmc_fast_d{1,2,3}.cu,
// mpmc_fast_{weno5js,teno5,teno6}.cu
PrimFn prim_fast_d1(int ns);
PrimFn prim_fast_d2(int ns);
PrimFn prim_fast_d3(int ns);
FaceFn face_fast_d1(int ns);
FaceFn face_fast_d2(int ns);
FaceFn face_fast_d3(int ns);
FaceFn face_fast_weno5js(int dim, int ns);
FaceFn face_fast_teno5(int dim, int ns);
FaceFn face_fast_teno6(int dim, int ns);
// the same for mixed-precision contexts: mpmc_mixed_recon_{weno5js,teno5,teno6}.cu
FaceFn face_mixed_weno5js(int dim, int ns);
FaceFn face_mixed_teno5(int dim, int ns);
FaceFn face_mixed_teno6(int dim, int ns);

using AdjFaceFn = decltype(AdjOps::face);
// adjoint face passes with Sec. 4.1's other interpolations:
// mpmc_adjoint_recon_{weno5js,teno5,teno6}.cu
AdjFaceFn adj_face_weno5js(int dim, int ns);
AdjFaceFn adj_face_teno5(int dim, int ns);
AdjFaceFn adj_face_teno6(int dim, int ns);

inline PrimFn prim_fast(int dim, int ns) {
  return dim == 1 ? prim_fast_d1(ns) : (dim == 2 ? prim_fast_d2(ns) : prim_fast_d3(ns));
}
inline FaceFn face_fast_weno5z(int dim, int ns) {
  return dim == 1 ? face_fast_d1(ns) : (dim == 2 ? face_fast_d2(ns) : face_fast_d3(ns));
}

// per-dimension tables, defined in mpmc_kernels_d{1,2,3}.cu (FP64) and
// mpmc_mixed_d{1,2,3}.cu (mixed precision; init is the FP64 one)
Ops ops_fp64_d1(int ns);
Ops ops_fp64_d2(int ns);
Ops ops_fp64_d3(int ns);
Ops ops_mixed_d1(int ns);
Ops ops_mixed_d2(int ns);
Ops ops_mixed_d3(int ns);
// defined in mpmc_adjoint_d{1,2,3}.cu
AdjOps adj_ops_d1(int ns);
AdjOps adj_ops_d2(int ns);
AdjOps adj_ops_d3(int ns);

}  // namespace mpmc
