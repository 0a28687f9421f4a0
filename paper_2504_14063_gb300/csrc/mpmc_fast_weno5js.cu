// Forward FP64 face-pass instantiations with the WENO5-JS interpolation (Sec. 4.1),
// every dimension and species count.
#include "mpmc_fast.cuh"

namespace mpmc {

FaceFn face_fast_weno5js(int dim, int ns) { return fast::face<RC_WENO5JS>(dim, ns); }

}  // namespace mpmc
