// Forward FP64 face-pass instantiations with the TENO5 interpolation (Sec. 4.1),
// every dimension and species count.
#include "mpmc_fast.cuh"

namespace mpmc {

FaceFn face_fast_teno5(int dim, int ns) { return fast::face<RC_TENO5>(dim, ns); }

}  // namespace mpmc
