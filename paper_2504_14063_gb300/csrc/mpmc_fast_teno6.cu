// Forward FP64 face-pass instantiations with the TENO6 interpolation (Sec. 4.1),
// every dimension and species count.
#include "mpmc_fast.cuh"

namespace mpmc {

FaceFn face_fast_teno6(int dim, int ns) { return fast::face<RC_TENO6>(dim, ns); }

}  // namespace mpmc
