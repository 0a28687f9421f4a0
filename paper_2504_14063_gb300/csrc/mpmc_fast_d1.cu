// Forward FP64 primitive- and face-pass instantiations (WENO5-Z) for dimension 1, species counts 1..4.
#include "mpmc_fast.cuh"

namespace mpmc {

FaceFn face_fast_d1(int ns) {
  switch (ns) {
    case 1: return &fast::FaceImpl<1, 1, RC_WENO5Z>::face;
    case 2: return &fast::FaceImpl<2, 1, RC_WENO5Z>::face;
    case 3: return &fast::FaceImpl<3, 1, RC_WENO5Z>::face;
    case 4: return &fast::FaceImpl<4, 1, RC_WENO5Z>::face;
    default: return nullptr;
  }
}

PrimFn prim_fast_d1(int ns) {
  switch (ns) {
    case 1: return &fast::prim<1, 1>;
    case 2: return &fast::prim<2, 1>;
    case 3: return &fast::prim<3, 1>;
    case 4: return &fast::prim<4, 1>;
    default: return nullptr;
  }
}

}  // namespace mpmc
