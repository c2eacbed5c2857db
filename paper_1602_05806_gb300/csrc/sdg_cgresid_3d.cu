// Instantiations of the resident solve's residual replacement for dim = 3.
#include "sdg_cgresid.cuh"

namespace sdg {

cudaError_t resid_dispatch_3d(const sdg_handle* h, const ResPlan& pl, const ResidArgs& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_resid_t<3, 1>(h, pl, a, s);
    case 2: return launch_resid_t<3, 2>(h, pl, a, s);
    case 3: return launch_resid_t<3, 3>(h, pl, a, s);
    case 4: return launch_resid_t<3, 4>(h, pl, a, s);
    case 5: return launch_resid_t<3, 5>(h, pl, a, s);
    case 6: return launch_resid_t<3, 6>(h, pl, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sdg
