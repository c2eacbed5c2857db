// Instantiations of the resident CG kernel for dim = 3, float.
#include "sdg_cgres.cuh"

namespace sdg {

cudaError_t res_dispatch_3d(const sdg_handle* h, const ResPlan& pl, const ResArgs<float>& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_res_t<float, 3, 1>(h, pl, a, s);
    case 2: return launch_res_t<float, 3, 2>(h, pl, a, s);
    case 3: return launch_res_t<float, 3, 3>(h, pl, a, s);
    case 4: return launch_res_t<float, 3, 4>(h, pl, a, s);
    case 5: return launch_res_t<float, 3, 5>(h, pl, a, s);
    case 6: return launch_res_t<float, 3, 6>(h, pl, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sdg
