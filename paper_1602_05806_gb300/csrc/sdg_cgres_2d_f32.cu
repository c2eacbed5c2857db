// Instantiations of the resident CG kernel for dim = 2, float.
#include "sdg_cgres.cuh"

namespace sdg {

cudaError_t res_dispatch_2d(const sdg_handle* h, const ResPlan& pl, const ResArgs<float>& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_res_t<float, 2, 1>(h, pl, a, s);
    case 2: return launch_res_t<float, 2, 2>(h, pl, a, s);
    case 3: return launch_res_t<float, 2, 3>(h, pl, a, s);
    case 4: return launch_res_t<float, 2, 4>(h, pl, a, s);
    case 5: return launch_res_t<float, 2, 5>(h, pl, a, s);
    case 6: return launch_res_t<float, 2, 6>(h, pl, a, s);
    case 7: return launch_res_t<float, 2, 7>(h, pl, a, s);
    case 8: return launch_res_t<float, 2, 8>(h, pl, a, s);
    case 9: return launch_res_t<float, 2, 9>(h, pl, a, s);
    case 10: return launch_res_t<float, 2, 10>(h, pl, a, s);
    case 11: return launch_res_t<float, 2, 11>(h, pl, a, s);
    case 12: return launch_res_t<float, 2, 12>(h, pl, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sdg
