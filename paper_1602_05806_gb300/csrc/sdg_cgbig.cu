// Instantiations of the resident CG kernel for large 2D FP32 tiles.
#include "sdg_cgbig.cuh"

namespace sdg {

cudaError_t big_dispatch(const sdg_handle* h, const ResPlan& pl, const ResArgs<float>& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_big<1>(h, pl, a, s);
    case 2: return launch_big<2>(h, pl, a, s);
    case 3: return launch_big<3>(h, pl, a, s);
    case 4: return launch_big<4>(h, pl, a, s);
    case 5: return launch_big<5>(h, pl, a, s);
    case 6: return launch_big<6>(h, pl, a, s);
    case 7: return launch_big<7>(h, pl, a, s);
    case 8: return launch_big<8>(h, pl, a, s);
    case 9: return launch_big<9>(h, pl, a, s);
    case 10: return launch_big<10>(h, pl, a, s);
    case 11: return launch_big<11>(h, pl, a, s);
    case 12: return launch_big<12>(h, pl, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sdg
