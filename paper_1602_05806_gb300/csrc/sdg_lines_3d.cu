// Instantiations of the line-wise stage kernels for dim = 3.
#include "sdg_lines.cuh"

namespace sdg {

cudaError_t pair_dispatch_3d(const sdg_handle* h, const PairArgs& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_pair<3, 1>(h, a, s);
    case 2: return launch_pair<3, 2>(h, a, s);
    case 3: return launch_pair<3, 3>(h, a, s);
    case 4: return launch_pair<3, 4>(h, a, s);
    case 5: return launch_pair<3, 5>(h, a, s);
    case 6: return launch_pair<3, 6>(h, a, s);
    case 7: return launch_pair<3, 7>(h, a, s);
    case 8: return launch_pair<3, 8>(h, a, s);
    case 9: return launch_pair<3, 9>(h, a, s);
    case 10: return launch_pair<3, 10>(h, a, s);
    case 11: return launch_pair<3, 11>(h, a, s);
    case 12: return launch_pair<3, 12>(h, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t div_dispatch_3d(const sdg_handle* h, const DivArgs& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_div<3, 1>(h, a, s);
    case 2: return launch_div<3, 2>(h, a, s);
    case 3: return launch_div<3, 3>(h, a, s);
    case 4: return launch_div<3, 4>(h, a, s);
    case 5: return launch_div<3, 5>(h, a, s);
    case 6: return launch_div<3, 6>(h, a, s);
    case 7: return launch_div<3, 7>(h, a, s);
    case 8: return launch_div<3, 8>(h, a, s);
    case 9: return launch_div<3, 9>(h, a, s);
    case 10: return launch_div<3, 10>(h, a, s);
    case 11: return launch_div<3, 11>(h, a, s);
    case 12: return launch_div<3, 12>(h, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t conv_dispatch_3d(const sdg_handle* h, const ConvArgs& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_conv<3, 1>(h, a, s);
    case 2: return launch_conv<3, 2>(h, a, s);
    case 3: return launch_conv<3, 3>(h, a, s);
    case 4: return launch_conv<3, 4>(h, a, s);
    case 5: return launch_conv<3, 5>(h, a, s);
    case 6: return launch_conv<3, 6>(h, a, s);
    case 7: return launch_conv<3, 7>(h, a, s);
    case 8: return launch_conv<3, 8>(h, a, s);
    case 9: return launch_conv<3, 9>(h, a, s);
    case 10: return launch_conv<3, 10>(h, a, s);
    case 11: return launch_conv<3, 11>(h, a, s);
    case 12: return launch_conv<3, 12>(h, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sdg
