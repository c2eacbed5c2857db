// Instantiations of the line-wise stage kernels for dim = 2.
#include "sdg_lines.cuh"

namespace sdg {

cudaError_t pair_dispatch_2d(const sdg_handle* h, const PairArgs& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_pair<2, 1>(h, a, s);
    case 2: return launch_pair<2, 2>(h, a, s);
    case 3: return launch_pair<2, 3>(h, a, s);
    case 4: return launch_pair<2, 4>(h, a, s);
    case 5: return launch_pair<2, 5>(h, a, s);
    case 6: return launch_pair<2, 6>(h, a, s);
    case 7: return launch_pair<2, 7>(h, a, s);
    case 8: return launch_pair<2, 8>(h, a, s);
    case 9: return launch_pair<2, 9>(h, a, s);
    case 10: return launch_pair<2, 10>(h, a, s);
    case 11: return launch_pair<2, 11>(h, a, s);
    case 12: return launch_pair<2, 12>(h, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t div_dispatch_2d(const sdg_handle* h, const DivArgs& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_div<2, 1>(h, a, s);
    case 2: return launch_div<2, 2>(h, a, s);
    case 3: return launch_div<2, 3>(h, a, s);
    case 4: return launch_div<2, 4>(h, a, s);
    case 5: return launch_div<2, 5>(h, a, s);
    case 6: return launch_div<2, 6>(h, a, s);
    case 7: return launch_div<2, 7>(h, a, s);
    case 8: return launch_div<2, 8>(h, a, s);
    case 9: return launch_div<2, 9>(h, a, s);
    case 10: return launch_div<2, 10>(h, a, s);
    case 11: return launch_div<2, 11>(h, a, s);
    case 12: return launch_div<2, 12>(h, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t conv_dispatch_2d(const sdg_handle* h, const ConvArgs& a, cudaStream_t s) {
  switch (h->g.n1) {
    case 1: return launch_conv<2, 1>(h, a, s);
    case 2: return launch_conv<2, 2>(h, a, s);
    case 3: return launch_conv<2, 3>(h, a, s);
    case 4: return launch_conv<2, 4>(h, a, s);
    case 5: return launch_conv<2, 5>(h, a, s);
    case 6: return launch_conv<2, 6>(h, a, s);
    case 7: return launch_conv<2, 7>(h, a, s);
    case 8: return launch_conv<2, 8>(h, a, s);
    case 9: return launch_conv<2, 9>(h, a, s);
    case 10: return launch_conv<2, 10>(h, a, s);
    case 11: return launch_conv<2, 11>(h, a, s);
    case 12: return launch_conv<2, 12>(h, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sdg
