// Register-resident complex64 product passes for the padded lengths
// 375 = 15 x 25, 378 = 18 x 21 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_h(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 375: return fast::run_product_pass<float, 15, 25>(pass, a);
    case 378: return fast::run_product_pass<float, 18, 21>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
