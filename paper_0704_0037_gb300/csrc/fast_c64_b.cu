// Register-resident complex64 product passes for the padded lengths
// 147 = 7 x 21, 150 = 10 x 15, 160 = 10 x 16 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_b(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 147: return fast::run_product_pass<float, 7, 21>(pass, a);
    case 150: return fast::run_product_pass<float, 10, 15>(pass, a);
    case 160: return fast::run_product_pass<float, 10, 16>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
