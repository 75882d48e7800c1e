// Register-resident complex64 product passes for the padded lengths
// 162 = 9 x 18, 168 = 12 x 14, 175 = 7 x 25 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_c(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 162: return fast::run_product_pass<float, 9, 18>(pass, a);
    case 168: return fast::run_product_pass<float, 12, 14>(pass, a);
    case 175: return fast::run_product_pass<float, 7, 25>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
