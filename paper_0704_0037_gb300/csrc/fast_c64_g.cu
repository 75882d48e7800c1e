// Register-resident complex64 product passes for the padded lengths
// 336 = 16 x 21, 350 = 14 x 25, 360 = 18 x 20 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_g(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 336: return fast::run_product_pass<float, 16, 21>(pass, a);
    case 350: return fast::run_product_pass<float, 14, 25>(pass, a);
    case 360: return fast::run_product_pass<float, 18, 20>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
