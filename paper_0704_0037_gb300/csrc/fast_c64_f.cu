// Register-resident complex64 product passes for the padded lengths
// 315 = 15 x 21, 320 = 16 x 20, 324 = 18 x 18 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_f(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 315: return fast::run_product_pass<float, 15, 21>(pass, a);
    case 320: return fast::run_product_pass<float, 16, 20>(pass, a);
    case 324: return fast::run_product_pass<float, 18, 18>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
