// Register-resident complex64 product passes for the padded lengths
// 288 = 16 x 18, 294 = 14 x 21, 300 = 15 x 20 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_e(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 288: return fast::run_product_pass<float, 16, 18>(pass, a);
    case 294: return fast::run_product_pass<float, 14, 21>(pass, a);
    case 300: return fast::run_product_pass<float, 15, 20>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
