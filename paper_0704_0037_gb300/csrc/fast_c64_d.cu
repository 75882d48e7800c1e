// Register-resident complex64 product passes for the padded lengths
// 180 = 12 x 15, 189 = 9 x 21, 280 = 14 x 20 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_d(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 180: return fast::run_product_pass<float, 12, 15>(pass, a);
    case 189: return fast::run_product_pass<float, 9, 21>(pass, a);
    case 280: return fast::run_product_pass<float, 14, 20>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
