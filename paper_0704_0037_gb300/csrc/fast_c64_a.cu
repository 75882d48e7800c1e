// Register-resident complex64 product passes for the padded lengths
// 135 = 9 x 15, 140 = 10 x 14, 144 = 12 x 12 (fast_c64_pass).
#include "fast_impl.cuh"

namespace dda {
cudaError_t fast_pass_c64_a(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 135: return fast::run_product_pass<float, 9, 15>(pass, a);
    case 140: return fast::run_product_pass<float, 10, 14>(pass, a);
    case 144: return fast::run_product_pass<float, 12, 12>(pass, a);
  }
  return cudaErrorNotSupported;
}
}  // namespace dda
