// Register-resident product passes for M = 32 = 4 x 8, 64 = 8 x 8 and
// 128 = 8 x 16 (the 16^3, 32^3 and 64^3 spheres), and the length dispatch.
#include "fast_impl.cuh"

namespace dda {

template <typename R> cudaError_t fast_pass_small(int M, int pass, const FastArgs& a) {
  switch (M) {
    case 32: return fast::run_pass<R, 4, 8>(pass, a);
    case 64: return fast::run_pass<R, 8, 8>(pass, a);
    case 128: return fast::run_pass<R, 8, 16>(pass, a);
  }
  return cudaErrorNotSupported;
}
template cudaError_t fast_pass_small<float>(int, int, const FastArgs&);
template cudaError_t fast_pass_small<double>(int, int, const FastArgs&);

bool fast_supported(int M) {
  return M == 32 || M == 40 || M == 48 || M == 64 || M == 80 || M == 96 || M == 128 || M == 256 ||
         M == 270;
}
bool fast_tile_variants(int M) { return fast_supported(M) || M == 512 || M == 1080; }

// complex64 passes of the 7-smooth lengths an axis of 65 to 95 or 136 to 189
// cells is padded to (343 = 7^3 has no split into two register transforms of
// balanced length): the units that hold them.  The Stockham passes these
// lengths ran on make log M trips through shared memory; a 77 x 93 x 71
// ellipsoid's adjoint product with two right-hand sides (160 x 189 x 144)
// took 1,076 us on them and takes 228 us on these (z pass 643 -> 95 us).  The
// padded lengths themselves are unchanged, so complex128 and double-float
// work on these grids is as before (FP64 passes are bound by the FP64 pipe
// either way).
namespace {
using C64Pass = cudaError_t (*)(int, int, const FastArgs&);
C64Pass c64_pass(int M) {
  switch (M) {
    case 135: case 140: case 144: return fast_pass_c64_a;
    case 147: case 150: case 160: return fast_pass_c64_b;
    case 162: case 168: case 175: return fast_pass_c64_c;
    case 180: case 189: case 280: return fast_pass_c64_d;
    case 288: case 294: case 300: return fast_pass_c64_e;
    case 315: case 320: case 324: return fast_pass_c64_f;
    case 336: case 350: case 360: return fast_pass_c64_g;
    case 375: case 378: return fast_pass_c64_h;
  }
  return nullptr;
}
}  // namespace
bool fast_supported_c64(int M) { return fast_tile_variants(M) || c64_pass(M) != nullptr; }

template <typename R> cudaError_t fast_pass(int M, int pass, const FastArgs& a) {
  if (M == 270) return fast_pass_270<R>(pass, a);
  if (M == 256) return fast_pass_256<R>(pass, a);
  if constexpr (std::is_same<R, float>::value) {
    if (M == 512) return fast_pass_512_c64(pass, a);
    if (M == 1080) return fast_pass_1080_c64(pass, a);
    if (C64Pass f = c64_pass(M)) return f(M, pass, a);
  }
  if (M == 40 || M == 48 || M == 80 || M == 96) return fast_pass_mid<R>(M, pass, a);
  return fast_pass_small<R>(M, pass, a);
}
template cudaError_t fast_pass<float>(int, int, const FastArgs&);
template cudaError_t fast_pass<double>(int, int, const FastArgs&);
template <> cudaError_t fast_pass<df>(int M, int pass, const FastArgs& a) {
  if (M == 270) return fast_pass_270_df(pass, a);
  if (M == 256) return fast_pass_256_df(pass, a);
  if (M == 40 || M == 48 || M == 80 || M == 96) return fast_pass_mid_df(M, pass, a);
  return fast_pass_small_df(M, pass, a);
}

}  // namespace dda
