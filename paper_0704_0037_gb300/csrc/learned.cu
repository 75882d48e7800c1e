// Learned right preconditioner: a small 3D convolutional network that maps a
// residual r of Eq. (3) to an approximation of the error A^-1 r, trained on
// (residual -> error) pairs the solver itself produces, and used inside a
// flexible Bi-CGSTAB whose residual is that of the exact product.  Sec. 4 of
// the paper traces the slow convergence for large m to the system itself and
// Sec. 5 names better preconditioning as the way forward; the paper trains
// nothing, so this whole file has no counterpart there.
//
// Network (1,033,430 parameters; BF16 weights in every product, FP32
// master copy, activations and accumulation):
//   features at half resolution s0 = ceil(n/2) per axis: the 2x2x2 average of
//   (Re, Im) of the three components of r / rms(r) and the occupied fraction
//   L0 conv3 7->16 relu [s0] -> pool2 -> L1 conv3 16->32 relu [s1]
//   -> pool2 -> L2 conv3 32->160 relu, L3 conv3 160->160 relu [s2]
//   -> up2, concat L1 -> L4 conv3 192->32 relu [s1]
//   -> up2, concat L0 -> L5 conv3 48->16 relu [s0] -> L6 conv1 16->6 [s0]
//   output: r plus the value of each dipole's half-resolution cell times
//   rms(r) (identity plus a learned correction: an untrained network with
//   its small last layer is close to no preconditioner at all).
// conv3 = 3x3x3, zero padding 1; pool2 = average of the existing children;
// up2 = nearest.  Loss: |N(r) - e|^2 / |e|^2 over the dipoles; Adam.
// Every reduction has a fixed order (per-block partials, then one block), so
// training and inference are deterministic.
#include <cuda_bf16.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <new>
#include <random>
#include <vector>

#include "internal.h"
#include "pcconv.cuh"

namespace dda {
namespace pc {

constexpr int NL = 7;
struct LayerSpec { int cin, cout, k, relu; };
constexpr LayerSpec kSpec[NL] = {{7, 16, 3, 1},   {16, 32, 3, 1},  {32, 160, 3, 1}, {160, 160, 3, 1},
                                 {192, 32, 3, 1}, {48, 16, 3, 1},  {16, 6, 1, 0}};
// Blocks below nb = cout ceil(cin / 8): g[co][ci][t] += sum over chunks of
// part[chunk][t][co][ci] (fixed order) for one co and 8 ci, a thread per
// weight, read along ci, turned in shared memory and written along t; block
// nb + co: gb[co] += sum_v gout[co][v] (fixed-order reduction)
__global__ void __launch_bounds__(256) k_sum_chunks(const float* __restrict__ part, int chunks, int k3,
                                                    int cin, int cout, float* __restrict__ g, int nb,
                                                    const float* __restrict__ gout, long long nv,
                                                    float* __restrict__ gb) {
  __shared__ float sh[256];
  if ((int)blockIdx.x < nb) {
    const int cb = (cin + 7) / 8, co = blockIdx.x / cb, c0 = (blockIdx.x % cb) * 8, nc = min(8, cin - c0);
    const long long n = (long long)k3 * cout * cin;
    const int t = threadIdx.x >> 3, ci = threadIdx.x & 7;
    if (t < k3 && ci < nc) {
      const float* p = part + ((long long)t * cout + co) * cin + c0 + ci;
      float s = 0.0f;
#pragma unroll 16
      for (int c = 0; c < chunks; ++c) s += p[c * n];
      sh[ci * k3 + t] = s;
    }
    __syncthreads();
    if ((int)threadIdx.x < nc * k3) g[((long long)co * cin + c0) * k3 + threadIdx.x] += sh[threadIdx.x];
    return;
  }
  const int co = blockIdx.x - nb;
  float s = 0.0f;
#pragma unroll 8
  for (long long v = threadIdx.x; v < nv; v += 256) s += gout[co * nv + v];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) gb[co] += sh[0];
}

// ---------------------------------------------------------------- pooling
// out[c][p] = mean of in[c][children of p] (children inside the grid)
__global__ void k_pool2(const float* __restrict__ in, Dims di, float* __restrict__ out, Dims dout,
                        int ch) {
  const long long n = dout.n() * ch;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / dout.n());
    const long long p = i - c * dout.n();
    const int X = (int)(p % dout.x), Y = (int)((p / dout.x) % dout.y), Z = (int)(p / ((long long)dout.x * dout.y));
    float s = 0.0f;
    int cnt = 0;
    for (int dz = 0; dz < 2; ++dz)
      for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx) {
          const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
          if (x < di.x && y < di.y && z < di.z) {
            s += in[c * di.n() + ((long long)z * di.y + y) * di.x + x];
            ++cnt;
          }
        }
    out[i] = s / (float)cnt;
  }
}
// k_pool2 over split units, a thread per voxel and 8 channels
__global__ void __launch_bounds__(128) k_pool2_split(const uint4* __restrict__ in, Dims di, uint4* __restrict__ out,
                                                     Dims dout, int ch) {
  const long long nin = di.n(), no = dout.n(), n = no * (ch / 8);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / no);
    const long long p = i - c * no;
    const int X = (int)(p % dout.x), Y = (int)((p / dout.x) % dout.y), Z = (int)(p / ((long long)dout.x * dout.y));
    float s[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    int cnt = 0;
    for (int dz = 0; dz < 2; ++dz)
      for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx) {
          const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
          if (x < di.x && y < di.y && z < di.z) {
            const long long v = ((long long)z * di.y + y) * di.x + x;
            uint4 u[3];
            float f[8];
#pragma unroll
            for (int k = 0; k < 3; ++k) u[k] = in[(3LL * c + k) * nin + v];
            join_unit(u, f);
#pragma unroll
            for (int k = 0; k < 8; ++k) s[k] += f[k];
            ++cnt;
          }
        }
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] /= (float)cnt;
    uint4 u[3];
    split_unit(s, u);
#pragma unroll
    for (int k = 0; k < 3; ++k) out[(3LL * c + k) * no + p] = u[k];
  }
}
// gin[c][v] += gout[c][parent(v)] / children(parent), then zero where the
// activation act[c][v] <= 0 (gradient behind its relu)
__global__ void k_pool2_back(const float* __restrict__ gout, Dims dout, float* __restrict__ gin,
                             Dims di, int ch, const float* __restrict__ act) {
  const long long n = di.n() * ch;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / di.n());
    const long long v = i - c * di.n();
    const int x = (int)(v % di.x), y = (int)((v / di.x) % di.y), z = (int)(v / ((long long)di.x * di.y));
    const int X = x / 2, Y = y / 2, Z = z / 2;
    const int cnt = (min(2, di.x - 2 * X)) * (min(2, di.y - 2 * Y)) * (min(2, di.z - 2 * Z));
    const float r = gin[i] + gout[c * dout.n() + ((long long)Z * dout.y + Y) * dout.x + X] / (float)cnt;
    gin[i] = act[i] > 0.0f ? r : 0.0f;
  }
}
// gin[c][p] = sum of gout[c][children of p], zero where act[c][p] <= 0
__global__ void k_up2_back(const float* __restrict__ gout, Dims df, float* __restrict__ gin,
                           Dims dc, int ch, const float* __restrict__ act) {
  const long long n = dc.n() * ch;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / dc.n());
    const long long p = i - c * dc.n();
    const int X = (int)(p % dc.x), Y = (int)((p / dc.x) % dc.y), Z = (int)(p / ((long long)dc.x * dc.y));
    float s = 0.0f;
    for (int dz = 0; dz < 2; ++dz)
      for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx) {
          const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
          if (x < df.x && y < df.y && z < df.z) s += gout[c * df.n() + ((long long)z * df.y + y) * df.x + x];
        }
    gin[i] = act[i] > 0.0f ? s : 0.0f;
  }
}

// ---------------------------------------------------------------- lattice <-> grid
// map[(z ny + y) nx + x] = dipole index (or -1), one thread per dipole
__global__ void k_idx_map(LatticeDev lat, int nx, int ny, int nrows, int* __restrict__ map) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int row = warp; row < nrows; row += nwarps)
    for (long long i = lat.row_off[row] + lane; i < lat.row_off[row + 1]; i += 32)
      map[(long long)row * nx + lat.xi[i]] = (int)i;
}
// features at s0: channel 2c / 2c+1 = mean of Re / Im of v_c / rms over the
// cell's children (void children count as zero), channel 6 = occupied
// fraction; a thread per cell and component
__global__ void __launch_bounds__(256) k_feat_in(const c128* __restrict__ v, long long n_occ,
                                                 const int* __restrict__ map, Dims dl, Dims d0,
                                                 const double* __restrict__ scl, float* __restrict__ f) {
  const double inv = scl[5] * 0.125;           // exact: a power of two
  const int c = blockIdx.y;
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < d0.n();
       p += (long long)gridDim.x * blockDim.x) {
    const int X = (int)(p % d0.x), Y = (int)((p / d0.x) % d0.y), Z = (int)(p / ((long long)d0.x * d0.y));
    int id[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int x = 2 * X + (k & 1), y = 2 * Y + ((k >> 1) & 1), z = 2 * Z + (k >> 2);
      id[k] = x < dl.x && y < dl.y && z < dl.z ? map[((long long)z * dl.y + y) * dl.x + x] : -1;
    }
    double re = 0.0, im = 0.0;
    int occ = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (id[k] < 0) continue;               // FP64 additions only where there are dipoles
      const c128 a = v[c * n_occ + id[k]];
      ++occ;
      re += a.x;
      im += a.y;
    }
    f[(2 * c) * d0.n() + p] = (float)(re * inv);
    f[(2 * c + 1) * d0.n() + p] = (float)(im * inv);
    if (c == 0) f[6 * d0.n() + p] = occ * 0.125f;
  }
}
// (double)x, in integer instructions for zero and normal x: the sweep below is
// bound by the FP64 pipe, which also does the conversions
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m >= 0x7f800000u || (m < 0x00800000u && m)) return (double)x;      // infinity, NaN, subnormal
  const unsigned hi = m ? (m >> 3) + 0x38000000u : 0u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}
// z_i = v_i + rms * out6[.][cell(i)] for every dipole (complex128): the
// identity plus the learned correction
__global__ void k_feat_out(const float* __restrict__ o6, Dims d0, LatticeDev lat, int nx, int ny,
                           int nrows, long long n_occ, const double* __restrict__ scl,
                           const c128* __restrict__ v, c128* __restrict__ z) {
  const double s = scl[0];
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int row = warp; row < nrows; row += nwarps) {
    const int y = row % ny, zz = row / ny;
    for (long long i = lat.row_off[row] + lane; i < lat.row_off[row + 1]; i += 32) {
      const long long p = ((long long)(zz / 2) * d0.y + y / 2) * d0.x + lat.xi[i] / 2;
      for (int c = 0; c < 3; ++c)
        z[c * n_occ + i] = fmas<double>(mk<double>(widen(o6[(2 * c) * d0.n() + p]), widen(o6[(2 * c + 1) * d0.n() + p])),
                                        s, v[c * n_occ + i]);
    }
  }
}
// gradient of |z - e|^2 / |e|^2 with respect to out6 (z = rms * out6[cell]):
// g6[ch][p] = rms * sum over the cell's dipoles of 2 (z - e)_ch / |e|^2; a
// thread per cell and component
__global__ void __launch_bounds__(256) k_loss_grad(const c128* __restrict__ zz, const c128* __restrict__ e,
                                                   long long n_occ, const int* __restrict__ map, Dims dl,
                                                   Dims d0, const double* __restrict__ scl,
                                                   float* __restrict__ g6) {
  const double w = 2.0 * scl[0] * scl[6];
  const int c = blockIdx.y;
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < d0.n();
       p += (long long)gridDim.x * blockDim.x) {
    const int X = (int)(p % d0.x), Y = (int)((p / d0.x) % d0.y), Z = (int)(p / ((long long)d0.x * d0.y));
    int id[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int x = 2 * X + (k & 1), y = 2 * Y + ((k >> 1) & 1), z = 2 * Z + (k >> 2);
      id[k] = x < dl.x && y < dl.y && z < dl.z ? map[((long long)z * dl.y + y) * dl.x + x] : -1;
    }
    double re = 0.0, im = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (id[k] < 0) continue;
      const c128 d = zz[c * n_occ + id[k]] - e[c * n_occ + id[k]];
      re += d.x;
      im += d.y;
    }
    g6[(2 * c) * d0.n() + p] = (float)(w * re);
    g6[(2 * c + 1) * d0.n() + p] = (float)(w * im);
  }
}

// per-block partial sums of |a|^2 (slot 0) and |a - b|^2 (slot 1; b may be
// null), four elements in flight per thread; k_sq_fin adds the sq_blocks(n) of
// them (at most kSqB) in a fixed order
constexpr int kSqB = 1024;
inline int sq_blocks(long long n) { return (int)std::max<long long>(1, std::min<long long>((n + 1023) / 1024, kSqB)); }
__global__ void __launch_bounds__(256) k_sq_part(const c128* __restrict__ a, const c128* __restrict__ b,
                                                 long long n, double* __restrict__ part) {
  __shared__ double sh[2][256];
  double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
    const c128 x = a[i];
    s0 = fma(x.x, x.x, fma(x.y, x.y, s0));
    if (b) {
      const c128 d = x - b[i];
      s1 = fma(d.x, d.x, fma(d.y, d.y, s1));
    }
  }
  sh[0][threadIdx.x] = s0;
  sh[1][threadIdx.x] = s1;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = sh[0][0];
    part[2 * blockIdx.x + 1] = sh[1][0];
  }
}
// one block of 256 threads: the sums of slots 0 and 1 go to sc[0] as rms =
// sqrt(s0 / n), sc[5] = 1 / rms (n > 0), or to sc[3] = s0, sc[4] = s1 and sc[6]
// = 1 / s0 (n = 0); reciprocals of zero are 0
__global__ void __launch_bounds__(256) k_sq_fin(const double* __restrict__ part, int nb,
                                                double* __restrict__ sc, long long n) {
  __shared__ double sh[2][256];
  double s0 = 0.0, s1 = 0.0;
  for (int b = threadIdx.x; b < nb; b += 256) { s0 += part[2 * b]; s1 += part[2 * b + 1]; }
  sh[0][threadIdx.x] = s0;
  sh[1][threadIdx.x] = s1;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x) return;
  s0 = sh[0][0];
  s1 = sh[1][0];
  if (n > 0) {
    const double rms = sqrt(s0 / (double)n);
    sc[0] = rms;
    sc[5] = rms > 0.0 ? 1.0 / rms : 0.0;
  } else {
    sc[3] = s0;
    sc[4] = s1;
    sc[6] = s0 > 0.0 ? 1.0 / s0 : 0.0;
  }
}

// Adam (bias-corrected), then the BF16 copy used by the products
__global__ void k_adam(float* __restrict__ w, __nv_bfloat16* __restrict__ wb, const float* __restrict__ g,
                       float* __restrict__ m1, float* __restrict__ m2, long long n, float lr, float b1,
                       float b2, float c1, float c2, float eps) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.0f - b1) * gi;
    const float b = b2 * m2[i] + (1.0f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    const float wi = w[i] - lr * (a / c1) / (sqrtf(b / c2) + eps);
    w[i] = wi;
    wb[i] = __float2bfloat16(wi);
  }
}
__global__ void k_to_bf16(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    wb[i] = __float2bfloat16(w[i]);
}

inline int gs(long long n) { return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 4096)); }

}  // namespace pc
}  // namespace dda

using namespace dda;
using namespace dda::pc;

// The network and its working memory (grown to the largest lattice seen).
struct dda_pcnet {
  int device = 0;
  long long nparam = 0;
  long long woff[NL] = {}, boff[NL] = {};
  float* w = nullptr;           // FP32 master weights and biases
  __nv_bfloat16* wb = nullptr;  // BF16 copy (weights and biases; products use the weights)
  uint2* wp = nullptr;          // BF16 weights in fragment order (forward products of apply)
  float* wf = nullptr;          // FP32 copies for training: forward, then input gradients
  PackList pack = {}, packf = {};   // their layouts: item L forward, item NL + L input gradient
  float* g = nullptr;           // gradients
  float* m1 = nullptr;
  float* m2 = nullptr;
  int step = 0;
  // activations and gradients
  void* arena = nullptr;
  size_t arena_bytes = 0;
  float* part = nullptr;        // weight-gradient partials
  size_t part_bytes = 0;
  int* map = nullptr;           // dipole index map of the current handle
  size_t map_bytes = 0;
  long long map_of = 0;         // uid of the handle the map was built for
  double* scal = nullptr;       // k_sq_fin: [0] rms(v), [3] |e|^2, [4] |e - z|^2, [5] 1 / [0], [6] 1 / [3]
  double* red = nullptr;        // reduction partials
  std::string err;
};

namespace {

int pc_fail(dda_pcnet_t n, int code, const std::string& m) {
  if (n) n->err = m;
  return code;
}

// Buffers of one forward/backward pass for lattice dims dl.
struct Acts {
  Dims d0, d1, d2;
  float *f0, *a0, *a5, *o6, *p1, *a1, *a4, *p2, *a2, *a3;
  float *g6, *ga5, *gcat0, *gcat1, *ga4, *ga3, *ga2, *gp2, *gp1;
  void* arena_split;                           // split activations of a pass without gradient
};

size_t acts_floats(Dims d0, Dims d1, Dims d2) {
  return (size_t)d0.n() * (7 + 16 + 16 + 6 + 6 + 16 + 48) + (size_t)d1.n() * (16 + 32 + 32 + 192 + 32 + 16) +
         (size_t)d2.n() * (32 + 160 + 160 + 160 + 160 + 32);
}

int ensure_arena(dda_pcnet_t net, dda_t h, Acts& A) {
  const Dims dl{h->g.nx, h->g.ny, h->g.nz};
  A.d0 = halved(dl);
  A.d1 = halved(A.d0);
  A.d2 = halved(A.d1);
  const size_t need = acts_floats(A.d0, A.d1, A.d2) * sizeof(float) + 256;
  if (net->arena_bytes < need) {
    dev_free(net->arena, h->stream);
    net->arena = nullptr;
    net->arena_bytes = 0;
    if (dev_malloc(&net->arena, need) != cudaSuccess) {
      cudaGetLastError();
      return pc_fail(net, DDA_ERR_OOM, "network activations");
    }
    net->arena_bytes = need;
  }
  float* p = (float*)net->arena;
  auto take = [&](long long n) { float* r = p; p += n; return r; };
  A.f0 = take(7 * A.d0.n());
  A.o6 = take(6 * A.d0.n());
  A.arena_split = (void*)(((size_t)p + 15) & ~(size_t)15);
  A.a0 = take(16 * A.d0.n());
  A.a5 = take(16 * A.d0.n());
  A.g6 = take(6 * A.d0.n());
  A.ga5 = take(16 * A.d0.n());
  A.gcat0 = take(48 * A.d0.n());
  A.p1 = take(16 * A.d1.n());
  A.a1 = take(32 * A.d1.n());
  A.a4 = take(32 * A.d1.n());
  A.gcat1 = take(192 * A.d1.n());
  A.ga4 = take(32 * A.d1.n());
  A.gp1 = take(16 * A.d1.n());
  A.p2 = take(32 * A.d2.n());
  A.a2 = take(160 * A.d2.n());
  A.a3 = take(160 * A.d2.n());
  A.ga3 = take(160 * A.d2.n());
  A.ga2 = take(160 * A.d2.n());
  A.gp2 = take(32 * A.d2.n());
  // the dipole index map of this handle
  const long long nbox = (long long)dl.x * dl.y * dl.z;
  if (net->map_bytes < (size_t)nbox * sizeof(int)) {
    dev_free(net->map, h->stream);
    net->map = nullptr;
    net->map_bytes = 0;
    if (dev_malloc(&net->map, (size_t)nbox * sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      return pc_fail(net, DDA_ERR_OOM, "network index map");
    }
    net->map_bytes = (size_t)nbox * sizeof(int);
    net->map_of = 0;
  }
  if (net->map_of != h->uid) {
    if (cudaMemsetAsync(net->map, 0xff, (size_t)nbox * sizeof(int), h->stream) != cudaSuccess)
      return pc_fail(net, DDA_ERR_CUDA, "index map");
    k_idx_map<<<std::min(4096, (h->g.nrows + 7) / 8), 256, 0, h->stream>>>(h->lat(), h->g.nx, h->g.ny,
                                                                           h->g.nrows, net->map);
    count_launch();
    net->map_of = h->uid;
  }
  return DDA_OK;
}

// input of layer L: one array, or the upsampled coarse channels and the skip
// connection of the decoder layers
ConvIn layer_input(const Acts& A, int L) {
  const Dims no{0, 0, 0};
  switch (L) {
    case 0: return {A.f0, 7, no, false, nullptr, 0};
    case 1: return {A.p1, 16, no, false, nullptr, 0};
    case 2: return {A.p2, 32, no, false, nullptr, 0};
    case 3: return {A.a2, 160, no, false, nullptr, 0};
    case 4: return {A.a3, 160, A.d2, true, A.a1, 32};
    case 5: return {A.a4, 32, A.d1, true, A.a0, 16};
    default: return {A.a5, 16, no, false, nullptr, 0};
  }
}

cudaError_t conv_fwd(dda_pcnet_t net, int L, const Acts& A, float* out, Dims d, cudaStream_t st) {
  const LayerSpec& s = kSpec[L];
  return conv_f32(s.k, layer_input(A, L), net->wf + net->packf.item[L].at, net->w + net->boff[L], nullptr, out,
                  s.cout, d, s.relu, st);
}

// The seven layers of a pass that keeps nothing for a gradient: features A.f0
// to A.o6, activations split (244 bytes per voxel of d0, 480 of d1, 2,112 of
// d2, in the arena of a training pass's 460, 1,280 and 2,816)
cudaError_t layers_split(dda_pcnet_t net, const Acts& A, cudaStream_t st) {
  const long long n0 = A.d0.n(), n1 = A.d1.n(), n2 = A.d2.n();
  uint4* p = (uint4*)(A.arena_split);
  auto take = [&](int ch, long long n) { uint4* r = p; p += (long long)ch / 8 * 3 * n; return r; };
  uint4 *a0 = take(16, n0), *a5 = take(16, n0), *p1 = take(16, n1), *a1 = take(32, n1), *a4 = take(32, n1),
        *p2 = take(32, n2), *a2 = take(160, n2), *a3 = take(160, n2);
  const Dims no{0, 0, 0};
  cudaError_t e = cudaSuccess;
  auto conv = [&](int L, const SplitIn& in, const SplitOut& out, Dims d) {
    const LayerSpec& s = kSpec[L];
    if (e == cudaSuccess)
      e = conv_mma(s.k, in, net->wp + net->pack.item[L].at, net->w + net->boff[L], out, s.cout, d, s.relu, st);
  };
  auto pool = [&](const uint4* in, Dims di, uint4* out, Dims dout, int ch) {
    const long long n = dout.n() * (ch / 8);
    k_pool2_split<<<(unsigned)std::min<long long>((n + 127) / 128, 1 << 20), 128, 0, st>>>(in, di, out, dout, ch);
    count_launch();
  };
  conv(0, {nullptr, 0, no, false, nullptr, 0, A.f0, 7}, {a0, nullptr}, A.d0);
  pool(a0, A.d0, p1, A.d1, 16);
  conv(1, {p1, 16, no, false, nullptr, 0, nullptr, 0}, {a1, nullptr}, A.d1);
  pool(a1, A.d1, p2, A.d2, 32);
  conv(2, {p2, 32, no, false, nullptr, 0, nullptr, 0}, {a2, nullptr}, A.d2);
  conv(3, {a2, 160, no, false, nullptr, 0, nullptr, 0}, {a3, nullptr}, A.d2);
  conv(4, {a3, 160, A.d2, true, a1, 32, nullptr, 0}, {a4, nullptr}, A.d1);
  conv(5, {a4, 32, A.d1, true, a0, 16, nullptr, 0}, {a5, nullptr}, A.d0);
  conv(6, {a5, 16, no, false, nullptr, 0, nullptr, 0}, {nullptr, A.o6}, A.d0);
  return e;
}

// input gradient of layer L: gin = conv(gout, wT) (no bias), zero where the
// activation act <= 0 (act null: no relu in front)
cudaError_t conv_bwd_data(dda_pcnet_t net, int L, const float* gout, float* gin, const float* act, Dims d,
                          cudaStream_t st) {
  const LayerSpec& s = kSpec[L];
  const ConvIn in{gout, s.cout, {0, 0, 0}, false, nullptr, 0};
  return conv_f32(s.k, in, net->wf + net->packf.item[NL + L].at, nullptr, act, gin, s.cin, d, 0, st);
}

int conv_bwd_weight(dda_pcnet_t net, int L, const Acts& A, const float* gout, Dims d, cudaStream_t st) {
  const LayerSpec& s = kSpec[L];
  const int K3 = s.k * s.k * s.k;
  // voxel tiles in up to 16 chunks (the order of the sums)
  const int tiles = ((d.x + kWX - 1) / kWX) * ((d.y + kWY - 1) / kWY) * ((d.z + kWZ - 1) / kWZ);
  const int chunks = std::max(1, std::min(tiles, 16));
  const int per = (tiles + chunks - 1) / chunks;
  const long long nw = (long long)s.cout * s.cin * K3;
  const size_t need = (size_t)chunks * nw * sizeof(float);
  if (net->part_bytes < need) {
    dev_free(net->part, st);
    net->part = nullptr;
    net->part_bytes = 0;
    if (dev_malloc(&net->part, need) != cudaSuccess) {
      cudaGetLastError();
      return pc_fail(net, DDA_ERR_OOM, "weight-gradient partials");
    }
    net->part_bytes = need;
  }
  if (s.k == 3) {
    const size_t sm = (size_t)(per > 1 ? 2 : 1) * kWTile * sizeof(float);
    cudaError_t e = ensure_smem((const void*)k_wgrad_f32, sm);
    if (e == cudaSuccess) e = ensure_carveout_max((const void*)k_wgrad_f32);
    if (e != cudaSuccess) return pc_fail(net, DDA_ERR_CUDA, cudaGetErrorString(e));
    k_wgrad_f32<<<dim3(chunks, (s.cout + 7) / 8, (s.cin + 15) / 16), 216, sm, st>>>(layer_input(A, L), gout,
                                                                                    s.cout, d, net->part, per);
  } else
    k_wgrad1<<<chunks, 96, 0, st>>>(A.a5, s.cin, gout, s.cout, d, net->part, per);
  count_launch();
  const int nb = s.cout * ((s.cin + 7) / 8);
  k_sum_chunks<<<nb + s.cout, 256, 0, st>>>(net->part, chunks, K3, s.cin, s.cout, net->g + net->woff[L], nb, gout,
                                            d.n(), net->g + net->boff[L]);
  count_launch();
  return DDA_OK;
}

// the copies of the weights the convolutions read, after every change of them
// (the callers synchronise before they return, so any stream may read them)
void pack_weights(dda_pcnet_t net, cudaStream_t st) {
  auto size = [](const PackList& pl) { return pl.item[pl.count - 1].at + pl.item[pl.count - 1].n; };
  k_pack_weights<<<gs(size(net->pack)), 256, 0, st>>>(net->wb, net->pack, net->wp, size(net->pack));
  count_launch();
  k_pack_f32<<<gs(size(net->packf)), 256, 0, st>>>(net->wb, net->packf, net->wf, size(net->packf));
  count_launch();
}

// z = N(v) on the handle's lattice (v, z complex128 [3][N_occ]); leaves the
// activations in A for a backward pass
int forward(dda_pcnet_t net, dda_t h, const c128* v, c128* z, Acts& A, bool train) {
  cudaStream_t st = h->stream;
  const long long n = 3 * h->g.n_occ;
  const Dims dl{h->g.nx, h->g.ny, h->g.nz};
  k_sq_part<<<sq_blocks(n), 256, 0, st>>>(v, nullptr, n, net->red);
  count_launch();
  k_sq_fin<<<1, 256, 0, st>>>(net->red, sq_blocks(n), net->scal, n);     // rms(v)
  count_launch();
  k_feat_in<<<dim3(gs(A.d0.n()), 3), 256, 0, st>>>(v, h->g.n_occ, net->map, dl, A.d0, net->scal, A.f0);
  count_launch();
  cudaError_t e;
  if (!train) {
    e = layers_split(net, A, st);
  } else {
    e = conv_fwd(net, 0, A, A.a0, A.d0, st);
    k_pool2<<<gs(16 * A.d1.n()), 256, 0, st>>>(A.a0, A.d0, A.p1, A.d1, 16); count_launch();
    if (e == cudaSuccess) e = conv_fwd(net, 1, A, A.a1, A.d1, st);
    k_pool2<<<gs(32 * A.d2.n()), 256, 0, st>>>(A.a1, A.d1, A.p2, A.d2, 32); count_launch();
    if (e == cudaSuccess) e = conv_fwd(net, 2, A, A.a2, A.d2, st);
    if (e == cudaSuccess) e = conv_fwd(net, 3, A, A.a3, A.d2, st);
    if (e == cudaSuccess) e = conv_fwd(net, 4, A, A.a4, A.d1, st);
    if (e == cudaSuccess) e = conv_fwd(net, 5, A, A.a5, A.d0, st);
    if (e == cudaSuccess) e = conv_fwd(net, 6, A, A.o6, A.d0, st);
  }
  k_feat_out<<<std::min(4096, (h->g.nrows + 7) / 8), 256, 0, st>>>(A.o6, A.d0, h->lat(), h->g.nx, h->g.ny,
                                                                  h->g.nrows, h->g.n_occ, net->scal, v, z);
  count_launch();
  if (e == cudaSuccess) e = cudaGetLastError();
  return e == cudaSuccess ? DDA_OK : pc_fail(net, DDA_ERR_CUDA, cudaGetErrorString(e));
}

int backward(dda_pcnet_t net, dda_t h, const c128* z, const c128* e, Acts& A) {
  cudaStream_t st = h->stream;
  const Dims dl{h->g.nx, h->g.ny, h->g.nz};
  float* ga0 = A.gcat0 + 32 * A.d0.n();
  float* ga1 = A.gcat1 + 160 * A.d1.n();
  k_loss_grad<<<dim3(gs(A.d0.n()), 3), 256, 0, st>>>(z, e, h->g.n_occ, net->map, dl, A.d0, net->scal, A.g6);
  count_launch();
  int rc;
  cudaError_t er = cudaSuccess;
  auto data = [&](int L, const float* gout, float* gin, const float* act, Dims d) {
    if (er == cudaSuccess) er = conv_bwd_data(net, L, gout, gin, act, d, st);
  };
  // L6 (conv1, linear)
  if ((rc = conv_bwd_weight(net, 6, A, A.g6, A.d0, st)) != DDA_OK) return rc;
  data(6, A.g6, A.ga5, A.a5, A.d0);
  // L5
  if ((rc = conv_bwd_weight(net, 5, A, A.ga5, A.d0, st)) != DDA_OK) return rc;
  data(5, A.ga5, A.gcat0, nullptr, A.d0);
  // up2 back to L4's output
  k_up2_back<<<gs(32 * A.d1.n()), 256, 0, st>>>(A.gcat0, A.d0, A.ga4, A.d1, 32, A.a4); count_launch();
  // L4
  if ((rc = conv_bwd_weight(net, 4, A, A.ga4, A.d1, st)) != DDA_OK) return rc;
  data(4, A.ga4, A.gcat1, nullptr, A.d1);
  k_up2_back<<<gs(160 * A.d2.n()), 256, 0, st>>>(A.gcat1, A.d1, A.ga3, A.d2, 160, A.a3); count_launch();
  // L3
  if ((rc = conv_bwd_weight(net, 3, A, A.ga3, A.d2, st)) != DDA_OK) return rc;
  data(3, A.ga3, A.ga2, A.a2, A.d2);
  // L2
  if ((rc = conv_bwd_weight(net, 2, A, A.ga2, A.d2, st)) != DDA_OK) return rc;
  data(2, A.ga2, A.gp2, nullptr, A.d2);
  // pool back into L1's output (skip gradient already in gcat1[160..])
  k_pool2_back<<<gs(32 * A.d1.n()), 256, 0, st>>>(A.gp2, A.d2, ga1, A.d1, 32, A.a1); count_launch();
  // L1
  if ((rc = conv_bwd_weight(net, 1, A, ga1, A.d1, st)) != DDA_OK) return rc;
  data(1, ga1, A.gp1, nullptr, A.d1);
  k_pool2_back<<<gs(16 * A.d0.n()), 256, 0, st>>>(A.gp1, A.d1, ga0, A.d0, 16, A.a0); count_launch();
  // L0 (no input gradient)
  if ((rc = conv_bwd_weight(net, 0, A, ga0, A.d0, st)) != DDA_OK) return rc;
  if (er == cudaSuccess) er = cudaGetLastError();
  return er == cudaSuccess ? DDA_OK : pc_fail(net, DDA_ERR_CUDA, cudaGetErrorString(er));
}

bool pc_device_ok(dda_pcnet_t net, dda_t h) { return net->device == h->device; }

}  // namespace

// ---------------------------------------------------------------- C-ABI
extern "C" int dda_pcnet_create(dda_pcnet_t* out, unsigned long long seed) {
  if (!out) return DDA_ERR_ARG;
  *out = nullptr;
  dda_pcnet* net = new (std::nothrow) dda_pcnet();
  if (!net) return DDA_ERR_OOM;
  if (cudaGetDevice(&net->device) != cudaSuccess) {
    cudaGetLastError();
    delete net;
    return DDA_ERR_CUDA;
  }
  long long off = 0;
  for (int L = 0; L < NL; ++L) {
    net->woff[L] = off;
    off += (long long)kSpec[L].cout * kSpec[L].cin * kSpec[L].k * kSpec[L].k * kSpec[L].k;
    net->boff[L] = off;
    off += kSpec[L].cout;
  }
  net->nparam = off;
  int pat = 0, patf = 0;
  net->pack.count = NL;
  net->packf.count = 2 * NL;
  for (int q = 0; q < 2 * NL; ++q) {
    const LayerSpec& s = kSpec[q % NL];
    const int flip = q >= NL, ni = flip ? s.cout : s.cin, no = flip ? s.cin : s.cout, k3 = s.k * s.k * s.k;
    const int n = ((ni + 15) / 16) * k3 * ((no + 7) / 8) * 32, nf = ni * k3 * ((no + 7) / 8 * 8);
    if (!flip) {
      net->pack.item[q] = {(int)net->woff[q], s.cin, s.cout, k3, 0, pat, n};
      pat += n;
    }
    net->packf.item[q] = {(int)net->woff[q % NL], s.cin, s.cout, k3, flip, patf, nf};
    patf += nf;
  }
  // He-normal weights from a seeded host generator, zero biases; the last
  // layer starts small so that the untrained network is close to zero
  std::vector<float> hw((size_t)off, 0.0f);
  std::mt19937_64 rng(seed);
  std::normal_distribution<float> nd(0.0f, 1.0f);
  for (int L = 0; L < NL; ++L) {
    const int fan = kSpec[L].cin * kSpec[L].k * kSpec[L].k * kSpec[L].k;
    const float sd = std::sqrt(2.0f / fan) * (L == NL - 1 ? 0.1f : 1.0f);
    for (long long i = net->woff[L]; i < net->boff[L]; ++i) hw[i] = sd * nd(rng);
  }
  int rc = DDA_OK;
  if (dev_malloc(&net->w, off * sizeof(float)) != cudaSuccess ||
      dev_malloc(&net->wb, off * sizeof(__nv_bfloat16)) != cudaSuccess ||
      dev_malloc(&net->wp, pat * sizeof(uint2)) != cudaSuccess ||
      dev_malloc(&net->wf, patf * sizeof(float)) != cudaSuccess ||
      dev_malloc(&net->g, off * sizeof(float)) != cudaSuccess ||
      dev_malloc(&net->m1, off * sizeof(float)) != cudaSuccess ||
      dev_malloc(&net->m2, off * sizeof(float)) != cudaSuccess ||
      dev_malloc(&net->scal, 8 * sizeof(double)) != cudaSuccess ||
      dev_malloc(&net->red, 2 * kSqB * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    rc = DDA_ERR_OOM;
  } else if (cudaMemcpy(net->w, hw.data(), off * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
             cudaMemset(net->m1, 0, off * sizeof(float)) != cudaSuccess ||
             cudaMemset(net->m2, 0, off * sizeof(float)) != cudaSuccess ||
             cudaMemset(net->scal, 0, 8 * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    rc = DDA_ERR_CUDA;
  } else {
    k_to_bf16<<<gs(off), 256>>>(net->w, net->wb, off);
    count_launch();
    pack_weights(net, 0);
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); rc = DDA_ERR_CUDA; }
  }
  if (rc != DDA_OK) {
    dda_pcnet_free(net);
    return rc;
  }
  *out = net;
  return DDA_OK;
}

extern "C" int dda_pcnet_free(dda_pcnet_t net) {
  if (!net) return DDA_OK;
  DeviceGuard dg(net->device);
  cudaDeviceSynchronize();
  dev_free(net->w, 0); dev_free(net->wb, 0); dev_free(net->wp, 0); dev_free(net->wf, 0); dev_free(net->g, 0);
  dev_free(net->m1, 0); dev_free(net->m2, 0); dev_free(net->arena, 0); dev_free(net->part, 0);
  dev_free(net->map, 0); dev_free(net->scal, 0); dev_free(net->red, 0);
  cudaGetLastError();
  delete net;
  return DDA_OK;
}

extern "C" int dda_pcnet_params(dda_pcnet_t net, long long* n) {
  if (!net || !n) return DDA_ERR_ARG;
  *n = net->nparam;
  return DDA_OK;
}

extern "C" const char* dda_pcnet_last_error(dda_pcnet_t net) { return net ? net->err.c_str() : "null network"; }

extern "C" int dda_pcnet_get_weights(dda_pcnet_t net, float* host) {
  if (!net || !host) return DDA_ERR_ARG;
  DeviceGuard dg(net->device);
  if (cudaMemcpy(host, net->w, net->nparam * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) {
    cudaGetLastError();
    return pc_fail(net, DDA_ERR_CUDA, "weights to host");
  }
  return DDA_OK;
}

extern "C" int dda_pcnet_set_weights(dda_pcnet_t net, const float* host) {
  if (!net || !host) return DDA_ERR_ARG;
  DeviceGuard dg(net->device);
  if (cudaMemcpy(net->w, host, net->nparam * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    return pc_fail(net, DDA_ERR_CUDA, "weights from host");
  }
  k_to_bf16<<<gs(net->nparam), 256>>>(net->w, net->wb, net->nparam);
  count_launch();
  pack_weights(net, 0);
  cudaMemset(net->m1, 0, net->nparam * sizeof(float));
  cudaMemset(net->m2, 0, net->nparam * sizeof(float));
  net->step = 0;
  if (cudaDeviceSynchronize() != cudaSuccess) {
    cudaGetLastError();
    return pc_fail(net, DDA_ERR_CUDA, "bf16 copy");
  }
  return DDA_OK;
}

extern "C" int dda_pcnet_apply(dda_pcnet_t net, dda_t h, const void* v_dev, void* z_dev) {
  if (!net || !h || !v_dev || !z_dev) return DDA_ERR_ARG;
  if (!pc_device_ok(net, h)) return pc_fail(net, DDA_ERR_ARG, "network and handle on different devices");
  DDA_ON_DEVICE(h);
  Acts A;
  int rc = ensure_arena(net, h, A);
  if (rc == DDA_OK) rc = forward(net, h, (const c128*)v_dev, (c128*)z_dev, A, false);
  return rc;
}

// One Adam step on the pair (r, e): loss |N(r) - e|^2 / |e|^2; z_dev receives
// N(r) before the step; loss_out (host) the loss.
extern "C" int dda_pcnet_train_step(dda_pcnet_t net, dda_t h, const void* r_dev, const void* e_dev,
                                    void* z_dev, float lr, double* loss_out) {
  if (!net || !h || !r_dev || !e_dev || !z_dev || !(lr > 0.0f)) return DDA_ERR_ARG;
  if (!pc_device_ok(net, h)) return pc_fail(net, DDA_ERR_ARG, "network and handle on different devices");
  DDA_ON_DEVICE(h);
  cudaStream_t st = h->stream;
  Acts A;
  int rc = ensure_arena(net, h, A);
  if (rc != DDA_OK) return rc;
  const c128* r = (const c128*)r_dev;
  const c128* e = (const c128*)e_dev;
  c128* z = (c128*)z_dev;
  if ((rc = forward(net, h, r, z, A, true)) != DDA_OK) return rc;
  // |e|^2 into scal[3], |z - e|^2 into scal[4] (scal[0] keeps rms(r))
  const long long n = 3 * h->g.n_occ;
  k_sq_part<<<sq_blocks(n), 256, 0, st>>>(e, z, n, net->red);
  count_launch();
  k_sq_fin<<<1, 256, 0, st>>>(net->red, sq_blocks(n), net->scal, 0);   // scal[3] = |e|^2, scal[4] = |e - z|^2
  count_launch();
  if (cudaMemsetAsync(net->g, 0, net->nparam * sizeof(float), st) != cudaSuccess)
    return pc_fail(net, DDA_ERR_CUDA, "gradient reset");
  if ((rc = backward(net, h, z, e, A)) != DDA_OK) return rc;
  net->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - std::pow(b1, (float)net->step), c2 = 1.0f - std::pow(b2, (float)net->step);
  k_adam<<<gs(net->nparam), 256, 0, st>>>(net->w, net->wb, net->g, net->m1, net->m2, net->nparam, lr,
                                         b1, b2, c1, c2, 1e-8f);
  count_launch();
  pack_weights(net, st);
  double hs[2];
  if (cudaMemcpyAsync(hs, net->scal + 3, 2 * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    cudaGetLastError();
    return pc_fail(net, DDA_ERR_CUDA, "loss readback");
  }
  if (loss_out) *loss_out = hs[0] > 0.0 ? hs[1] / hs[0] : 0.0;
  return std::isfinite(hs[1]) ? DDA_OK : pc_fail(net, DDA_ERR_NONFINITE, "non-finite loss");
}

// Gradients of the last train step (host, nparam floats): for tests.
extern "C" int dda_pcnet_get_grads(dda_pcnet_t net, float* host) {
  if (!net || !host) return DDA_ERR_ARG;
  DeviceGuard dg(net->device);
  if (cudaMemcpy(host, net->g, net->nparam * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) {
    cudaGetLastError();
    return pc_fail(net, DDA_ERR_CUDA, "gradients to host");
  }
  return DDA_OK;
}

// ---------------------------------------------------------------- flexible Bi-CGSTAB
// Right-preconditioned Bi-CGSTAB whose preconditioner may change from one
// application to the next (the network): with p^ = N(p), s^ = N(s),
//   v = A p^, alpha = rho / (r0, v), s = r - alpha v, t = A s^,
//   omega = (t, s) / (t, t), x += alpha p^ + omega s^, r = s - omega t.
// Hermitian products (Sec. 2's Bi-CGSTAB), complex128 vectors, the exact
// product (double-float where the handle has the double-float D-matrix, else
// FP64).  Convergence is declared on the true residual b - A x.  When the
// preconditioned iteration stalls (its residual has not improved by 1 % in
// 50 iterations) or breaks down, the solve continues from the current x
// without the network: the plain solver is the fallback.
namespace dda {
namespace pc {

// per-block partials of (a, b) = sum conj(a) b for up to three pairs
__global__ void k_hdot3(const c128* __restrict__ a0, const c128* __restrict__ b0,
                        const c128* __restrict__ a1, const c128* __restrict__ b1,
                        const c128* __restrict__ a2, const c128* __restrict__ b2, long long n,
                        double* __restrict__ part) {
  __shared__ double sh[6][256];
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
    const c128* as[3] = {a0, a1, a2};
    const c128* bs[3] = {b0, b1, b2};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (!as[k]) continue;
      const c128 x = as[k][i], y = bs[k][i];
      acc[2 * k] += x.x * y.x + x.y * y.y;
      acc[2 * k + 1] += x.x * y.y - x.y * y.x;
    }
  }
  for (int k = 0; k < 6; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o)
      for (int k = 0; k < 6; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 6; ++k) part[6 * blockIdx.x + k] = sh[k][0];
}
__global__ void k_hdot_fin(const double* __restrict__ part, int nb, double* __restrict__ out) {
  if (threadIdx.x != 0) return;
  double s[6] = {0, 0, 0, 0, 0, 0};
  for (int b = 0; b < nb; ++b)
    for (int k = 0; k < 6; ++k) s[k] += part[6 * b + k];
  for (int k = 0; k < 6; ++k) out[k] = s[k];
}
// y = a x + b y + c z (complex scalars; z may be null)
__global__ void k_axpbypcz(c128 a, const c128* __restrict__ x, c128 b, c128* __restrict__ y, c128 c,
                           const c128* __restrict__ z, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    c128 r = a * x[i] + b * y[i];
    if (z) r = r + c * z[i];
    y[i] = r;
  }
}
// P = beta x (Eq. (3))
__global__ void k_p_from_x(const c128* __restrict__ x, c128* __restrict__ P, const uint8_t* __restrict__ mat,
                           const c128* __restrict__ beta, long long n_occ) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 3 * n_occ;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / n_occ);
    P[i] = beta[mat[i - c * n_occ] * 3 + c] * x[i];
  }
}

}  // namespace pc
}  // namespace dda

namespace {

struct PcRun {
  dda_t h;
  cudaStream_t st;
  long long n;
  bool df;
  double* part;
  double* out;     // device [6]
  double* hout;    // host [6]
};

int pc_matvec(PcRun& R, const c128* x, c128* y) {
  dda_t h = R.h;
  const cudaError_t e = R.df ? launch_matvec_df(h->g, h->lat(), h->wdf, h->w64.beta, h->n_mat, x, y, 1, R.st)
                             : launch_matvec<double>(h->g, h->lat(), h->w64, h->w64.beta, h->n_mat, x, y, 1,
                                                     false, R.st);
  return e == cudaSuccess ? DDA_OK : dda_cuda_fail(h, e, "product");
}

// up to three Hermitian products, read back to R.hout as (re, im) pairs
int pc_dots(PcRun& R, const c128* a0, const c128* b0, const c128* a1 = nullptr, const c128* b1 = nullptr,
            const c128* a2 = nullptr, const c128* b2 = nullptr) {
  k_hdot3<<<256, 256, 0, R.st>>>(a0, b0, a1, b1, a2, b2, R.n, R.part);
  count_launch();
  k_hdot_fin<<<1, 32, 0, R.st>>>(R.part, 256, R.out);
  count_launch();
  DDA_CK(R.h, cudaMemcpyAsync(R.hout, R.out, 6 * sizeof(double), cudaMemcpyDeviceToHost, R.st));
  DDA_CK(R.h, cudaStreamSynchronize(R.st));
  return DDA_OK;
}

c128 cplx(const double* p) { return mk<double>(p[0], p[1]); }
double cabs2h(c128 a) { return a.x * a.x + a.y * a.y; }
c128 cdivh(c128 a, c128 b) {
  const double d = b.x * b.x + b.y * b.y;
  return mk<double>((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

}  // namespace

extern "C" int dda_solve_pc(dda_t h, dda_pcnet_t net, const dda_solve_opts* o, const double* prop,
                            const double* pol, void* P_dev, double* hist, int hist_len,
                            dda_solve_info* info) {
  DDA_ON_DEVICE(h);
  if (!o || !prop || !pol || !P_dev || !info || (hist && hist_len < 1))
    return dda_fail(h, DDA_ERR_ARG, "bad dda_solve_pc arguments");
  if (net && net->device != h->device) return dda_fail(h, DDA_ERR_ARG, "network on another device");
  if (!(o->tol > 0.0) || o->maxiter < 1 || o->pol < DDA_CM || o->pol > DDA_CLDR)
    return dda_fail(h, DDA_ERR_ARG, "bad solver options");
  if (!h->w64.have_D) return dda_fail(h, DDA_ERR_STATE, "D-matrix not built");
  auto t0 = std::chrono::steady_clock::now();
  int rc = dda_beta_internal(h, o->pol, 1, prop, pol);
  if (rc != DDA_OK) return rc;
  PcRun R;
  R.h = h;
  R.st = h->stream;
  R.n = 3 * h->g.n_occ;
  R.df = h->wdf.have_D;
  if (R.df) {
    if ((rc = ensure_work_cap<df>(h, h->wdf, 1)) != DDA_OK) return rc;
  } else {
    if ((rc = ensure_d64(h)) != DDA_OK || (rc = ensure_work_cap<double>(h, h->w64, 1)) != DDA_OK) return rc;
  }
  const long long n = R.n;
  c128* buf = nullptr;
  double* dbuf = nullptr;
  if (dev_malloc(&buf, (size_t)10 * n * sizeof(c128)) != cudaSuccess ||
      dev_malloc(&dbuf, (size_t)(6 * 256 + 6) * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    dev_free(buf, R.st);
    return dda_fail(h, DDA_ERR_OOM, "preconditioned solver vectors");
  }
  double hout[6];
  R.part = dbuf;
  R.out = dbuf + 6 * 256;
  R.hout = hout;
  c128 *b = buf, *x = buf + n, *r = buf + 2 * n, *r0 = buf + 3 * n, *p = buf + 4 * n, *v = buf + 5 * n;
  c128 *s = buf + 6 * n, *t = buf + 7 * n, *ph = buf + 8 * n, *sh = buf + 9 * n;
  const int nbk = (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 8LL * num_sms()));
  const c128 one = mk<double>(1.0, 0.0), zero = mk<double>(0.0, 0.0);
  int status = DDA_NOT_CONVERGED, iters = 0, matvecs = 0, napps = 0, fallback = 0;
  double res_true = NAN, res_rec = NAN;
  std::vector<double> hv;
  hv.push_back(1.0);
  auto done = [&](int code) {
    dev_free(buf, R.st);
    dev_free(dbuf, R.st);
    return code;
  };
#define PCK(call) do { const int rc_ = (call); if (rc_ != DDA_OK) return done(rc_); } while (0)
  PCK(launch_rhs(h, b, h->w64.beta, 1, prop, pol, R.st));
  DDA_CK(h, cudaMemsetAsync(x, 0, n * sizeof(c128), R.st));
  DDA_CK(h, cudaMemcpyAsync(r, b, n * sizeof(c128), cudaMemcpyDeviceToDevice, R.st));
  PCK(pc_dots(R, b, b));
  const double bn = std::sqrt(hout[0]);
  bool use_net = net != nullptr;
  auto precond = [&](const c128* in, c128* out) -> int {
    if (use_net) {
      ++napps;
      return dda_pcnet_apply(net, h, in, out) == DDA_OK ? DDA_OK
                                                        : dda_fail(h, DDA_ERR_CUDA, "network: " + net->err);
    }
    const cudaError_t e = cudaMemcpyAsync(out, in, n * sizeof(c128), cudaMemcpyDeviceToDevice, R.st);
    return e == cudaSuccess ? DDA_OK : dda_cuda_fail(h, e, "copy");
  };
  if (!(bn > 0.0)) {
    status = std::isfinite(bn) ? DDA_OK : DDA_ERR_NONFINITE;
    res_true = res_rec = std::isfinite(bn) ? 0.0 : NAN;
  }
  double best = 1.0;
  int best_it = 0;
  while (status == DDA_NOT_CONVERGED && iters < o->maxiter) {
    // (re)start from the current x: r0 = r, p = v = 0, rho = alpha = omega = 1
    DDA_CK(h, cudaMemcpyAsync(r0, r, n * sizeof(c128), cudaMemcpyDeviceToDevice, R.st));
    DDA_CK(h, cudaMemsetAsync(p, 0, n * sizeof(c128), R.st));
    DDA_CK(h, cudaMemsetAsync(v, 0, n * sizeof(c128), R.st));
    c128 rho = one, alpha = one, omega = one;
    PCK(pc_dots(R, r0, r));
    c128 rho_new = cplx(hout);
    bool restart = false;
    while (!restart && iters < o->maxiter) {
      if (cabs2h(rho_new) == 0.0) { restart = true; break; }
      const c128 beta = cdivh(rho_new, rho) * cdivh(alpha, omega);
      rho = rho_new;
      // p = r + beta (p - omega v)
      k_axpbypcz<<<nbk, 256, 0, R.st>>>(one, r, beta, p, mk<double>(-(beta * omega).x, -(beta * omega).y), v, n);
      count_launch();
      PCK(precond(p, ph));
      PCK(pc_matvec(R, ph, v));
      ++matvecs;
      PCK(pc_dots(R, r0, v));
      const c128 rv = cplx(hout);
      if (cabs2h(rv) == 0.0) { restart = true; break; }
      alpha = cdivh(rho, rv);
      // s = r - alpha v
      DDA_CK(h, cudaMemcpyAsync(s, r, n * sizeof(c128), cudaMemcpyDeviceToDevice, R.st));
      k_axpbypcz<<<nbk, 256, 0, R.st>>>(mk<double>(-alpha.x, -alpha.y), v, one, s, zero, nullptr, n);
      count_launch();
      PCK(precond(s, sh));
      PCK(pc_matvec(R, sh, t));
      ++matvecs;
      PCK(pc_dots(R, t, s, t, t));
      const c128 ts = cplx(hout);
      const double tt = hout[2];
      omega = tt > 0.0 ? mk<double>(ts.x / tt, ts.y / tt) : zero;
      // x += alpha p^ + omega s^ ; r = s - omega t
      k_axpbypcz<<<nbk, 256, 0, R.st>>>(alpha, ph, one, x, omega, sh, n);
      count_launch();
      DDA_CK(h, cudaMemcpyAsync(r, s, n * sizeof(c128), cudaMemcpyDeviceToDevice, R.st));
      k_axpbypcz<<<nbk, 256, 0, R.st>>>(mk<double>(-omega.x, -omega.y), t, one, r, zero, nullptr, n);
      count_launch();
      ++iters;
      PCK(pc_dots(R, r, r, r0, r));
      const double res = std::sqrt(hout[0]) / bn;
      rho_new = cplx(hout + 2);
      res_rec = res;
      hv.push_back(res);
      if (!std::isfinite(res)) { status = DDA_ERR_NONFINITE; break; }
      if (res < best * 0.99) { best = res; best_it = iters; }
      if (res < o->tol) break;
      if (cabs2h(omega) == 0.0) { restart = true; break; }
      if (use_net && iters - best_it >= 50) {   // stalled: continue without the network
        use_net = false;
        fallback = iters;
        restart = true;
        best_it = iters;
      }
    }
    if (status != DDA_NOT_CONVERGED) break;
    // the judge: the true residual with the exact product
    PCK(pc_matvec(R, x, t));
    ++matvecs;
    DDA_CK(h, cudaMemcpyAsync(r, b, n * sizeof(c128), cudaMemcpyDeviceToDevice, R.st));
    k_axpbypcz<<<nbk, 256, 0, R.st>>>(mk<double>(-1.0, 0.0), t, one, r, zero, nullptr, n);
    count_launch();
    PCK(pc_dots(R, r, r));
    res_true = std::sqrt(hout[0]) / bn;
    if (!std::isfinite(res_true)) { status = DDA_ERR_NONFINITE; break; }
    if (res_true < o->tol) { status = DDA_OK; break; }
  }
  if (status == DDA_NOT_CONVERGED && std::isnan(res_true)) {
    PCK(pc_matvec(R, x, t));
    ++matvecs;
    DDA_CK(h, cudaMemcpyAsync(r, b, n * sizeof(c128), cudaMemcpyDeviceToDevice, R.st));
    k_axpbypcz<<<nbk, 256, 0, R.st>>>(mk<double>(-1.0, 0.0), t, one, r, zero, nullptr, n);
    count_launch();
    PCK(pc_dots(R, r, r));
    res_true = std::sqrt(hout[0]) / bn;
  }
  k_p_from_x<<<nbk, 256, 0, R.st>>>(x, (c128*)P_dev, h->d_mat, h->w64.beta, h->g.n_occ);
  count_launch();
  DDA_CK(h, cudaStreamSynchronize(R.st));
#undef PCK
  dda_solve_info& inf = info[0];
  inf = dda_solve_info{};
  inf.status = status;
  inf.iters = iters;
  inf.matvecs = matvecs;
  inf.matvecs_fp64 = matvecs;
  inf.outer = fallback;             // iteration at which the network was dropped (0: never)
  inf.rel_res_true = res_true;
  inf.rel_res_recur = res_rec;
  inf.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  if (hist)
    for (int i = 0; i < hist_len; ++i) hist[i] = i < (int)hv.size() ? hv[i] : -1.0;
  (void)napps;
  return done(status);
}

// ---------------------------------------------------------------- training pairs
namespace dda {
namespace pc {
// e = (Ps - Pk) / beta per dipole and component (beta = 0: e = 0)
__global__ void k_err_from_P(const c128* __restrict__ Ps, const c128* __restrict__ Pk,
                             const uint8_t* __restrict__ mat, const c128* __restrict__ beta,
                             long long n_occ, c128* __restrict__ e) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 3 * n_occ;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / n_occ);
    const c128 b = beta[mat[i - c * n_occ] * 3 + c];
    const double d = b.x * b.x + b.y * b.y;
    const c128 p = Ps[i] - Pk[i];
    e[i] = d > 0.0 ? mk<double>((p.x * b.x + p.y * b.y) / d, (p.y * b.x - p.x * b.y) / d)
                   : mk<double>(0.0, 0.0);
  }
}
}  // namespace pc
}  // namespace dda

extern "C" int dda_pcnet_pair(dda_t h, int pol_prescription, const double* prop_host,
                              const double* pol_host, const void* P_star, const void* P_k, void* r_out,
                              void* e_out) {
  DDA_ON_DEVICE(h);
  if (!prop_host || !pol_host || !P_star || !P_k || !r_out || !e_out)
    return dda_fail(h, DDA_ERR_ARG, "bad dda_pcnet_pair arguments");
  if (!h->w64.have_D) return dda_fail(h, DDA_ERR_STATE, "D-matrix not built");
  int rc = dda_beta_internal(h, pol_prescription, 1, prop_host, pol_host);
  if (rc != DDA_OK) return rc;
  const bool use_df = h->wdf.have_D;
  if (use_df) rc = ensure_work_cap<dda::df>(h, h->wdf, 1);
  else if ((rc = ensure_d64(h)) == DDA_OK) rc = ensure_work_cap<double>(h, h->w64, 1);
  if (rc != DDA_OK) return rc;
  const long long n = 3 * h->g.n_occ;
  k_err_from_P<<<(int)std::min<long long>((n + 255) / 256, 8LL * num_sms()), 256, 0, h->stream>>>(
      (const c128*)P_star, (const c128*)P_k, h->d_mat, h->w64.beta, h->g.n_occ, (c128*)e_out);
  count_launch();
  const cudaError_t e = use_df ? launch_matvec_df(h->g, h->lat(), h->wdf, h->w64.beta, h->n_mat,
                                                  (const c128*)e_out, (c128*)r_out, 1, h->stream)
                           : launch_matvec<double>(h->g, h->lat(), h->w64, h->w64.beta, h->n_mat,
                                                   (const c128*)e_out, (c128*)r_out, 1, false, h->stream);
  if (e != cudaSuccess) return dda_cuda_fail(h, e, "pair product");
  DDA_CK(h, cudaStreamSynchronize(h->stream));
  return DDA_OK;
}
