// Convolutions of the learned preconditioner on the tensor cores.
//
// Activations and gradients are FP32, the weights bf16.  A 24-bit float is the
// exact sum of three bf16 numbers (hi + mid + lo, 8 bits each), so a product
// with a bf16 weight is three bf16 products, each exact, and only the FP32
// sums round.  The tensor cores truncate where the FP32 pipe rounds, which
// would shrink every layer a little: the hi products of one tap and 16
// channels leave the tensor core after a single instruction and are summed on
// the FP32 pipe (4 additions to 3 matrix instructions); the mid and lo
// products, 256 times smaller, accumulate over the 9 taps of a z plane.
//
// The convolution is an implicit matrix product: rows are voxels, columns
// output channels, the inner dimension is 16 input channels of one tap.
// Activations live in global memory already split, as 16-byte units of 8
// channels, [8-channel block][part][voxel]: the kernel that produces a value
// splits it once instead of every tile that reads it (with halos and output
// blocks about six), and a tile with its halo arrives by 16-byte asynchronous
// copies in the layout it is used from, [part][half][voxel], where the rows of
// a tap are ldmatrix rows at a shifted voxel and eight neighbours in x fill
// the 32 banks.  The weights come in fragment order (packed when they change).
// Each warp holds MT tiles of 16 voxels (two x rows of 8) by NT tiles of 8
// channels; several blocks share an SM, so that copies of one run under the
// matrix instructions of another.  Where the layer has too few tiles for that
// (1/8 resolution), KG groups of 4 warps in a block take every KG-th 16
// channels each and their sums are added at the end.
//
// 128^3 sphere (31 GFLOP a pass, 93 with the three products): 2.09 ms of
// convolutions on the FP32 pipe; on the tensor cores 0.38 ms when every tile
// split the FP32 channels it read, 0.33 ms now (48 to 16 channels at 64^3 voxels
// 435, 121 and 96 us, 160 to 160 at 16^3 69 and 53 us between the last two);
// the matrix pipe is 60 to 66 % busy in the large layers.  The pass 2.36, 0.50
// and 0.45 ms; error of N(r) against 64 bits 4.5e-7 before, 1.4e-7 now.
#pragma once

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "internal.h"

namespace dda {
namespace pc {

struct Dims {
  int x, y, z;
  __host__ __device__ long long n() const { return (long long)x * y * z; }
};
inline Dims halved(Dims d) { return {(d.x + 1) / 2, (d.y + 1) / 2, (d.z + 1) / 2}; }

// Input of a convolution: channels [0, ca) from a (planar [ca][voxels]; at
// half resolution, nearest, when up), channels [ca, ca + cb) from b.  ca is a
// multiple of 16 when cb > 0.
struct ConvIn {
  const float* a;
  int ca;
  Dims da;
  bool up;
  const float* b;
  int cb;
};

__device__ __forceinline__ void cp4(void* smem, const float* gmem, bool ok) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int n = ok ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp16(void* smem, const void* gmem, bool ok) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void ldm4(unsigned (&r)[4], const void* smem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(sa) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// x = hi + mid + lo, exact for floats of 2^-110 and more (below, mid and lo are
// subnormal bf16: to within 2^-134).  What rounds beyond bf16's largest number is
// truncated; infinity is hi alone (its remainder would be NaN, which the relu of
// the next layer turns into 0).
__device__ __forceinline__ void split3(float x, __nv_bfloat16 (&s)[3]) {
  const unsigned u = __float_as_uint(x);
  const unsigned m = u & 0x7fffffffu;
  const bool inf = m == 0x7f800000u;
  s[0] = m >= 0x7f7f8000u && m <= 0x7f800000u ? __ushort_as_bfloat16((unsigned short)(u >> 16)) : __float2bfloat16_rn(x);
  const float r = inf ? 0.0f : x - __bfloat162float(s[0]);
  s[1] = __float2bfloat16_rn(r);
  s[2] = __float2bfloat16_rn(r - __bfloat162float(s[1]));
}
// 8 floats as three units of 8 bf16, and back (exact)
__device__ __forceinline__ void split_unit(const float (&f)[8], uint4 (&u)[3]) {
  __nv_bfloat16 s[3][8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    __nv_bfloat16 t[3];
    split3(f[c], t);
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k][c] = t[k];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) u[k] = *reinterpret_cast<const uint4*>(s[k]);
}
__device__ __forceinline__ void join_unit(const uint4 (&u)[3], float (&f)[8]) {
  const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&u[0]);
  const __nv_bfloat16* m = reinterpret_cast<const __nv_bfloat16*>(&u[1]);
  const __nv_bfloat16* l = reinterpret_cast<const __nv_bfloat16*>(&u[2]);
#pragma unroll
  for (int c = 0; c < 8; ++c) f[c] = (__bfloat162float(h[c]) + __bfloat162float(m[c])) + __bfloat162float(l[c]);
}
// 2 floats as three pairs of bf16
__device__ __forceinline__ void split_pair(float a, float b, unsigned (&u)[3]) {
  __nv_bfloat16 s[3], t[3];
  split3(a, s);
  split3(b, t);
#pragma unroll
  for (int k = 0; k < 3; ++k)
    u[k] = (unsigned)__bfloat16_as_ushort(s[k]) | (unsigned)__bfloat16_as_ushort(t[k]) << 16;
}

// Input of a convolution of the apply pass: split units as ConvIn's arrays (ca
// and cb multiples of 16), or, for the first layer, FP32 channels f (at most
// 16, split as they are staged).
struct SplitIn {
  const uint4* a;
  int ca;
  Dims da;
  bool up;
  const uint4* b;
  int cb;
  const float* f;
  int cf;
};
// Output: split units, or FP32 channels (the last layer)
struct SplitOut {
  uint4* s;
  float* f;
};

// Voxel tile of 8 x 4 x TZ and its halo for kernels of K^3 taps
template <int K, int TZ> struct Tile {
  static constexpr int H = K / 2, HX = 8 + 2 * H, HY = 4 + 2 * H, HZ = TZ + 2 * H, HV = HX * HY * HZ;
};

// out[co][v] = bias[co] + sum_ci sum_t w[co][ci][t] in[ci][v + t - H], then
// relu.  wp: packed weights [16-channel block][tap][8-channel tile][lane]; grid
// (voxel tiles, output-channel blocks of 8 NT); 4 KG warps.  FIN: the input is
// FP32 channels (one block of 16), else split units.
template <int K, int MT, int NT, int KG, bool FIN>
__global__ void __launch_bounds__(128 * KG) k_conv_mma(SplitIn in, const uint2* __restrict__ wp, int ntn,
                                                       const float* __restrict__ bias, SplitOut out,
                                                       int cout, Dims d, int relu) {
  constexpr int TZ = 2 * MT, K3 = K * K * K;
  using T = Tile<K, TZ>;
  constexpr int NV = (T::HV + 127) / 128;      // halo voxels per thread
  constexpr int GB = 6 * T::HV * 16 + K3 * NT * 256;       // shared memory of a group
  static_assert(MT * NT * 4 * 128 * 4 <= GB, "a group's sums fit its buffers");
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x & 127, grp = threadIdx.x >> 7, lane = threadIdx.x & 31, warp = tid >> 5;
  uint4* s_t = reinterpret_cast<uint4*>(smem + grp * GB);                 // [3][2][HV]
  uint2* s_w = reinterpret_cast<uint2*>(s_t + 6 * T::HV);                 // [K3][NT][32]
  const int ntx = (d.x + 7) / 8, nty = (d.y + 3) / 4;
  const int tx0 = (blockIdx.x % ntx) * 8, ty0 = ((blockIdx.x / ntx) % nty) * 4,
            tz0 = (blockIdx.x / (ntx * nty)) * TZ;
  const long long nv = d.n(), na = in.up ? in.da.n() : nv;
  const int nblk = FIN ? 1 : (in.ca + in.cb) / 16;
  // this thread's halo voxels: index in b (fine) and in a, -1 outside
  int vf[NV], va[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int hv = tid + 128 * i;
    const int x = tx0 + hv % T::HX - T::H, y = ty0 + (hv / T::HX) % T::HY - T::H,
              z = tz0 + hv / (T::HX * T::HY) - T::H;
    const bool ok = hv < T::HV && x >= 0 && y >= 0 && z >= 0 && x < d.x && y < d.y && z < d.z;
    vf[i] = ok ? (z * d.y + y) * d.x + x : -1;
    va[i] = !ok ? -1 : in.up ? ((z / 2) * in.da.y + y / 2) * in.da.x + x / 2 : vf[i];
  }
  auto group_sync = [&] {
    if constexpr (KG == 1) __syncthreads();
    else asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory");
  };
  float acc[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[i][n][k] = 0.0f;
  // ldmatrix row of this lane for tile i at tap (0, 0, 0)
  int row[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int m = warp * MT + i;               // z = m / 2, rows y = 2 (m % 2) and + 1
    row[i] = ((m >> 1) * T::HY + 2 * (m & 1) + ((lane >> 3) & 1)) * T::HX + (lane & 7) + (lane >> 4) * T::HV;
  }
  for (int blk = grp; blk < nblk; blk += KG) {
    if (blk >= KG) group_sync();               // the previous channels' products are done
    const uint2* sw = wp + ((long long)blk * K3 * ntn + blockIdx.y * NT) * 32;
    for (int i = tid; i < K3 * NT * 16; i += 128) {                  // 16-byte pieces
      const int t = i / (NT * 16), r = i - t * NT * 16;
      cp16(s_w + t * NT * 32 + 2 * r, sw + (long long)t * ntn * 32 + 2 * r, true);
    }
    if constexpr (FIN) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int hv = tid + 128 * i;
        if (hv < T::HV) {
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            float f[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) f[c] = vf[i] >= 0 && 8 * half + c < in.cf ? in.f[(8 * half + c) * nv + vf[i]] : 0.0f;
            uint4 u[3];
            split_unit(f, u);
#pragma unroll
            for (int k = 0; k < 3; ++k) s_t[(2 * k + half) * T::HV + hv] = u[k];
          }
        }
      }
    } else {
      const bool fa = 16 * blk < in.ca;
      const long long cs = fa ? na : nv;       // units of a part of 8 channels
      const uint4* src = fa ? in.a + 6LL * blk * cs : in.b + 6LL * (blk - in.ca / 16) * cs;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int hv = tid + 128 * i, v = fa ? va[i] : vf[i];
        if (hv < T::HV) {
#pragma unroll
          for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int k = 0; k < 3; ++k)
              cp16(s_t + (2 * k + half) * T::HV + hv, v >= 0 ? src + (3 * half + k) * cs + v : in.a, v >= 0);
        }
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    group_sync();
    const uint2* wb = s_w + lane;
#pragma unroll 1
    for (int kz = 0; kz < K; ++kz) {
      float lo[MT][NT][4];
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) lo[i][n][k] = 0.0f;
#pragma unroll
      for (int t = 0; t < K * K; ++t) {
        uint2 b[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) b[n] = wb[((kz * K * K + t) * NT + n) * 32];
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          const uint4* p = s_t + row[i] + (kz * T::HY + t / K) * T::HX + t % K;
          unsigned a0[4], a1[4], a2[4];
          ldm4(a0, p);
          ldm4(a1, p + 2 * T::HV);
          ldm4(a2, p + 4 * T::HV);
#pragma unroll
          for (int n = 0; n < NT; ++n) mma_bf16(lo[i][n], a2, b[n].x, b[n].y);
          float hi[NT][4];
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            hi[n][0] = hi[n][1] = hi[n][2] = hi[n][3] = 0.0f;
            mma_bf16(hi[n], a0, b[n].x, b[n].y);
          }
#pragma unroll
          for (int n = 0; n < NT; ++n) mma_bf16(lo[i][n], a1, b[n].x, b[n].y);
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[i][n][k] += hi[n][k];
        }
      }
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[i][n][k] += lo[i][n][k];
    }
  }
  if constexpr (KG > 1) {                      // the groups' sums, in order
    float* s_a = reinterpret_cast<float*>(smem + grp * GB);
    group_sync();
    if (grp > 0) {
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) s_a[((i * NT + n) * 4 + k) * 128 + tid] = acc[i][n][k];
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int g = 1; g < KG; ++g) {
      const float* p = reinterpret_cast<const float*>(smem + g * GB);
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[i][n][k] += p[((i * NT + n) * 4 + k) * 128 + tid];
    }
  }
  // accumulator (row r, columns c, c + 1): x = r, output channels c, c + 1
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int m = warp * MT + i;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int x = tx0 + (lane >> 2), y = ty0 + 2 * (m & 1) + h, z = tz0 + (m >> 1);
      if (x < d.x && y < d.y && z < d.z) {
        const long long v = ((long long)z * d.y + y) * d.x + x;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const int cb = blockIdx.y * NT + n, co = cb * 8 + (lane & 3) * 2;
          if (co < cout) {                     // cout is even
            float r[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              r[e] = acc[i][n][2 * h + e] + bias[co + e];
              if (relu) r[e] = fmaxf(r[e], 0.0f);
            }
            if (out.s) {
              unsigned u[3];
              split_pair(r[0], r[1], u);
#pragma unroll
              for (int k = 0; k < 3; ++k)
                reinterpret_cast<unsigned*>(out.s + (3LL * cb + k) * nv + v)[lane & 3] = u[k];
            } else {
              out.f[co * nv + v] = r[0];
              out.f[(co + 1) * nv + v] = r[1];
            }
          }
        }
      }
    }
  }
}

// Weights in fragment order, all layers in one launch: entry of layer L's
// forward product (output channels co, input ci) or of its input gradient
// (output ci, input co, taps reversed).
struct PackItem { int w, cin, cout, k3, flip, at, n; };   // weights from w; n elements from at
struct PackList { PackItem item[14]; int count; };
__global__ void k_pack_weights(const __nv_bfloat16* __restrict__ w, const __grid_constant__ PackList pl,
                               uint2* __restrict__ out, int total) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    int q = 0;
    while (q + 1 < pl.count && i >= pl.item[q + 1].at) ++q;
    const PackItem& p = pl.item[q];
    const int ni = p.flip ? p.cout : p.cin, no = p.flip ? p.cin : p.cout, ntn = (no + 7) / 8;
    int j = i - p.at;
    const int lane = j & 31;
    j >>= 5;
    const int nt = j % ntn;
    j /= ntn;
    const int t = j % p.k3, blk = j / p.k3;
    const int o = nt * 8 + (lane >> 2);
    unsigned r[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      unsigned u = 0;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int c = blk * 16 + b * 8 + (lane & 3) * 2 + e;
        if (c < ni && o < no) {
          const int at = p.flip ? (c * p.cin + o) * p.k3 + (p.k3 - 1 - t) : (o * p.cin + c) * p.k3 + t;
          u |= (unsigned)__bfloat16_as_ushort(w[p.w + at]) << (16 * e);
        }
      }
      r[b] = u;
    }
    out[i] = make_uint2(r[0], r[1]);
  }
}

template <int K, int MT, int NT, int KG, bool FIN>
cudaError_t conv_mma_t(const SplitIn& in, const uint2* wp, const float* bias, const SplitOut& out, int cout, Dims d,
                       int relu, cudaStream_t st) {
  using T = Tile<K, 2 * MT>;
  const size_t sm = (size_t)KG * (T::HV * 6 * 16 + (size_t)K * K * K * NT * 256);
  auto kernel = k_conv_mma<K, MT, NT, KG, FIN>;
  cudaError_t e = ensure_smem((const void*)kernel, sm);
  if (e == cudaSuccess) e = ensure_carveout_max((const void*)kernel);
  if (e != cudaSuccess) return e;
  const int ntn = (cout + 7) / 8;
  const int tiles = ((d.x + 7) / 8) * ((d.y + 3) / 4) * ((d.z + 2 * MT - 1) / (2 * MT));
  kernel<<<dim3(tiles, (ntn + NT - 1) / NT), 128 * KG, sm, st>>>(in, wp, ntn, bias, out, cout, d, relu);
  count_launch();
  return cudaGetLastError();
}

// Tile of a convolution (K = 3): 128 or 64 voxels by 40, 32, 16 or 8 output
// channels, in 1, 2 or 4 groups; the one with the least estimated time.  Per 16
// channels a block issues 324 MT NT matrix instructions, half a one a clock
// when several groups share an SM (the small tiles up to twice that long: they
// load more fragments per instruction); alone a group takes twice as long, and
// about 1,500 clocks more for its copies.
inline cudaError_t conv_mma(int K, const SplitIn& in, const uint2* wp, const float* bias, const SplitOut& out,
                            int cout, Dims d, int relu, cudaStream_t st) {
  if (K == 1) return conv_mma_t<1, 2, 1, 1, false>(in, wp, bias, out, cout, d, relu, st);
  if (in.f) return conv_mma_t<3, 2, 2, 1, true>(in, wp, bias, out, cout, d, relu, st);
  const int nblk = (in.ca + in.cb) / 16;
  auto cost = [&](int mt, int nt, int kg, int resident, double load) {
    if (cout % (8 * nt) != 0) return 1e30;
    const long long b = (long long)((d.x + 7) / 8) * ((d.y + 3) / 4) * ((d.z + 2 * mt - 1) / (2 * mt)) * (cout / (8 * nt));
    const double per = (double)((b + num_sms() - 1) / num_sms());
    const double mma = 648.0 * mt * nt * load, alone = (nblk + kg - 1) / kg * (2.0 * mma + 1500.0);
    return std::max(std::ceil(per / resident) * alone, per * nblk * mma * 1.2);
  };
  const double c[6] = {cost(2, 4, 1, 2, 1.0), cost(2, 5, 2, 1, 1.0), cost(2, 4, 2, 1, 1.0),
                       cost(2, 2, 1, 4, 1.1), cost(1, 2, 2, 2, 1.4), cost(1, 1, 4, 1, 2.0)};
  switch ((int)(std::min_element(c, c + 6) - c)) {
    case 0: return conv_mma_t<3, 2, 4, 1, false>(in, wp, bias, out, cout, d, relu, st);
    case 1: return conv_mma_t<3, 2, 5, 2, false>(in, wp, bias, out, cout, d, relu, st);
    case 2: return conv_mma_t<3, 2, 4, 2, false>(in, wp, bias, out, cout, d, relu, st);
    case 3: return conv_mma_t<3, 2, 2, 1, false>(in, wp, bias, out, cout, d, relu, st);
    case 4: return conv_mma_t<3, 1, 2, 2, false>(in, wp, bias, out, cout, d, relu, st);
  }
  return conv_mma_t<3, 1, 1, 4, false>(in, wp, bias, out, cout, d, relu, st);
}

// ---------------------------------------------------------------- training
// A training step is a chain of decisions: a difference of one rounding flips a
// relu or the bf16 rounding of a weight and shows in later gradients at 1e-5.
// So training keeps one order for every sum, on the FP32 pipe: an output is
// bias, then channel by channel, tap by tap, one fused multiply-add each.
// Pairs of outputs run in the paired instruction (each half rounds as the
// scalar one).  On small lattices a sum is one long dependent chain: what
// helps is every SM busy, operands copied ahead and few instructions per tap.
// 64 x 45 x 37 ellipsoid: training step 2.60 -> 0.82 ms, same bits.

// a thread's CO outputs at one voxel, pairwise
__device__ __forceinline__ unsigned long long pair2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpair2(unsigned long long r) {
  float2 o;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
  return o;
}

// out[co][v] = bias[co] + sum_ci sum_t w[co][ci][t] in[ci][v + t - H], then
// relu, or zero where mask[co][v] <= 0 (gradient behind a relu), from FP32
// copies of the weights wf [ci][t][coutp].  A warp
// takes the 8 x 4 voxels of a z plane and CO channels; 4 warps: ZW planes by
// 4 / ZW channel groups (8 channels per block).  Eight input channels with
// their halo and weights are copied while the eight before are summed.
template <int K, int ZW, int CO>
__global__ void __launch_bounds__(128) k_conv_f32(ConvIn in, const float* __restrict__ wf, int coutp,
                                                  const float* __restrict__ bias,
                                                  const float* __restrict__ mask,
                                                  float* __restrict__ out, int cout, Dims d, int relu) {
  using T = Tile<K, ZW>;
  constexpr int K3 = K * K * K, CB = 8, NB = 8, NV = (T::HV + 127) / 128;
  static_assert(CO * (4 / ZW) == NB, "8 channels per block");
  // rows in x are 24 floats apart, two channels to a row: the four rows of a warp
  // fill the 32 banks.  The weights of a warp's CO channels lie together, tap by
  // tap, so that 16 bytes are one tap of 4 channels or two taps of 2.
  constexpr int P = 24, PV = T::HY * T::HZ * P, KP = K3 + 1;
  __shared__ __align__(16) float s_in[2][CB / 2][PV];
  __shared__ __align__(16) float s_w[2][CB][NB / CO][KP * CO];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wz = warp % ZW, cg = warp / ZW;
  const int ntx = (d.x + 7) / 8, nty = (d.y + 3) / 4;
  const int tx0 = (blockIdx.x % ntx) * 8, ty0 = ((blockIdx.x / ntx) % nty) * 4,
            tz0 = (blockIdx.x / (ntx * nty)) * ZW;
  const int co0 = blockIdx.y * NB;
  const long long nv = d.n(), na = in.up ? in.da.n() : nv;
  const int cin = in.ca + in.cb, nblk = (cin + CB - 1) / CB;
  int vf[NV], va[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int hv = threadIdx.x + 128 * i;
    const int x = tx0 + hv % T::HX - T::H, y = ty0 + (hv / T::HX) % T::HY - T::H,
              z = tz0 + hv / (T::HX * T::HY) - T::H;
    const bool ok = hv < T::HV && x >= 0 && y >= 0 && z >= 0 && x < d.x && y < d.y && z < d.z;
    vf[i] = ok ? (z * d.y + y) * d.x + x : -1;
    va[i] = !ok ? -1 : in.up ? ((z / 2) * in.da.y + y / 2) * in.da.x + x / 2 : vf[i];
  }
  auto fetch = [&](int blk) {
    const int c0 = blk * CB, b = blk & 1;
    const bool fa = c0 < in.ca;
    const float* src = fa ? in.a + (long long)c0 * na : in.b + (long long)(c0 - in.ca) * nv;
    const long long cs = fa ? na : nv;
    const int lim = (fa ? in.ca : cin) - c0;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int hv = threadIdx.x + 128 * i, v = fa ? va[i] : vf[i];
      if (hv < T::HV) {
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          const bool ok = v >= 0 && c < lim;
          cp4(&s_in[b][c >> 1][(hv / T::HX) * P + hv % T::HX + (c & 1) * (P / 2)], ok ? src + c * cs + v : in.a, ok);
        }
      }
    }
    const int nc = min(CB, cin - c0);
    for (int i = threadIdx.x; i < nc * K3 * 2; i += 128) {           // 16-byte pieces
      const int h = i & 1, c = (i >> 1) / K3, t = (i >> 1) - c * K3;
      const float* g = wf + ((long long)c0 * K3 + (i >> 1)) * coutp + co0 + 4 * h;
      if constexpr (CO == 2) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const unsigned sa = (unsigned)__cvta_generic_to_shared(&s_w[b][c][2 * h + e][t * CO]);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(g + 2 * e) : "memory");
        }
      } else {
        const unsigned sa = (unsigned)__cvta_generic_to_shared(CO == 4 ? &s_w[b][c][h][t * CO] : &s_w[b][c][0][t * CO + 4 * h]);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(g) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  // pairs for 8 channels; fewer run the scalar instruction, whose result is
  // back sooner (with few warps the chain of a sum is what takes the time)
  constexpr bool PAIRS = CO == 8;
  unsigned long long acc2[PAIRS ? CO / 2 : 1];
  float acc[CO];
#pragma unroll
  for (int k = 0; k < CO; ++k) {
    const int co = co0 + cg * CO + k;
    acc[k] = bias && co < cout ? bias[co] : 0.0f;
  }
  if constexpr (PAIRS) {
#pragma unroll
    for (int k = 0; k < CO / 2; ++k) acc2[k] = pair2(acc[2 * k], acc[2 * k + 1]);
  }
  const int hv0 = (wz * T::HY + (lane >> 3)) * P + (lane & 7);
  fetch(0);
  for (int blk = 0; blk < nblk; ++blk) {
    __syncthreads();                         // the sums over the buffer fetched next are done
    if (blk + 1 < nblk) {
      fetch(blk + 1);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    const int nc = min(CB, cin - blk * CB), b = blk & 1;
#pragma unroll 1
    for (int c = 0; c < nc; ++c) {
      const float* si = &s_in[b][c >> 1][hv0 + (c & 1) * (P / 2)];
      const float* sw = &s_w[b][c][cg][0];
      float4 w2 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int t = 0; t < K3; ++t) {
        const float v = si[((t / (K * K)) * T::HY + (t / K) % K) * P + t % K];
        if constexpr (PAIRS) {
          const unsigned long long vv = pair2(v, v);
          const unsigned long long* w = reinterpret_cast<const unsigned long long*>(sw + t * CO);
#pragma unroll
          for (int k = 0; k < CO / 2; ++k) fma2(acc2[k], w[k], vv);
        } else {
          if (CO == 4 || t % 2 == 0) w2 = *reinterpret_cast<const float4*>(sw + t * CO);
          const float w[4] = {w2.x, w2.y, w2.z, w2.w};
#pragma unroll
          for (int k = 0; k < CO; ++k) acc[k] = fmaf(w[CO == 2 && t % 2 ? 2 + k : k], v, acc[k]);
        }
      }
    }
  }
  if constexpr (PAIRS) {
#pragma unroll
    for (int k = 0; k < CO / 2; ++k) {
      const float2 r = unpair2(acc2[k]);
      acc[2 * k] = r.x;
      acc[2 * k + 1] = r.y;
    }
  }
  const int x = tx0 + (lane & 7), y = ty0 + (lane >> 3), z = tz0 + wz;
  if (x >= d.x || y >= d.y || z >= d.z) return;
  const long long v = ((long long)z * d.y + y) * d.x + x;
#pragma unroll
  for (int k = 0; k < CO; ++k) {
    const int co = co0 + cg * CO + k;
    if (co < cout) {
      float r = acc[k];
      if (relu) r = fmaxf(r, 0.0f);
      if (mask && !(mask[co * nv + v] > 0.0f)) r = 0.0f;
      out[co * nv + v] = r;
    }
  }
}

// FP32 weights [ci][t][coutp] of every layer's forward product and of its
// input gradient (input co, output ci, taps reversed); n floats from at
__global__ void k_pack_f32(const __nv_bfloat16* __restrict__ w, const __grid_constant__ PackList pl,
                           float* __restrict__ out, int total) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    int q = 0;
    while (q + 1 < pl.count && i >= pl.item[q + 1].at) ++q;
    const PackItem& p = pl.item[q];
    const int no = p.flip ? p.cin : p.cout, nop = (no + 7) / 8 * 8;
    const int j = i - p.at, r0 = j / nop, o = j - r0 * nop, c = r0 / p.k3, t = r0 - c * p.k3;
    float r = 0.0f;
    if (o < no)
      r = __bfloat162float(w[p.w + (p.flip ? (c * p.cin + o) * p.k3 + (p.k3 - 1 - t)
                                           : (o * p.cin + c) * p.k3 + t)]);
    out[i] = r;
  }
}

template <int K, int ZW, int CO>
cudaError_t conv_f32_t(const ConvIn& in, const float* wf, const float* bias, const float* mask, float* out,
                       int cout, Dims d, int relu, cudaStream_t st) {
  const int tiles = ((d.x + 7) / 8) * ((d.y + 3) / 4) * ((d.z + ZW - 1) / ZW), cb = (cout + 7) / 8;
  k_conv_f32<K, ZW, CO><<<dim3(tiles, cb), 128, 0, st>>>(in, wf, 8 * cb, bias, mask, out, cout, d, relu);
  count_launch();
  return cudaGetLastError();
}

// 128, 64 or 32 voxels per block: the least rounds of blocks over the SMs
// times instructions per tap (8, 5.5 and 4.5 with their loads).  Of the layers
// at 1/4 and 1/8 resolution, 31 us with the 64-voxel tile this picks and 42 with
// the 32-voxel one (one round of blocks against two).
inline cudaError_t conv_f32(int K, const ConvIn& in, const float* wf, const float* bias, const float* mask,
                            float* out, int cout, Dims d, int relu, cudaStream_t st) {
  if (K == 1) return conv_f32_t<1, 1, 2>(in, wf, bias, mask, out, cout, d, relu, st);
  auto cost = [&](int zw, double tap) {
    const long long b = (long long)((d.x + 7) / 8) * ((d.y + 3) / 4) * ((d.z + zw - 1) / zw) * ((cout + 7) / 8);
    return (double)((b + num_sms() - 1) / num_sms()) * tap;
  };
  const double a = cost(4, 8.0), b = cost(2, 5.5), c = cost(1, 4.5);
  if (a <= b && a <= c) return conv_f32_t<3, 4, 8>(in, wf, bias, mask, out, cout, d, relu, st);
  if (b <= c) return conv_f32_t<3, 2, 4>(in, wf, bias, mask, out, cout, d, relu, st);
  return conv_f32_t<3, 1, 2>(in, wf, bias, mask, out, cout, d, relu, st);
}

// ---------------------------------------------------------------- weight gradients
// part[chunk][t][co][ci] = sum over the voxels of this chunk's tiles (8 x 8 x 4
// voxels, in order; void voxels count as zeros) of gout[co][v] in[ci][v + t - H].
// A block takes 8 output and 16 input channels, a thread one tap and 4 x 4 of
// their sums: 2 shared-memory loads for 8 paired multiply-adds.  grid (chunks,
// output-channel blocks, input-channel blocks), 216 threads.
constexpr int kWX = 8, kWY = 8, kWZ = 4, kWV = kWX * kWY * kWZ;
constexpr int kWHX = kWX + 2, kWHY = kWY + 2, kWHV = kWHX * kWHY * (kWZ + 2);
// halo rows are 11 voxels apart in shared memory: taps t and t + 1 are then an
// odd number of 64-byte voxels apart, and a quarter warp (two taps) reads all
// 32 banks
constexpr int kWPX = kWX + 3, kWPV = kWPX * kWHY * (kWZ + 2);
constexpr int kWTile = kWPV * 16 + kWV * 8;               // floats of a tile: [halo voxel][16], [voxel][8]
__global__ void __launch_bounds__(216) k_wgrad_f32(ConvIn in, const float* __restrict__ gout, int cout,
                                                   Dims d, float* __restrict__ part, int tiles_per_chunk) {
  extern __shared__ __align__(16) float smem_w[];          // two tiles: one arrives while one is summed
  const int ntx = (d.x + kWX - 1) / kWX, nty = (d.y + kWY - 1) / kWY, ntz = (d.z + kWZ - 1) / kWZ;
  const int ntiles = ntx * nty * ntz, co0 = blockIdx.y * 8, c0 = blockIdx.z * 16, cin = in.ca + in.cb;
  const long long nv = d.n(), na = in.up ? in.da.n() : nv;
  const bool fa = c0 < in.ca, up = fa && in.up;
  const float* src = fa ? in.a + (long long)c0 * na : in.b + (long long)(c0 - in.ca) * nv;
  const long long cs = fa ? na : nv;
  const int lim = (fa ? in.ca : cin) - c0;
  const int cig = threadIdx.x & 3, t = (threadIdx.x >> 2) % 27, cog = threadIdx.x / 108;
  const int hv0 = ((t / 9) * kWHY + (t / 3) % 3) * kWPX + t % 3;
  // a quarter warp copies 8 voxels of a channel, the four quarters four channels
  auto fetch = [&](int tile, float* buf) {
    const int tx0 = (tile % ntx) * kWX, ty0 = ((tile / ntx) % nty) * kWY, tz0 = (tile / (ntx * nty)) * kWZ;
    for (int i = threadIdx.x; i < kWHV * 4; i += 216) {
      const int q = i & 3, hv = i >> 2;
      const int x = tx0 + hv % kWHX - 1, y = ty0 + (hv / kWHX) % kWHY - 1, z = tz0 + hv / (kWHX * kWHY) - 1;
      const bool ok = x >= 0 && y >= 0 && z >= 0 && x < d.x && y < d.y && z < d.z;
      const long long v = up ? ((long long)(z / 2) * in.da.y + y / 2) * in.da.x + x / 2
                             : ((long long)z * d.y + y) * d.x + x;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int ch = 4 * c + q;
        const bool k = ok && ch < lim;
        cp4(buf + (hv / kWHX * kWPX + hv % kWHX) * 16 + ch, k ? src + ch * cs + v : in.a, k);
      }
    }
    float* g = buf + kWPV * 16;
    for (int i = threadIdx.x; i < kWV * 4; i += 216) {
      const int q = i & 3, u = i >> 2;
      const int x = tx0 + u % kWX, y = ty0 + (u / kWX) % kWY, z = tz0 + u / (kWX * kWY);
      const bool ok = x < d.x && y < d.y && z < d.z;
      const long long v = ((long long)z * d.y + y) * d.x + x;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int co = 4 * c + q;
        const bool k = ok && co0 + co < cout;
        cp4(g + u * 8 + co, k ? gout + (co0 + co) * nv + v : gout, k);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  unsigned long long acc[4][2];                // [output channel][pair of input channels]
#pragma unroll
  for (int k = 0; k < 4; ++k) acc[k][0] = acc[k][1] = 0ull;
  const int t0 = blockIdx.x * tiles_per_chunk, t1 = min(ntiles, t0 + tiles_per_chunk);
  if (t0 < t1) fetch(t0, smem_w);
  for (int tile = t0; tile < t1; ++tile) {
    const float* buf = smem_w + ((tile - t0) & 1) * kWTile;
    __syncthreads();                           // the sums over the buffer fetched next are done
    if (tile + 1 < t1) {
      fetch(tile + 1, smem_w + ((tile + 1 - t0) & 1) * kWTile);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    for (int r = 0; r < kWY * kWZ; ++r) {
      const float* a = buf + (hv0 + ((r / kWY) * kWHY + r % kWY) * kWPX) * 16 + 4 * cig;
      const float* g = buf + kWPV * 16 + r * kWX * 8 + 4 * cog;
#pragma unroll
      for (int u = 0; u < kWX; ++u) {
        const ulonglong2 x2 = *reinterpret_cast<const ulonglong2*>(a + 16 * u);
        const float4 gv = *reinterpret_cast<const float4*>(g + 8 * u);
        const float gs_[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const unsigned long long gg = pair2(gs_[k], gs_[k]);
          fma2(acc[k][0], gg, x2.x);
          fma2(acc[k][1], gg, x2.y);
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float2 r = unpair2(acc[k][e]);
      const int co = co0 + 4 * cog + k, ci = c0 + 4 * cig + 2 * e;
      float* p = part + (((long long)blockIdx.x * 27 + t) * cout + co) * cin + ci;
      if (co < cout && ci < cin) p[0] = r.x;
      if (co < cout && ci + 1 < cin) p[1] = r.y;
    }
}

// The same for K = 1 and at most 6 x 16 channels: one thread per weight
__global__ void __launch_bounds__(96) k_wgrad1(const float* __restrict__ in, int cin,
                                               const float* __restrict__ gout, int cout, Dims d,
                                               float* __restrict__ part, int tiles_per_chunk) {
  __shared__ float s_a[16][kWV + 1], s_g[6][kWV + 1];
  const int ntx = (d.x + kWX - 1) / kWX, nty = (d.y + kWY - 1) / kWY, ntz = (d.z + kWZ - 1) / kWZ;
  const int ntiles = ntx * nty * ntz, co = threadIdx.x / 16, ci = threadIdx.x % 16;
  const long long nv = d.n();
  float acc = 0.0f;
  const int t0 = blockIdx.x * tiles_per_chunk, t1 = min(ntiles, t0 + tiles_per_chunk);
  for (int tile = t0; tile < t1; ++tile) {
    const int tx0 = (tile % ntx) * kWX, ty0 = ((tile / ntx) % nty) * kWY, tz0 = (tile / (ntx * nty)) * kWZ;
    __syncthreads();
    for (int u = threadIdx.x; u < kWV; u += 96) {
      const int x = tx0 + u % kWX, y = ty0 + (u / kWX) % kWY, z = tz0 + u / (kWX * kWY);
      const bool ok = x < d.x && y < d.y && z < d.z;
      const long long v = ((long long)z * d.y + y) * d.x + x;
#pragma unroll
      for (int c = 0; c < 16; ++c) s_a[c][u] = ok && c < cin ? in[c * nv + v] : 0.0f;
#pragma unroll
      for (int c = 0; c < 6; ++c) s_g[c][u] = ok && c < cout ? gout[c * nv + v] : 0.0f;
    }
    __syncthreads();
#pragma unroll 8
    for (int u = 0; u < kWV; ++u) acc = fmaf(s_g[co][u], s_a[ci][u], acc);
  }
  if (co < cout && ci < cin) part[((long long)blockIdx.x * cout + co) * cin + ci] = acc;
}

}  // namespace pc
}  // namespace dda
