// Far-field sums of dda_scatter as exact integer matrix products on the
// tensor cores (arXiv:0704.0037, Sec. 3.1: amplitudes in many directions).
//
//   S_c(n_d) = sum_j P_c,j exp(-i kd n_d . r_j)
//
// The phase factorises over the axes.  Along x the cells are folded about the
// box centre, with S = P(x) + P(-x) and D = P(x) - P(-x):
//   sum_x P e^{-i phi} = sum_{x > 0} (S cos phi - i D sin phi),
// so a row of the lattice is a real product of [S.re | D.im] (real part) and
// [S.im | -D.re] (imaginary part) with the columns [cos | sin] of the
// directions: a matrix product whose rows are (lattice row, component, part),
// whose columns are the directions and whose inner length is n_x.
//
// On this part the FP64 pipe does 2 fused multiply-adds per clock and SM, and
// the direct sum (22 FP64 operations per dipole and direction) is bound by it.
// So the product runs on the bf16 tensor cores without rounding (Ozaki's
// error-free splitting of a matrix product): both factors are fixed-point
// numbers of 55 bits, relative to the largest entry of their (lattice row,
// component) and to 1, cut into seven signed 8-bit digits that bf16 holds
// exactly; the products of digits i and j with i + j = g go to accumulator g
// (34 of the 49 pairs, g <= 7).  What is left out is 2^-59 of the row's scale
// for digits of any value, 2^-52.5 if all were largest and of one sign; without
// g = 7 (28 pairs) it was 2^-51 and 2^-44, as large as the roundings of the
// phases (error on random fields 1.1 to 1.25 times the direct sums').  A product
// of two digits is at most 2^14 and an accumulator adds at most 7 K <= 7 * 144 of
// them, below 2^24: every FP32 sum of the tensor cores is exact.  The eight
// accumulators are put together in 64-bit integers; FP64 work is left only for
// the (y, z) phase of each row.
//
// One block holds the digits of 8 lattice rows (48 matrix rows, up to 144
// inner columns: 97 KB) in shared memory, in the order the tensor-core
// fragments are loaded, and runs all directions past them in tiles of 32.  Each
// of 4 warps takes 8 directions, whose digits it streams from L2 in fragment
// order, against the three tiles of 16 matrix rows (8 lattice rows, real and
// imaginary part, of one component): 102 matrix instructions for 28 fragment
// loads.  The warps meet only when the digits of the next rows are made, and
// two blocks share an SM, so that one warp's sums (FP64 and integer pipes)
// overlap another's products (tensor pipe).
//
// 128^3 sphere, 1,152 directions, per right-hand side: direct FP64 sums 65.4 ms;
// this product with 16 rows and 12 warps in one block per SM 3.26 ms, with two
// blocks and integer scaling 2.58 ms; digits made in integer instructions 2.31 ms;
// warps that meet only once per row block 2.0 ms; with the pairs i + j = 7 2.2 ms.
#include <algorithm>

#include "internal.h"

#include <cuda_bf16.h>

namespace dda {
namespace {

constexpr int kSl = kFfSl, kRows = kFfRows, kDirs = kFfDirs, kJMax = kFfJMax, kBBlk = kFfBBlk;
constexpr int kNT = 128;          // threads

// t = sum of dg[i] 256^(6 - i), -128 <= dg[i] <= 127 for i > 0
__device__ __forceinline__ void digits(long long t, int (&dg)[kSl]) {
#pragma unroll
  for (int i = kSl - 1; i > 0; --i) {
    const int d = (int)(signed char)(t & 0xff);
    dg[i] = d;
    t = (t - d) >> 8;
  }
  dg[0] = (int)t;
}
__device__ __forceinline__ unsigned pack2(int a, int b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn((float)a, (float)b);
  return *reinterpret_cast<const unsigned*>(&v);
}
// v 2^(54 - e) rounded to an integer, for |v| <= 2^e and e >= -900, in integer
// instructions (the FP64 pipe is the busiest one): the mantissa shifted by the
// difference of the exponents
__device__ __forceinline__ long long to_fixed(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int ev = (int)(b >> 52) & 0x7ff, k = 1022 + e - ev;      // v = m 2^(ev - 1075)
  if (k > 55 || ev == 0) return 0;
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (1ull << 52);
  const long long t = (long long)(k < 0 ? m << 2 : ((m << 1) + ((1ull << k) >> 1)) >> k);   // k = -1: |v| = 2^e
  return b < 0 ? -t : t;
}

// exp(-i kd n_mu r_mu) for the cells of x, then y, then z: tab[cell][n_dir].
// Cells k and n - 1 - k of an axis lie at r and -r: one sincos for both (the
// FP64 pipe bounds this table).
__global__ void k_ff_tab(const double* __restrict__ dirs, int n_dir, double kd, int nx, int ny,
                         int nz, c128* __restrict__ tab) {
  const int hx = (nx + 1) / 2, hy = (ny + 1) / 2, hz = (nz + 1) / 2;
  const long long total = (long long)n_dir * (hx + hy + hz);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    int k = (int)(i / n_dir);
    const int d = (int)(i - (long long)k * n_dir);
    int axis = 0, n = nx, base = 0;
    if (k >= hx) { k -= hx; axis = 1; n = ny; base = nx; if (k >= hy) { k -= hy; axis = 2; n = nz; base = nx + ny; } }
    const double r = 0.5 * (2 * k + 1 - n);
    double s, c;
    sincos(-kd * dirs[3 * d + axis] * r, &s, &c);
    tab[(long long)(base + k) * n_dir + d] = mk<double>(c, s);
    tab[(long long)(base + n - 1 - k) * n_dir + d] = mk<double>(c, -s);
  }
}

// Digits of [cos | sin] in fragment order: block (chunk, tile, step) of kBBlk
// bytes, then digit, 8-direction group, lane, k half
__global__ void k_ff_pack(const c128* __restrict__ tab, int n_dir, int nx, FfShape sh, int ntiles,
                          unsigned* __restrict__ B) {
  const long long total = (long long)sh.nchunk * ntiles * sh.ks * 256;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int w = (int)(i & 255);
    const long long blk = i >> 8;
    const int s = (int)(blk % sh.ks);
    const int tile = (int)((blk / sh.ks) % ntiles), ch = (int)(blk / ((long long)sh.ks * ntiles));
    const int lane = (w >> 1) & 31, b = w & 1;
    const int d = tile * kDirs + (w >> 6) * 8 + (lane >> 2);
    int dg[2][kSl];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int k = s * 16 + (lane & 3) * 2 + b * 8 + u;
      const int j = ch * sh.J + (k < sh.J ? k : k - sh.J);
      double v = 0.0;
      if (k < 2 * sh.J && j < sh.H && d < n_dir) {
        const c128 t = tab[(long long)(nx - sh.H + j) * n_dir + d];
        v = k < sh.J ? t.x : -t.y;
      }
      digits(to_fixed(v, 0), dg[u]);
    }
    unsigned* o = B + blk * (kBBlk / 4) + w;
#pragma unroll
    for (int q = 0; q < kSl; ++q) o[q * 256] = pack2(dg[0][q], dg[1][q]);
  }
}

__device__ __forceinline__ void mma(float (&c)[4], const uint4& a, unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
               "{%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// t 2^e, rounded to nearest, put together in integer instructions: the FP64
// pipe, which the row phases need, is left alone.  e keeps the result from
// underflow; a result of 2^1024 and more becomes non-finite.
__device__ __forceinline__ double scaled(long long t, int e) {
  const unsigned long long m = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
  const int lz = __clzll((long long)m);
  const unsigned long long u = m << lz;                       // bit 63 set
  const unsigned long long v = (u >> 11) + ((u >> 10) & 1);   // 2^52 .. 2^53
  const unsigned long long bits = ((unsigned long long)min(1085 - lz + e, 2046) << 52) + v;
  return __longlong_as_double((long long)(t == 0 ? 0ull : bits | ((unsigned long long)t & (1ull << 63))));
}

// shared memory behind the A digits: the gather stage of the build phase (4
// warps x 2 J cells), then the row phases of the directions of each warp
constexpr int kTail = kNT / 32 * 2 * kJMax * 16;
constexpr int kBad = 1 << 20;     // scale exponent of a row with NaN or infinity
static_assert(kRows * kDirs * 16 <= kTail, "the row phases fit in the gather stage");

// Partial sums of the row blocks u = blockIdx.x, + gridDim.x, ... (of units =
// row blocks x chunks) for the direction tiles of blockIdx.y:
// part[blockIdx.x][n_dir][6] (components, re/im).  Rows are those of lat.arow
// (or all nr rows).
__global__ void __launch_bounds__(kNT, 2)
    k_ff_mma(const c128* __restrict__ P, LatticeDev lat, const c128* __restrict__ tab,
             const unsigned char* __restrict__ B, int n_dir, int nx, int ny, int nr, long long n_occ,
             FfShape sh, int ntiles, int tiles_per_y, int units, double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_e[kRows * 3], s_iy[kRows], s_iz[kRows];
  unsigned* A = reinterpret_cast<unsigned*>(smem);
  unsigned char* tail = smem + 3 * sh.ks * kSl * 512;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2;
  c128* s_w = reinterpret_cast<c128*>(tail) + warp * kRows * 8;   // [row][direction] of this warp
  const int t0 = blockIdx.y * tiles_per_y, t1 = min(ntiles, t0 + tiles_per_y);
  const long long* off = lat.arow ? lat.aoff : lat.row_off;

  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int rb = u / sh.nchunk, ch = u - rb * sh.nchunk, j0 = ch * sh.J;
    __syncthreads();                         // the previous unit's reads of A and the row phases
    // ---- digits of the 8 rows: a warp per (row, component)
    c128* stage = reinterpret_cast<c128*>(tail) + warp * 2 * kJMax;
    for (int p = warp; p < 3 * kRows; p += kNT / 32) {
      const int r = p / 3, c = p - 3 * r, ri = rb * kRows + r;
      for (int k = lane; k < 2 * sh.J; k += 32) stage[k] = mk<double>(0.0, 0.0);
      __syncwarp();
      if (ri < nr) {
        const long long s1 = off[ri + 1];
        for (long long i = off[ri] + lane; i < s1; i += 32) {
          const int x = lat.xi[i], hi = x - (nx - sh.H);
          const int j = (hi >= 0 ? hi : (nx & 1) - 1 - hi) - j0;
          if (j >= 0 && j < sh.J) stage[hi >= 0 ? j : sh.J + j] = P[c * n_occ + i];
        }
      }
      if (c == 0 && lane == 0) {
        const int row = ri < nr ? (lat.arow ? lat.arow[ri] : ri) : 0;
        s_iy[r] = row % ny;
        s_iz[r] = row / ny;
      }
      __syncwarp();
      // S and D in place of P(x) and P(-x), and the largest exponent field of
      // their parts (2047: infinity or NaN)
      int m = 0;
      for (int k = lane; k < sh.J; k += 32) {
        const c128 h = stage[k], l = stage[sh.J + k];
        const c128 s = h + l, d = h - l;
        stage[k] = s;
        stage[sh.J + k] = d;
        m = max(max(max(m, __double2hiint(s.x) & 0x7ff00000), __double2hiint(s.y) & 0x7ff00000),
                max(__double2hiint(d.x) & 0x7ff00000, __double2hiint(d.y) & 0x7ff00000));
      }
      m = __reduce_max_sync(0xffffffffu, m) >> 20;
      const bool bad = m == 0x7ff;
      // |values| < 2^e (e no smaller than -900: below that the row counts as tiny)
      const int e = max(m - 1022, -900);
      if (lane == 0) s_e[p] = bad ? kBad : e - 56;
      __syncwarp();
      for (int kp = lane; kp < sh.ks * 8; kp += 32) {
        int dr[2][kSl], di[2][kSl];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int k = 2 * kp + q;
          double re = 0.0, im = 0.0;
          if (k < 2 * sh.J && !bad) {
            const c128 v = stage[k];
            re = k < sh.J ? v.x : v.y;         // S.re, S.im | D.im, -D.re
            im = k < sh.J ? v.y : -v.x;
          }
          digits(to_fixed(re, e), dr[q]);
          digits(to_fixed(im, e), di[q]);
        }
        const int s = kp >> 3, kin = (2 * kp) & 15;
        uint2* o = reinterpret_cast<uint2*>(A + ((c * sh.ks + s) * kSl) * 128 +
                                            (r * 4 + ((kin & 7) >> 1)) * 4 + (kin >= 8 ? 2 : 0));
#pragma unroll
        for (int q = 0; q < kSl; ++q) o[q * 64] = make_uint2(pack2(dr[0][q], dr[1][q]), pack2(di[0][q], di[1][q]));
      }
      __syncwarp();
    }
    __syncthreads();
    // ---- the product with tiles t0 .. t1 - 1, one step of 16 columns at a time
    const int e3[3] = {s_e[3 * g], s_e[3 * g + 1], s_e[3 * g + 2]};
    // (each warp on its own: it streams the digits of its 8 directions of every
    // tile from L2 a step ahead, so one warp's sums overlap another's products)
    const int q0 = (ch * ntiles + t0) * sh.ks, q1 = (ch * ntiles + t1) * sh.ks;
    const uint2* bp = reinterpret_cast<const uint2*>(B) + warp * 32 + lane;
    uint2 bn[kSl];
#pragma unroll
    for (int k = 0; k < kSl; ++k) bn[k] = bp[(size_t)q0 * (kBBlk / 8) + k * 128];
    int q = q0;
    for (int tile = t0; tile < t1; ++tile) {
      for (int i = lane; i < kRows * 8; i += 32) {
        const int r = i >> 3, d = tile * kDirs + warp * 8 + (i & 7);
        c128 w = mk<double>(0.0, 0.0);
        if (rb * kRows + r < nr && d < n_dir)
          w = tab[(long long)(nx + s_iy[r]) * n_dir + d] * tab[(long long)(nx + ny + s_iz[r]) * n_dir + d];
        s_w[i] = w;
      }
      // after the reduction over rows a lane holds part (lane bit 4), column
      // (bit 3) of its warp's 8 directions; the partial sums so far
      const int dl = warp * 8 + (lane & 3) * 2 + ((lane >> 3) & 1), d = tile * kDirs + dl;
      double* o = part + ((long long)blockIdx.x * n_dir + d) * 6 + (lane >> 4);
      const bool mine = (lane & 4) == 0 && d < n_dir;
      double old[3] = {0.0, 0.0, 0.0};
      if (mine && u != (int)blockIdx.x) { old[0] = o[0]; old[1] = o[2]; old[2] = o[4]; }
      float acc[3][kSl + 1][4];
#pragma unroll
      for (int n = 0; n < 3; ++n)
#pragma unroll
        for (int k = 0; k <= kSl; ++k)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[n][k][v] = 0.0f;
      for (int s = 0; s < sh.ks; ++s, ++q) {
        uint2 bf[kSl];
#pragma unroll
        for (int k = 0; k < kSl; ++k) bf[k] = bn[k];
        if (q + 1 < q1) {
#pragma unroll
          for (int k = 0; k < kSl; ++k) bn[k] = bp[(size_t)(q + 1) * (kBBlk / 8) + k * 128];
        }
        uint4 af[3][kSl];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int k = 0; k < kSl; ++k)
            af[c][k] = reinterpret_cast<const uint4*>(A)[((c * sh.ks + s) * kSl + k) * 32 + lane];
#pragma unroll
        for (int i = 0; i < kSl; ++i)
#pragma unroll
          for (int j = 0; j < (i ? kSl + 1 - i : kSl); ++j)
#pragma unroll
            for (int c = 0; c < 3; ++c) mma(acc[c][i + j], af[c][i], bf[j].x, bf[j].y);
      }
      // ---- 64-bit sums, row phases, sum over the 8 rows
      __syncwarp();
      double v[3][2][2];                     // [component][column][re, im]
#pragma unroll
      for (int col = 0; col < 2; ++col) {
        const c128 w = s_w[g * 8 + (lane & 3) * 2 + col];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          double z[2];
#pragma unroll
          for (int im = 0; im < 2; ++im) {
            long long t = __float2int_rn(acc[c][0][2 * im + col]);
#pragma unroll
            for (int k = 1; k < kSl - 1; ++k) t = t * 256 + __float2int_rn(acc[c][k][2 * im + col]);
            const int last = __float2int_rn(acc[c][kSl - 1][2 * im + col]) +
                             (__float2int_rn(acc[c][kSl][2 * im + col]) >> 8);
            t = t * 16 + ((last + 8) >> 4);
            z[im] = e3[c] == kBad ? nan("") : scaled(t, e3[c]);
          }
          v[c][col][0] = z[0] * w.x - z[1] * w.y;
          v[c][col][1] = z[0] * w.y + z[1] * w.x;
        }
      }
      const bool b4 = lane & 16, b3 = lane & 8;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        double p[2];
#pragma unroll
        for (int col = 0; col < 2; ++col)
          p[col] = (b4 ? v[c][col][1] : v[c][col][0]) +
                   __shfl_xor_sync(0xffffffffu, b4 ? v[c][col][0] : v[c][col][1], 16);
        double a = (b3 ? p[1] : p[0]) + __shfl_xor_sync(0xffffffffu, b3 ? p[0] : p[1], 8);
        a += __shfl_xor_sync(0xffffffffu, a, 4);
        if (mine) o[2 * c] = old[c] + a;
      }
      __syncwarp();                          // every read of the row phases
    }
  }
}

// F(n_d) from the nb partials (fixed order), then the transverse projection:
// 8 directions per block, 8 strided sums per value
__global__ void __launch_bounds__(384) k_ff_fin(const double* __restrict__ part, int nb, int n_dir,
                                                const double* __restrict__ dirs, double kd,
                                                double* __restrict__ F) {
  __shared__ double sh[8][48];
  const int t = threadIdx.x % 48, q = threadIdx.x / 48, d0 = blockIdx.x * 8;
  const long long n6 = 6LL * n_dir;
  double s = 0.0;
  if (6 * d0 + t < n6)
    for (int b = q; b < nb; b += 8) s += part[b * n6 + 6 * d0 + t];
  sh[q][t] = s;
  __syncthreads();
  if (threadIdx.x < 48) {
    for (int b = 1; b < 8; ++b) s += sh[b][t];
    sh[0][t] = s;
  }
  __syncthreads();
  const int d = d0 + threadIdx.x;
  if (threadIdx.x >= 8 || d >= n_dir) return;
  const double* a = &sh[0][6 * threadIdx.x];
  const double nx = dirs[3 * d], ny = dirs[3 * d + 1], nz = dirs[3 * d + 2];
  const double dr = nx * a[0] + ny * a[2] + nz * a[4];
  const double di = nx * a[1] + ny * a[3] + nz * a[5];
  const double n3[3] = {nx, ny, nz};
  const double k3 = kd * kd * kd;
  for (int c = 0; c < 3; ++c) {
    const double tr = a[2 * c] - n3[c] * dr;
    const double ti = a[2 * c + 1] - n3[c] * di;
    // -i k3 (tr + i ti) = k3 ti - i k3 tr
    F[6 * d + 2 * c] = k3 * ti;
    F[6 * d + 2 * c + 1] = -k3 * tr;
  }
}

}  // namespace

cudaError_t farfield_tables(void* ws, const double* dirs, int n_dir, double kd, int nx, int ny, int nz,
                            const FarfieldPlan& p, cudaStream_t st) {
  if (n_dir > p.cap) return cudaErrorInvalidValue;         // the workspace is p's
  const FfShape s = ff_shape(nx);
  const int nt = ff_tiles(n_dir);
  c128* tab = (c128*)ws;
  unsigned* pack = (unsigned*)((unsigned char*)ws + p.tab);
  const long long tt = (long long)n_dir * ((nx + 1) / 2 + (ny + 1) / 2 + (nz + 1) / 2), tp = (long long)s.nchunk * nt * s.ks * 256;
  k_ff_tab<<<(int)std::min<long long>((tt + 255) / 256, 8192), 256, 0, st>>>(dirs, n_dir, kd, nx, ny, nz, tab);
  count_launch();
  k_ff_pack<<<(int)std::min<long long>((tp + 255) / 256, 8192), 256, 0, st>>>(tab, n_dir, nx, s, nt, pack);
  count_launch();
  return cudaGetLastError();
}

cudaError_t farfield_sums(void* ws, const c128* P, const LatticeDev& lat, const double* dirs, int n_dir,
                          double kd, int nx, int ny, int nr, long long n_occ, const FarfieldPlan& p,
                          double* F, cudaStream_t st) {
  const FfShape s = ff_shape(nx);
  const int nt = ff_tiles(n_dir), units = ff_units(s, nr), G = p.groups;
  if (n_dir > p.cap || G > units) return cudaErrorInvalidValue;
  const c128* tab = (const c128*)ws;
  const unsigned char* pack = (const unsigned char*)ws + p.tab;
  double* part = (double*)((unsigned char*)ws + p.tab + p.pack);
  // direction tiles split over blockIdx.y: enough blocks for every SM and,
  // where the row blocks do not divide evenly over the SMs, finer pieces (of
  // 8 tiles at least, over which the digits of a row block are made once)
  const int slots = 2 * num_sms();
  const int want = G < slots ? (slots + G - 1) / G : 4;
  const int ny_ = std::max(1, std::min(want, G < slots ? nt : (nt + 7) / 8));
  const int per = (nt + ny_ - 1) / ny_;
  const size_t sm = (size_t)3 * s.ks * kSl * 512 + kTail;
  cudaError_t e = ensure_smem((const void*)k_ff_mma, sm);
  if (e != cudaSuccess) return e;
  e = ensure_carveout_max((const void*)k_ff_mma);
  if (e != cudaSuccess) return e;
  k_ff_mma<<<dim3(G, (nt + per - 1) / per), kNT, sm, st>>>(P, lat, tab, pack, n_dir, nx, ny, nr, n_occ, s,
                                                          nt, per, units, part);
  count_launch();
  k_ff_fin<<<(n_dir + 7) / 8, 384, 0, st>>>(part, G, n_dir, dirs, kd, F);
  count_launch();
  return cudaGetLastError();
}

}  // namespace dda
