// x and y passes of the complex64 product fused per z plane, for small grids
// (arXiv:0704.0037, Sec. 2: the same pruned 1D transforms).
//
// On grids of up to 96 points along x and y a pass is a few microseconds of
// work, and a product is bound by its five dependent launches.  Here a block
// holds one (right-hand side, component, z) plane in shared memory: the
// forward kernel gathers beta x, transforms the rows and then the columns
// (P1 and P2), the inverse one runs the columns and then the rows and forms
// y = x - beta u (P4 and P5), so that a product is three launches and its
// x-transformed rows never leave the SM.  The lengths are chosen at run time
// among codelets compiled into the one kernel (a switch per direction instead
// of a kernel per pair of lengths); each line is computed with the arithmetic
// of the separate passes (fastfft.cuh), so the products agree bit for bit.
// 16^3 sphere: 13.4 -> 11.5 us a product, 9.7 with the tables loaded ahead of the
// wait for the kernel before, 8.7 with the product in registers in the z pass
// and no division per item here.  With 16 right-hand sides on a 40 x 29 x 22
// ellipsoid the two kernels took what the four took (43.6 against 43.4 us; 37
// now), so the line lies at the lengths whose planes fit an SM twice.  A plane is
// one block's work, and few planes with long columns leave the chip idle where the
// passes per axis spread over it: from 64 points in y and more than 3,072 in a
// plane, (My - 32) / 3 planes (of all right-hand sides) are fused and fewer are
// not.  Fused against not, us: 96 x 96 points 20.6 and 16.4 (1 plane), 18.1 and
// 15.6 (16), 19.6 and 21.6 (24); 80 x 80 15.6 and 14.3 (12), 17.4 and 16.7 (24),
// 17.3 and 18.3 (32); 64 x 64 20.6 and 19.1 (4), 12.1 and 12.6 (12); 40 x 96 13.1
// and 12.6 (12), 13.8 and 14.3 (20); 96 x 40 12.1 and 12.8 (12); 48 x 64 12.5 and
// 12.8 (1); 32 x 32 10.5 and 12.5 (1).
#include "fastfft.cuh"

namespace dda {
namespace fast {
namespace {

constexpr int kXYT = 256;

// A thread's items threadIdx.x, threadIdx.x + kXYT, ... of (q, t), t < n: q = item
// / n and t = item % n advance by constants (one division, at the start); none
// when n = 0 (a plane without dipoles)
struct Items {
  int q, t, n, dq, dt;
  __device__ __forceinline__ explicit Items(int n_) : n(max(n_, 1)) {
    q = threadIdx.x / n;
    t = threadIdx.x - q * n;
    dq = kXYT / n;
    dt = kXYT - dq * n;
    if (n_ <= 0) q = 1 << 20;
  }
  __device__ __forceinline__ void next() {
    q += dq;
    t += dt;
    if (t >= n) { t -= n; ++q; }
  }
};

// Row transforms, nrow rows at P + t ld; Q is scratch of the same shape.
// Forward: P[t][n] (n < kHalf M2 may be nonzero) -> P[t][k].
template <int M1, int M2>
__device__ __forceinline__ void rows_fwd(c64* P, c64* Q, int nrow, int ld, const c64* tw) {
  for (Items it(nrow); it.q < M2; it.next()) {
    const int j = it.q, t = it.t;
    c64 v[M1];
#pragma unroll
    for (int i = 0; i < M1; ++i) v[i] = i < kHalf<M1, M2> ? P[t * ld + j + M2 * i] : zero<float>();
    dft_padded<float, M1, kHalf<M1, M2>>(v);
#pragma unroll
    for (int k1 = 1; k1 < M1; ++k1) v[k1] = twiddle<float, false>(v[k1], tw[j * k1]);
#pragma unroll
    for (int k1 = 0; k1 < M1; ++k1) Q[t * ld + k1 * M2 + j] = v[k1];
  }
  __syncthreads();
  for (Items it(nrow); it.q < M1; it.next()) {
    const int k1 = it.q, t = it.t;
    c64 u[M2];
#pragma unroll
    for (int j = 0; j < M2; ++j) u[j] = Q[t * ld + k1 * M2 + j];
    cl::Dft<float, false, M2>::run(u);
#pragma unroll
    for (int k2 = 0; k2 < M2; ++k2) P[t * ld + k1 + M1 * k2] = u[k2];
  }
}

// Inverse: P[t][k] -> P[t][n], n < kHalf M2.
template <int M1, int M2>
__device__ __forceinline__ void rows_inv(c64* P, c64* Q, int nrow, int ld, const c64* tw) {
  for (Items it(nrow); it.q < M1; it.next()) {
    const int k1 = it.q, t = it.t;
    c64 u[M2];
#pragma unroll
    for (int k2 = 0; k2 < M2; ++k2) u[k2] = P[t * ld + k1 + M1 * k2];
    cl::Dft<float, true, M2>::run(u);
#pragma unroll
    for (int j = 1; j < M2; ++j) u[j] = twiddle<float, true>(u[j], tw[j * k1]);
#pragma unroll
    for (int j = 0; j < M2; ++j) Q[t * ld + k1 * M2 + j] = u[j];
  }
  __syncthreads();
  for (Items it(nrow); it.q < M2; it.next()) {
    const int j = it.q, t = it.t;
    c64 v[M1];
#pragma unroll
    for (int k1 = 0; k1 < M1; ++k1) v[k1] = Q[t * ld + k1 * M2 + j];
    cl::Dft<float, true, M1>::run(v);
#pragma unroll
    for (int i = 0; i < kHalf<M1, M2>; ++i) P[t * ld + j + M2 * i] = v[i];
  }
}

// Column transforms of a plane, cw columns at a time; Q [M][cw].  Forward: rows
// y0 .. y0 + nrow - 1 of the plane are P[t][kx]; out[ky][Mx] in global memory.
template <int M1, int M2>
__device__ __forceinline__ void cols_fwd(const c64* P, c64* Q, int y0, int nrow, int ld, int Mx, int cw,
                                         const c64* tw, c64* __restrict__ out) {
  for (int kx0 = 0; kx0 < Mx; kx0 += cw) {
    const int w = min(cw, Mx - kx0);
    if (kx0) __syncthreads();                  // Q has been read
    for (Items it(w); it.q < M2; it.next()) {
      const int j = it.q, kx = kx0 + it.t;
      c64 v[M1];
#pragma unroll
      for (int i = 0; i < M1; ++i) {
        const int t = j + M2 * i - y0;
        v[i] = (i < kHalf<M1, M2> && t >= 0 && t < nrow) ? P[t * ld + kx] : zero<float>();
      }
      dft_padded<float, M1, kHalf<M1, M2>>(v);
#pragma unroll
      for (int k1 = 1; k1 < M1; ++k1) v[k1] = twiddle<float, false>(v[k1], tw[j * k1]);
#pragma unroll
      for (int k1 = 0; k1 < M1; ++k1) Q[(k1 * M2 + j) * w + it.t] = v[k1];
    }
    __syncthreads();
    for (Items it(w); it.q < M1; it.next()) {
      const int k1 = it.q, kx = kx0 + it.t;
      c64 u[M2];
#pragma unroll
      for (int j = 0; j < M2; ++j) u[j] = Q[(k1 * M2 + j) * w + it.t];
      cl::Dft<float, false, M2>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < M2; ++k2) out[(k1 + M1 * k2) * Mx + kx] = u[k2];
    }
  }
}

// Inverse: in[ky][Mx] in global memory -> P[t][kx] for rows y0 + t, t < nrow.
template <int M1, int M2>
__device__ __forceinline__ void cols_inv(const c64* __restrict__ in, c64* P, c64* Q, int y0, int nrow, int ld,
                                         int Mx, int cw, const c64* tw) {
  for (int kx0 = 0; kx0 < Mx; kx0 += cw) {
    const int w = min(cw, Mx - kx0);
    if (kx0) __syncthreads();                  // Q has been read
    for (Items it(w); it.q < M1; it.next()) {
      const int k1 = it.q, kx = kx0 + it.t;
      c64 u[M2];
#pragma unroll
      for (int k2 = 0; k2 < M2; ++k2) u[k2] = in[(k1 + M1 * k2) * Mx + kx];
      cl::Dft<float, true, M2>::run(u);
#pragma unroll
      for (int j = 1; j < M2; ++j) u[j] = twiddle<float, true>(u[j], tw[j * k1]);
#pragma unroll
      for (int j = 0; j < M2; ++j) Q[(k1 * M2 + j) * w + it.t] = u[j];
    }
    __syncthreads();
    for (Items it(w); it.q < M2; it.next()) {
      const int j = it.q, kx = kx0 + it.t;
      c64 v[M1];
#pragma unroll
      for (int k1 = 0; k1 < M1; ++k1) v[k1] = Q[(k1 * M2 + j) * w + it.t];
      cl::Dft<float, true, M1>::run(v);
#pragma unroll
      for (int i = 0; i < kHalf<M1, M2>; ++i) {
        const int t = j + M2 * i - y0;
        if (t >= 0 && t < nrow) P[t * ld + kx] = v[i];
      }
    }
  }
}

#define DDA_XY_LENGTHS(M, CALL)   \
  switch (M) {                    \
    case 32: CALL(4, 8); break;   \
    case 40: CALL(5, 8); break;   \
    case 48: CALL(6, 8); break;   \
    case 64: CALL(8, 8); break;   \
    case 80: CALL(8, 10); break;  \
    case 96: CALL(8, 12); break;  \
  }

// Shared memory of a plane: twiddles of both axes, P [nrow][ld], Q (the larger
// of P's shape and [My][cw]), and the row offsets (ny + 1).
struct PlaneMem {
  c64 *twx, *twy, *P, *Q;
  long long* off;
  int y0, nrow, ld;
};
__device__ __forceinline__ PlaneMem plane_mem(unsigned char* smem, const c64* __restrict__ tw, LatticeDev lat,
                                              int z, int ny, int Mx, int My) {
  PlaneMem m;
  m.ld = Mx + 1;                            // Mx is even: odd rows, no bank conflicts
  m.off = reinterpret_cast<long long*>(smem);
  m.twx = reinterpret_cast<c64*>(smem + 16 * ((ny + 2) / 2));
  m.twy = m.twx + Mx;
  m.P = m.twy + My;
  m.Q = m.P + ny * m.ld;
  for (int i = threadIdx.x; i < Mx + My; i += kXYT) m.twx[i] = tw[i];
  for (int i = threadIdx.x; i <= ny; i += kXYT) m.off[i] = lat.row_off[(long long)z * ny + i];
  m.y0 = lat.yr ? lat.yr[2 * z] : 0;        // rows outside the span hold no dipole
  m.nrow = lat.yr ? lat.yr[2 * z + 1] - m.y0 + 1 : ny;
  return m;
}
size_t plane_bytes(int ny, int Mx, int My, int cw) {
  const size_t p = (size_t)ny * (Mx + 1), q = (size_t)cw * My;
  return 16 * ((ny + 2) / 2) + (Mx + My + p + (p > q ? p : q)) * sizeof(c64);
}
// Columns transformed at a time: all, or half of them where whole planes let no
// more than `few` blocks share an SM and the launch fills those (96 x 96 points
// with 8 right-hand sides, two planes an SM: 35.1 -> 32.4 us forward, 42.0 -> 40.4
// inverse; 80 x 64 with 16, three: 18.3 -> 18.6 and 20.0 -> 18.9; 64 x 64, four:
// 19.4 -> 20.3 and 19.7 -> 20.5).
int plane_columns(const FastArgs& a, int few) {
  const long long fit = (227LL << 10) / (long long)(plane_bytes(a.ny, a.Mx, a.My, a.Mx) + 1024);
  return fit <= few && 3LL * a.nz * a.nrhs > fit * num_sms() ? a.Mx / 2 : a.Mx;
}
// Dipoles are taken row by row, half a warp to a row: no search for a dipole's
// row (40 x 29 x 22 ellipsoid, 16 right-hand sides, 18.3 -> 17.4 us forward, 19.2
// -> 18.7 inverse; 47^3, 8, 32.7 -> 29.3 and 39.5 -> 39.0).  kGU dipoles of a lane
// are loaded together.
constexpr int kRL = 16, kGU = 3;

// grid (nz, 3 nrhs)
template <bool CONJ>
__global__ void __launch_bounds__(kXYT, 4) fk_xy_fwd(const c64* __restrict__ x, c64* __restrict__ B2,
                                                  LatticeDev lat, const c64* __restrict__ beta,
                                                  long long n_occ, int ny, int Mx, int My, int cw,
                                                  const c64* __restrict__ tw, int bstride,
                                                  const int* __restrict__ skip) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int z = blockIdx.x, cc = blockIdx.y, c = cc % 3;
  beta += (long long)(cc / 3) * bstride;
  const PlaneMem m = plane_mem(smem_raw, tw, lat, z, ny, Mx, My);
  for (int i = threadIdx.x; i < m.nrow * m.ld; i += kXYT) m.P[i] = zero<float>();
  __syncthreads();
  pdl_wait();
  pdl_launch();
  if (skip && skip[cc / 3]) return;
  const c64* xc = x + (long long)cc * n_occ;
  for (int r = threadIdx.x / kRL; r < m.nrow; r += kXYT / kRL) {
    const long long S0 = m.off[m.y0 + r];
    const int n = (int)(m.off[m.y0 + r + 1] - S0);
    for (int k0 = threadIdx.x % kRL; k0 < n; k0 += kGU * kRL) {
      c64 xv[kGU];
      int xk[kGU], mk_[kGU];
#pragma unroll
      for (int u = 0; u < kGU; ++u) {
        const int k = k0 + u * kRL;
        if (k < n) { xv[u] = xc[S0 + k]; xk[u] = lat.xi[S0 + k]; mk_[u] = lat.mat[S0 + k]; }
      }
#pragma unroll
      for (int u = 0; u < kGU; ++u) {
        if (k0 + u * kRL < n) {
          const c64 v = CONJ ? conjg(xv[u]) : xv[u];
          m.P[r * m.ld + xk[u]] = beta[mk_[u] * 3 + c] * v;
        }
      }
    }
  }
  __syncthreads();
#define ROWS(A, B) rows_fwd<A, B>(m.P, m.Q, m.nrow, m.ld, m.twx)
  DDA_XY_LENGTHS(Mx, ROWS)
#undef ROWS
  __syncthreads();
  c64* out = B2 + ((long long)cc * gridDim.x + z) * My * Mx;
#define COLS(A, B) cols_fwd<A, B>(m.P, m.Q, m.y0, m.nrow, m.ld, Mx, cw, m.twy, out)
  DDA_XY_LENGTHS(My, COLS)
#undef COLS
}

// grid (nz, 3 nrhs); dotp (or null): the block's partial of x^T y
template <bool CONJ>
__global__ void __launch_bounds__(kXYT, 4) fk_yx_inv(const c64* __restrict__ B2, const c64* __restrict__ x,
                                                  c64* __restrict__ y, LatticeDev lat,
                                                  const c64* __restrict__ beta, long long n_occ, int ny,
                                                  int Mx, int My, int cw, const c64* __restrict__ tw,
                                                  double* __restrict__ dotp, int bstride,
                                                  const int* __restrict__ skip) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int z = blockIdx.x, cc = blockIdx.y, c = cc % 3;
  beta += (long long)(cc / 3) * bstride;
  const PlaneMem m = plane_mem(smem_raw, tw, lat, z, ny, Mx, My);
  __syncthreads();
  pdl_wait();
  pdl_launch();
  if (skip && skip[cc / 3]) return;
  const c64* in = B2 + ((long long)cc * gridDim.x + z) * My * Mx;
#define COLS(A, B) cols_inv<A, B>(in, m.P, m.Q, m.y0, m.nrow, m.ld, Mx, cw, m.twy)
  DDA_XY_LENGTHS(My, COLS)
#undef COLS
  __syncthreads();
#define ROWS(A, B) rows_inv<A, B>(m.P, m.Q, m.nrow, m.ld, m.twx)
  DDA_XY_LENGTHS(Mx, ROWS)
#undef ROWS
  __syncthreads();
  const c64* xc = x + (long long)cc * n_occ;
  c64* yc = y + (long long)cc * n_occ;
  float tr = 0.0f, ti = 0.0f;
  for (int r = threadIdx.x / kRL; r < m.nrow; r += kXYT / kRL) {
    const long long S0 = m.off[m.y0 + r];
    const int n = (int)(m.off[m.y0 + r + 1] - S0);
    for (int k0 = threadIdx.x % kRL; k0 < n; k0 += kGU * kRL) {
      c64 xv[kGU];
      int xk[kGU], mk_[kGU];
#pragma unroll
      for (int u = 0; u < kGU; ++u) {
        const int k = k0 + u * kRL;
        if (k < n) { xv[u] = xc[S0 + k]; xk[u] = lat.xi[S0 + k]; mk_[u] = lat.mat[S0 + k]; }
      }
#pragma unroll
      for (int u = 0; u < kGU; ++u) {
        const int k = k0 + u * kRL;
        if (k < n) {
          const c64 v = CONJ ? conjg(xv[u]) : xv[u];
          c64 o = v - beta[mk_[u] * 3 + c] * m.P[r * m.ld + xk[u]];
          if (CONJ) o = conjg(o);
          yc[S0 + k] = o;
          tr = tr + (xv[u].x * o.x - xv[u].y * o.y);
          ti = ti + (xv[u].x * o.y + xv[u].y * o.x);
        }
      }
    }
  }
  if (dotp) {
    // warps in FP32, the block in FP64
    __shared__ double sd[2][kXYT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      tr += __shfl_down_sync(0xffffffffu, tr, o);
      ti += __shfl_down_sync(0xffffffffu, ti, o);
    }
    if ((threadIdx.x & 31) == 0) { sd[0][threadIdx.x >> 5] = tr; sd[1][threadIdx.x >> 5] = ti; }
    __syncthreads();
    if (threadIdx.x < 16) {                 // lanes 0-7 the real parts, 8-15 the imaginary ones
      double s = sd[threadIdx.x >> 3][threadIdx.x & 7];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) s += __shfl_down_sync(0xffffu, s, o, 8);
      if ((threadIdx.x & 7) == 0) dotp[2 * ((long long)cc * gridDim.x + z) + (threadIdx.x >> 3)] = s;
    }
  }
}

bool xy_length(int M) { return M == 32 || M == 40 || M == 48 || M == 64 || M == 80 || M == 96; }

template <typename K, typename... Args>
cudaError_t launch_plane(K kernel, const FastArgs& a, int cw, Args... args) {
  const size_t sm = plane_bytes(a.ny, a.Mx, a.My, cw);
  cudaError_t e = ensure_smem((const void*)kernel, sm);
  if (e == cudaSuccess) e = ensure_carveout_max((const void*)kernel);
  if (e != cudaSuccess) return e;
  e = launch_pdl(a.pdl, kernel, dim3(a.nz, 3 * a.nrhs), dim3(kXYT), sm, a.st, args...);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace
}  // namespace fast

bool fast_xy_supported(int Mx, int My, long long planes) {
  if (!fast::xy_length(Mx) || !fast::xy_length(My)) return false;
  return My <= 48 || Mx * My <= 3072 || 3 * planes >= My - 32;
}

// a.in x, a.out B2, a.tw the twiddles of x, then y
cudaError_t fast_xy_fwd_c64(const FastArgs& a) {
  const c64 *x = (const c64*)a.in, *beta = (const c64*)a.beta, *tw = (const c64*)a.tw;
  c64* out = (c64*)a.out;
  const int cw = fast::plane_columns(a, 2);
  return a.adj ? fast::launch_plane(fast::fk_xy_fwd<true>, a, cw, x, out, a.lat, beta, a.n_occ, a.ny, a.Mx, a.My, cw, tw,
                                    a.bstride, a.skip)
               : fast::launch_plane(fast::fk_xy_fwd<false>, a, cw, x, out, a.lat, beta, a.n_occ, a.ny, a.Mx, a.My, cw, tw,
                                    a.bstride, a.skip);
}

// a.in B2, a.x the product's input, a.out y, a.dotp nz partials per component or null
cudaError_t fast_yx_inv_c64(const FastArgs& a) {
  const c64 *in = (const c64*)a.in, *x = (const c64*)a.x, *beta = (const c64*)a.beta, *tw = (const c64*)a.tw;
  c64* out = (c64*)a.out;
  const int cw = fast::plane_columns(a, 3);
  return a.adj ? fast::launch_plane(fast::fk_yx_inv<true>, a, cw, in, x, out, a.lat, beta, a.n_occ, a.ny, a.Mx, a.My, cw,
                                    tw, a.dotp, a.bstride, a.skip)
               : fast::launch_plane(fast::fk_yx_inv<false>, a, cw, in, x, out, a.lat, beta, a.n_occ, a.ny, a.Mx, a.My, cw,
                                    tw, a.dotp, a.bstride, a.skip);
}

}  // namespace dda
