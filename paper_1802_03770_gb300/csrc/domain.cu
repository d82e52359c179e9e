// The paper's preconditioner on an occluded domain Omega (Sec. 4.4): the
// finite-difference operator B_Omega = shift I + scale C h^d L restricted to
// the points of Omega, with Dirichlet conditions on every point of the box
// outside it.  The paper factorises B_Omega by sparse Cholesky; here it is
// applied exactly through the box operator B (the fast DST/tridiagonal solve
// of the full box) and a small dense system on the hole's boundary
// (capacitance matrix method, Buzbee, Dorr, George & Golub, SIAM J. Numer.
// Anal. 8, 1971):
//
//   Gamma = the points outside Omega with a grid neighbour in Omega,
//   E     = injection of Gamma into the box, C = E^T B^{-1} E (SPD),
//   w     = B^{-1} r~ (r~ = r on Omega, 0 elsewhere),
//   s     = -C^{-1} E^T w,
//   z     = R (w + B^{-1} E s).
//
// z~ = w + B^{-1} E s satisfies B z~ = r~ + E s and vanishes on Gamma; on
// the rest of the hole it solves the homogeneous equation with zero data on
// Gamma and the box boundary, so it vanishes there too.  On Omega,
// B z~ = r~ with z~ = 0 at every neighbour outside Omega: B_Omega z = r.
//
// C is formed once per (shift, scale) from |Gamma| FP64 box solves of unit
// vectors and factorised as L D L^T (right-looking, one launch per pivot);
// the same eliminations applied to the identity give W = L^{-1}.  Each
// application is then s = -W^T D^{-1} W E^T w: two triangular matrix-vector
// products (FP64, for either precision of the box solves), bound by the launches
// and the latency of the gathers (the FP64 pipe would take a quarter of the time
// at |Gamma| = 1023).  The blocked substitutions they replace ran in one CTA, one
// dependent block of 32 unknowns after another: 86 us for |Gamma| = 255 between
// events, now 13 + 7 (FP32 box solves 14 + 7); |Gamma| = 1023: 18 + 10 (30 + 10).
#include "chain.cuh"
#include "domain.h"

namespace fl {

namespace {

// e = unit vector at Gamma point `cur` (and the previous one cleared).
__global__ void k_dom_unit(double* e, const int* __restrict__ idx, int prev, int cur) {
  if (threadIdx.x == 0) {
    if (prev >= 0) e[idx[prev]] = 0.0;
    e[idx[cur]] = 1.0;
  }
}

// Column `col` of C: C[b][col] = z[Gamma_b].
__global__ void k_dom_gather(const double* __restrict__ z, const int* __restrict__ idx, int m,
                             double* __restrict__ C, int col) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < m) C[(size_t)b * m + col] = z[idx[b]];
}

// Lower triangle: (C + C^T) / 2 (the box solves are symmetric up to
// rounding).  Strict upper triangle: zeros, where W^T is built.
__global__ void k_dom_symmetrize(double* C, int m) {
  const int i = blockIdx.y * blockDim.y + threadIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m && j < i) {
    C[(size_t)i * m + j] = 0.5 * (C[(size_t)i * m + j] + C[(size_t)j * m + i]);
    C[(size_t)j * m + i] = 0.0;
  }
}

// Pivot k of the right-looking L D L^T factorisation, rows i > k, with the
// factors l_i = A_ik / A_kk (one division per row and CTA: FP64 divisions
// are tens of operations).  z = 0: A_ij -= l_i A_jk, k < j <= i (lower
// triangle); z = 1: W_ij -= l_i W_kj, j <= k (W_ij at [j][i], W_kk = 1).
constexpr int kDomTile = 16;
__global__ void k_dom_ldl_step(double* C, int m, int k) {
  __shared__ double l[kDomTile];
  const bool inv = blockIdx.z == 1;
  // the index that runs along threadIdx.x is the contiguous one: j of A, i of W
  const int i0 = k + 1 + (inv ? blockIdx.x : blockIdx.y) * kDomTile;
  if (threadIdx.y == 0 && i0 + threadIdx.x < m)
    l[threadIdx.x] = C[(size_t)(i0 + threadIdx.x) * m + k] / C[(size_t)k * m + k];
  __syncthreads();
  if (!inv) {
    const int i = i0 + threadIdx.y, j = k + 1 + blockIdx.x * kDomTile + threadIdx.x;
    if (i < m && j <= i) C[(size_t)i * m + j] -= l[threadIdx.y] * C[(size_t)j * m + k];
  } else {
    const int i = i0 + threadIdx.x, j = blockIdx.y * kDomTile + threadIdx.y;
    if (i < m && j <= k) C[(size_t)j * m + i] -= l[threadIdx.x] * (j < k ? C[(size_t)j * m + k] : 1.0);
  }
}

// t = -D^{-1} W w_Gamma: 32 rows per CTA (threadIdx.x), their columns split
// over threadIdx.y.
template <typename T>
__global__ void __launch_bounds__(1024) k_dom_fwd(const T* __restrict__ w, const int* __restrict__ idx,
                                                  const double* __restrict__ LD, int m,
                                                  double* __restrict__ t, const PcgState* st) {
  __shared__ double part[32][33];
  pdl_wait();
  if (st && st->done) return;
  const int i = blockIdx.x * 32 + threadIdx.x;
  double acc = 0.0;
  if (i < m) {
#pragma unroll 4
    for (int j = threadIdx.y; j < i; j += 32) acc += LD[(size_t)j * m + i] * (double)w[idx[j]];
  }
  part[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  // one warp per row
  double v = part[threadIdx.x][threadIdx.y];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int row = blockIdx.x * 32 + threadIdx.y;
  if (threadIdx.x == 0 && row < m) t[row] = -(v + (double)w[idx[row]]) / LD[(size_t)row * m + row];
  pdl_release();
}

// us = W^T t at Gamma (us is zero elsewhere and stays so): one warp per row.
constexpr int kDomBwdWarps = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kDomBwdWarps) k_dom_bwd(const double* __restrict__ t,
                                                              const int* __restrict__ idx,
                                                              const double* __restrict__ LD, int m,
                                                              T* __restrict__ us, const PcgState* st) {
  pdl_wait();
  if (st && st->done) return;
  const int j = blockIdx.x * kDomBwdWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j < m) {
    double acc = 0.0;
#pragma unroll 4
    for (int i = j + 1 + lane; i < m; i += 32) acc += LD[(size_t)j * m + i] * t[i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) us[idx[j]] = (T)(t[j] + acc);
  }
  pdl_release();
}

}  // namespace

cudaError_t dom_build_capacitance(const Geo& g, const Tables<double>& tb, const DomainData& dd,
                                  double shift, double scale, double* e, double* z, cudaStream_t s) {
  cudaError_t err = cudaMemsetAsync(e, 0, g.N * sizeof(double), s);
  for (int a = 0; a < dd.m && err == cudaSuccess; ++a) {
    FL_KERNEL("dom_unit", s, k_dom_unit<<<1, 32, 0, s>>>(e, dd.idx, a - 1, a));
    PrecIO<double> io;
    io.in = e; io.out = z; io.shift = shift; io.scale = scale;   // the box operator: no mask
    err = launch_precond<double>(g, tb, s, io);
    if (err == cudaSuccess) {
      FL_KERNEL("dom_gather", s, k_dom_gather<<<(dd.m + 255) / 256, 256, 0, s>>>(z, dd.idx, dd.m, dd.LD, a));
      err = cudaGetLastError();
    }
  }
  if (err != cudaSuccess) return err;
  const dim3 blk(kDomTile, kDomTile);
  const int tiles = (dd.m + kDomTile - 1) / kDomTile;
  FL_KERNEL("dom_symmetrize", s, k_dom_symmetrize<<<dim3(tiles, tiles), blk, 0, s>>>(dd.LD, dd.m));
  for (int k = 0; k + 1 < dd.m; ++k) {
    const int below = (dd.m - k - 1 + kDomTile - 1) / kDomTile, left = (k + kDomTile) / kDomTile;
    FL_KERNEL("dom_ldl_step", s,
              k_dom_ldl_step<<<dim3(below, below > left ? below : left, 2), blk, 0, s>>>(dd.LD, dd.m, k));
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t dom_interface_solve(const DomainData& dd, const T* w, T* us, const PcgState* st,
                                cudaStream_t s) {
  FL_KERNEL(sizeof(T) == 4 ? "dom_fwd<f32>" : "dom_fwd<f64>", s,
            pdl_launch(k_dom_fwd<T>, (dd.m + 31) / 32, dim3(32, 32), 0, s, w, (const int*)dd.idx,
                       (const double*)dd.LD, dd.m, dd.t, st));
  FL_KERNEL(sizeof(T) == 4 ? "dom_bwd<f32>" : "dom_bwd<f64>", s,
            pdl_launch(k_dom_bwd<T>, (dd.m + kDomBwdWarps - 1) / kDomBwdWarps, 32 * kDomBwdWarps, 0, s,
                       (const double*)dd.t, (const int*)dd.idx, (const double*)dd.LD, dd.m, us, st));
  return launch_status();
}

template cudaError_t dom_interface_solve<float>(const DomainData&, const float*, float*, const PcgState*,
                                                cudaStream_t);
template cudaError_t dom_interface_solve<double>(const DomainData&, const double*, double*,
                                                 const PcgState*, cudaStream_t);

}  // namespace fl
