// Pass kernels of the operator apply (paper Sec. 3.1, "Forward operator and
// application with FFT"), of the finite-difference preconditioner solve
// (Sec. 3.1, "Preconditioning"; Sec. 3.2) and of preconditioned CG.
//
// Data layout (row-major, last axis fastest):
//   real fields        n_0 x ... x n_{d-1}
//   operator spectrum  S: complex; axis d-1 holds H = L_{d-1}/2 + 1
//                      half-spectrum entries; in 3D the middle axis has room
//                      for L_1 entries: S[z][y][kx], z < n_0, y < L_1.
//   kernel symbol      sig: real, (L_0/2+1) x ... x (L_{d-1}/2+1), the even
//                      real DFT of the circularly embedded kernel, already
//                      divided by prod L_i.
//
// One operator apply is, for d = 2:  rows_fwd (masked R2C along x),
// cols CONV (FFT along y, x sig, inverse FFT), rows_inv (C2R along x,
// restrict, epilogue); for d = 3 a FWD and an INV cols pass along y wrap
// the CONV pass along z.
//
// The preconditioner z = (shift + scale C h^d L)^{-1} r is a DST-I along
// every axis, a divide by the eigenvalue, and the DST-I again.  Each DST-I
// of length n is a chirp-z (Bluestein) product: with c_m = exp(i pi m^2 /
// (2(n+1))), sin(pi jk/(n+1)) = Im(c_j c_k conj(c_{k-j})), so
// X_k = Im(c_k sum_j (c_j x_j) conj(c_{k-j})) -- a linear convolution of
// length-n sequences done with FFTs of the operator's length L >= 2n - 1.
// Rows with n + 1 = 2^k take the odd extension, two per transform, and FP32
// axes with n + 1 an odd prime Rader's convolution of length L/2.
#pragma once

#include "fft_core.cuh"
#include "fix_core.cuh"

#ifndef FL_ROW_MIN_CTAS
#define FL_ROW_MIN_CTAS 7
#endif

namespace fl {

// Programmatic dependent launch: a pass launched with the programmatic
// stream-serialization attribute may be scheduled while the previous pass
// is finishing; pdl_wait blocks, before anything the previous passes wrote
// is touched, until that pass has completed and its writes are visible.
// pdl_release, called by each CTA once its work is done, lets the next pass
// launch when every CTA of this one has released (releasing at entry placed
// the next pass's waiting CTAs unevenly and measured 6 % slower).  Both are
// no-ops for an ordinary launch.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Device-resident state of one CG solve (all reductions in FP64).
struct PcgState {
  double rz;       // r^T z of the current iterate
  double bb;       // ||b||^2
  double tol2;     // tol^2 ||b||^2
  double rr;       // ||r||^2 of the current iterate
  double beta;     // p = z + beta p for the next iteration
  double alpha;    // step length of the current iteration, rz / pq
  double pq;       // p^T A p of the current iteration
  int it;          // iterations done
  int maxit;
  int done;        // 1: stop (converged, failed or hit maxit)
  int status;      // 0 ok/converged, 2 not converged, 3 breakdown
  unsigned int arrive;  // CTAs of the current pass that stored their partial
};

enum { PRE_NONE = 0, PRE_PUPDATE = 1, PRE_ACCUM = 2 };
enum { COLS_FWD = 0, COLS_CONV = 1, COLS_INV = 2 };
enum { DPRE_NONE = 0, DPRE_UPDATE = 1 };
// What the last CTA of a pass does with the pass's partial sums:
// FIN_PQ: pq = sum, alpha = rz / pq; FIN_STEP: the CG scalar step.
enum { FIN_NONE = 0, FIN_PQ = 1, FIN_STEP = 2 };

// Sum `count` per-CTA partials in a fixed order (deterministic); every
// thread of the CTA gets the result.  The loads bypass L1, so partials
// stored by other CTAs of the running grid are seen (after arrive_last).
// Uses `red` (>= 32 doubles) of shared memory.
__device__ __forceinline__ double thread_sum_partials(const double* FL_RESTRICT part, int count) {
  // eight loads in flight per thread, then the adds (fixed order)
  double s = 0.0;
  const int nt = blockDim.x;
  int i = threadIdx.x;
  for (; i + 7 * nt < count; i += 8 * nt) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldcg(part + i + u * nt);
#pragma unroll
    for (int u = 0; u < 8; ++u) s += v[u];
  }
  for (; i < count; i += nt) s += __ldcg(part + i);
  return s;
}

__device__ __forceinline__ double cta_sum_partials(const double* FL_RESTRICT part, int count,
                                                   double* red) {
  double s = thread_sum_partials(part, count);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = s;
  __syncthreads();
  double t = 0.0;
  for (int i = 0; i < nw; ++i) t += red[i];
  __syncthreads();
  return t;
}

// Minimum resident CTAs per SM asked of the compiler for a pass kernel of
// THREADS threads.  The passes are latency-bound: the 128-thread FP32 row
// passes keep at least 7 CTAs (28 warps) per SM (<= 73 registers), the
// 256-thread ones 4 (64 registers), the 512-thread passes 2.
// The wide instantiations for the longest lines (LGLO > 4: one line of 4096
// or 8192 points per CTA) ask for one CTA only, so that the compiler keeps
// the row bodies' registers.
constexpr int min_ctas(int threads, int lglo = 4) {
  return lglo > 4 ? 1 : (threads <= 128 ? FL_ROW_MIN_CTAS : (threads == 256 ? 4 : 2));
}

// Column tiles: at most 2^kMaxLtx columns; a CTA of THREADS x VPT values
// holds 2^widest_ltx columns of lines of 2^lg.  The strided passes run the
// widest tile of every length from 2^kFixedLgMin up with the length and the
// width as compile-time constants (their bodies are inlined with constant
// arguments, so the index arithmetic of the loads, the stages and the
// epilogues folds); other shapes (tuned narrower tiles, short lines) take
// the same body with runtime values.
constexpr int kMaxLtx = 6;
constexpr int kFixedLgMin = 8;

__host__ __device__ constexpr int widest_ltx(int threads, int vpt, int lg) {
  return clog2(threads * vpt) - lg < kMaxLtx ? clog2(threads * vpt) - lg : kMaxLtx;
}

// CTA-wide sum of one value per thread; result valid in thread 0.
__device__ __forceinline__ double cta_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < nw; ++i) t += red[i];
  __syncthreads();
  return t;
}

// s + e == a + b exactly (Knuth's two-sum, round-to-nearest adds).
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

// CTA-wide sum of one float-float value (hi + lo) per thread: the warp tree
// in float-float arithmetic, then FP64 across warps; valid in thread 0.
__device__ __forceinline__ double cta_sum_ff(float hi, float lo, double* red) {
  for (int o = 16; o > 0; o >>= 1) {
    const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
    float e;
    const float s = two_sum(hi, h2, e);
    const float t = __fadd_rn(__fadd_rn(lo, l2), e);
    hi = __fadd_rn(s, t);
    lo = __fsub_rn(t, __fsub_rn(hi, s));
  }
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = (double)hi + (double)lo;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < nw; ++i) t += red[i];
  __syncthreads();
  return t;
}

// Per-thread accumulator of a CG dot product.  GB300 issues FP64 at a small
// fraction of the FP32 rate, so the FP32 passes keep FP64 off the per-element
// path: the FP32 products are added into a float-float (two-sum) total, the
// warp tree is float-float and the sums across warps and CTAs are FP64.  The
// sum of the products is then exact to ~2^-46 however a launch shape groups
// them.  FP64 passes accumulate in FP64 throughout.
template <typename T>
struct DotAcc {
  double acc = 0.0;
  __device__ __forceinline__ void add(double v) { acc += v; }
  // CTA total, valid in thread 0
  __device__ __forceinline__ double cta_total(double* red) const { return cta_sum(acc, red); }
};
template <>
struct DotAcc<float> {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float v) {
    float e;
    hi = two_sum(hi, v, e);
    lo = __fadd_rn(lo, e);
  }
  __device__ __forceinline__ double cta_total(double* red) const { return cta_sum_ff(hi, lo, red); }
};

// Every CTA of a pass calls this once, after its partial is stored; it
// returns true (in all threads) in the CTA that arrives last, which may
// then read every partial of the pass.  That CTA also resets the counter
// for the next pass.  No CTA waits for another.
__device__ __forceinline__ bool arrive_last(unsigned int* ctr, int nctas) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned int t = atomicAdd(ctr, 1u);
    s_last = (t + 1u == (unsigned int)nctas) ? 1 : 0;
    if (s_last) *ctr = 0u;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// The CG scalar step after an iteration (one thread): iteration count,
// convergence and breakdown tests, beta.
__device__ __forceinline__ void pcg_step(PcgState* st, double rr, double rz) {
  st->it += 1;
  st->rr = rr;
  const double pq = st->pq;
  if (!(pq > 0.0) || rr != rr || rz != rz) {
    st->done = 1;
    st->status = 3;
  } else if (rr <= st->tol2) {
    st->done = 1;
    st->status = 0;
  } else if (st->it >= st->maxit) {
    st->done = 1;
    st->status = 2;
  } else if (!(rz > 0.0)) {
    st->done = 1;
    st->status = 3;
  } else {
    st->beta = rz / st->rz;
    st->rz = rz;
  }
}

// Spectrum rows of a CTA's field rows row0, row0 + 1, ...: one division per
// CTA instead of one per element.
struct SpecRows {
  int plane, rem, rpp, ps, H;
  __device__ __forceinline__ SpecRows(int row0, int rows_per_plane, int plane_stride, int h)
      : plane(row0 / rows_per_plane), rem(row0 % rows_per_plane), rpp(rows_per_plane), ps(plane_stride), H(h) {}
  __device__ __forceinline__ size_t operator()(int dr) const {
    int p = plane, r = rem + dr;
    while (r >= rpp) {
      r -= rpp;
      ++p;
    }
    return ((size_t)p * ps + r) * H;
  }
};

// ---------------------------------------------------------------------------
// Operator pass 1: masked real-to-complex FFT along the last axis.
// Two real rows ra, rb are packed as ra + i rb, zero-padded to L and
// transformed together; X_a[k] = (Z[k] + conj Z[L-k]) / 2 and
// X_b[k] = (Z[k] - conj Z[L-k]) / (2i), k = 0..H-1.
template <typename T>
struct RowsFwdArgs {
  const T* u;              // PRE_NONE: input field; PRE_PUPDATE: z
  T* p;                    // PRE_PUPDATE: p (in: old p, out: z + beta p)
  double* acc;             // PRE_ACCUM: FP64 field updated as acc += x32 and transformed
  const float* x32;        // PRE_ACCUM
  const uint8_t* mask;     // nullable: Omega inside the box
  typename Cplx<T>::type* S;
  const PcgState* st;
  int rows, n, H, lg, lgmax;
  int rows_per_plane, plane_stride;  // spectrum row = (r / rpp) * ps + r % rpp
  int pre;
  const FxW* ftw;          // FP64: twiddles as fixed-point constants
};

template <typename T, int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void body_rows_fwd_at(const RowsFwdArgs<T>& a, int bx, int by, const int lg) {
  typedef typename Cplx<T>::type C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SBuf<C> buf{reinterpret_cast<C*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int L = 1 << lg;
  const int ls = L;
  const int NL = (VPT * THREADS) / L;       // complex lines (row pairs) per CTA
  const int pair0 = bx * NL;
  const int npairs = (a.rows + 1) / 2;
  const int nl = NL == 1 ? 1 : min(NL, npairs - pair0);
  const T beta = (a.pre == PRE_PUPDATE) ? (T)a.st->beta : (T)0;
  // loads first (U elements per thread in flight), then the stores.  Only
  // the lower half of each line is written (n <= L/2); the transform's first
  // stage reads the upper half as zeros.
  constexpr int U = 4;
  const int hL = L >> 1;
  const int tot = nl * hL;
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    T va[U], vb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int q = e >> (lg - 1), j = e & (hL - 1);
      const int ra = 2 * (pair0 + q), rb = ra + 1;
      va[u] = 0;
      vb[u] = 0;
      if (e < tot && j < a.n) {
        const size_t ia = (size_t)ra * a.n + j, ib = (size_t)rb * a.n + j;
        const bool hb = rb < a.rows;
        if (a.pre == PRE_PUPDATE) {
          // beta == 0 (first iteration): p = z, without reading the old p
          va[u] = beta != (T)0 ? a.u[ia] + beta * a.p[ia] : a.u[ia];
          if (hb) vb[u] = beta != (T)0 ? a.u[ib] + beta * a.p[ib] : a.u[ib];
        } else if (a.pre == PRE_ACCUM) {
          va[u] = (T)(a.acc[ia] + (double)a.x32[ia]);
          if (hb) vb[u] = (T)(a.acc[ib] + (double)a.x32[ib]);
        } else {
          va[u] = a.u[ia];
          if (hb) vb[u] = a.u[ib];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      if (e >= tot) continue;
      const int q = e >> (lg - 1), j = e & (hL - 1);
      const int ra = 2 * (pair0 + q), rb = ra + 1;
      T xa = va[u], xb = vb[u];
      if (j < a.n) {
        const size_t ia = (size_t)ra * a.n + j, ib = (size_t)rb * a.n + j;
        const bool hb = rb < a.rows;
        if (a.pre == PRE_PUPDATE) {
          a.p[ia] = xa;
          if (hb) a.p[ib] = xb;
        } else if (a.pre == PRE_ACCUM) {
          a.acc[ia] = (double)xa;
          if (hb) a.acc[ib] = (double)xb;
        }
        if (a.mask) {
          if (!a.mask[ia]) xa = 0;
          if (hb && !a.mask[ib]) xb = 0;
        }
      }
      buf[q * ls + j] = cmake<C>(xa, xb);
    }
  }
  __syncthreads();
  {
    const C* const calc = nullptr;   // twiddles are computed
    auto ld = [=](int q, int k) -> C { return k < hL ? buf[q * ls + k] : cmake<C>((T)0, (T)0); };
    auto st = [=](int q, int k, C v) { buf[q * ls + k] = v; };
    fft_io<VPT, false, true, LGHI, LGLO>(buf, lg, ls, 0, nl, calc, a.lgmax, false, ld,
                                                       true, st, true);
  }
  __syncthreads();
  // all lines of the CTA in one index space (a loop over lines cost a CTA of
  // 16 lines of 128 points 2900 instructions per warp, most of them idle
  // lanes' loop overhead); k = L/2 afterwards
  const SpecRows spec(2 * pair0, a.rows_per_plane, a.plane_stride, a.H);
  auto put = [&](int q, int k) {
    const SBuf<C> lb = buf.at(q * ls);
    const C z = lb[k];
    const C w = cconj(lb[(L - k) & (L - 1)]);
    a.S[spec(2 * q) + k] = cmake<C>((z.x + w.x) * (T)0.5, (z.y + w.y) * (T)0.5);
    if (2 * (pair0 + q) + 1 < a.rows)
      a.S[spec(2 * q + 1) + k] = cmake<C>((z.y - w.y) * (T)0.5, (w.x - z.x) * (T)0.5);
  };
#pragma unroll 4
  for (int e = threadIdx.x; e < tot; e += THREADS) put(e >> (lg - 1), e & (hL - 1));
  for (int q = threadIdx.x; q < nl; q += THREADS) put(q, hL);
}

// body_rows_fwd with the line length 2^LG .. 2^LGHI as a compile-time
// constant (the lengths below 2^kFixedLgMin at run time)
template <typename T, int THREADS, int VPT, int LGLO, int LGHI, int LG>
__device__ __forceinline__ void body_rows_fwd_fixed(const RowsFwdArgs<T>& a, int bx, int by) {
  if constexpr (LG <= LGHI) {
    if (a.lg == LG) {
      body_rows_fwd_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, by, LG);
      return;
    }
    body_rows_fwd_fixed<T, THREADS, VPT, LGLO, LGHI, LG + 1>(a, bx, by);
  } else if constexpr (LGLO < kFixedLgMin) {
    body_rows_fwd_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, by, a.lg);
  }
}

// FP64: fixed-point lines (fix_passes.cuh)
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_rows_fwd(const RowsFwdArgs<double>& a, int bx);

template <typename T, int THREADS, int VPT, int LGLO = 4, int LGHI = clog2(THREADS * VPT)>
__device__ __forceinline__ void body_rows_fwd(const RowsFwdArgs<T>& a, int bx, int by) {
  if constexpr (sizeof(T) == 8) fx_body_rows_fwd<THREADS, VPT, LGLO, LGHI>(a, bx);
  else body_rows_fwd_fixed<T, THREADS, VPT, LGLO, LGHI, (LGLO > kFixedLgMin ? LGLO : kFixedLgMin)>(a, bx, by);
}

template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_rows_fwd(RowsFwdArgs<T> a) {
  pdl_wait();
  body_rows_fwd<T, THREADS, VPT, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}

// ---------------------------------------------------------------------------
// Operator strided pass: complex FFTs along a slow axis for a tile of TX
// consecutive half-spectrum columns kx.  Line element r of column kx at
// outer index o is S[o * ostride + r * lstride + kx].
template <typename T>
struct ColsArgs {
  typename Cplx<T>::type* S;
  const typename Cplx<T>::type* ptw;   // FP32: the stages' twiddle tables (place_twiddles)
  const T* sig;            // FP32, COLS_CONV: symbol
  const PcgState* st;
  int H, lg, lgmax;
  int rows_in, rows_out;
  long long ostride, lstride;
  int nouter;
  int mode;
  // symbol index = kk * sig_line + min(o, Lo - o) * sig_outer + kx, kk = min(k, L-k)
  long long sig_line, sig_outer;
  int Lo;                  // length of the outer axis in the spectrum (3D: L_1), 0 if unused
  int ltx;                 // log2 of the columns per CTA
  // FP64: twiddles and symbol as fixed-point constants, the symbol divided
  // by 2^sig_exp
  const FxW* ftw;
  const FxR* fsig;
  int sig_exp;
};

// Row of the staged symbol that holds frequency kk: one pad row after every
// 16, since neighbouring blocks of the middle stage are 16 frequencies apart
// (the same bank without the pad).
__device__ __forceinline__ int sig_row(int kk) { return kk + (kk >> 4); }

// FP32.  The tile keeps its natural layout, buf[r * TX + c] (row r of the line,
// column c); its transforms are in place (fft_places): legs of the first stage
// come from global memory, outputs of the last stage go there.  A convolution
// (forward transform, symbol, inverse) takes 2 (S - 1) trips through shared
// memory for S stages.  In 3D the middle axis is kept in the places of its
// transform between its forward and inverse passes (place_frequency).
//
// Bound by instruction issue and shared memory.  Against autosort stages with
// the tile staged first: 256^3 convolution pass 367 -> 337 us, middle-axis
// passes 157, 160 -> 116, 133 us, 1024^2 convolution 24.5 -> 22.4 us (between
// events).
template <typename T, int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void body_cols_at(const ColsArgs<T>& a, int kx0, int by, const int lg,
                                             const int ltx) {
  typedef typename Cplx<T>::type C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SBuf<C> buf{reinterpret_cast<C*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int L = 1 << lg;
  const int TX = 1 << ltx;
  const int o = by;
  const int ncol = min(TX, a.H - kx0);
  C* base = a.S + (size_t)o * a.ostride + kx0;
  // the stages' twiddles (place_twiddles) beside the tile, and for a convolution
  // the symbol's rows kk = 0..L/2 for the tile's columns (row sig_row(kk) of TX
  // values): asynchronous copies that run beside the first stage's loads
  C* stw = reinterpret_cast<C*>(smem_raw + sbuf_elems((long long)TX * L) * sizeof(C));
  const int ntw = place_table_len(lg);
  T* ssig = reinterpret_cast<T*>(smem_raw + (sbuf_elems((long long)TX * L) + ntw) * sizeof(C));
  for (int m = threadIdx.x; m < ntw; m += THREADS) cp_async<sizeof(C)>(&stw[m], &a.ptw[m]);
  const int rows_in = a.rows_in, rows_out = a.rows_out;
  const long long lstride = a.lstride;
  auto mid = [=](int c, int k, int, C v) -> C { return cscale(cswap(v), ssig[(sig_row(min(k, L - k)) << ltx) + c]); };
  auto out = [=](int c, int n, C v) {
    if (c < ncol && n < rows_out) base[(size_t)n * lstride + c] = cswap(v);
  };
  auto ld = [=](int c, int n0, auto lgs, auto cnt, C* v) {
#pragma unroll
    for (int r = 0; r < decltype(cnt)::v; ++r) {
      const int n = n0 + (r << decltype(lgs)::v);
      v[r] = (c < ncol && n < rows_in) ? base[(size_t)n * lstride + c] : cmake<C>((T)0, (T)0);
    }
  };
  if (a.mode == COLS_CONV) {
    const T* FL_RESTRICT sig = a.sig + kx0;
    if (a.Lo) {
      const int f = place_frequency(o, 31 - __clz(a.Lo), VPT);
      sig += (size_t)min(f, a.Lo - f) * a.sig_outer;
    }
    const int nsym = ((L >> 1) + 1) << ltx;
    for (int e = threadIdx.x; e < nsym; e += THREADS) {
      const int kk = e >> ltx, c = e & (TX - 1);
      T* d = ssig + (sig_row(kk) << ltx) + c;
      if (c < ncol) cp_async<sizeof(T)>(d, &sig[(size_t)kk * a.sig_line + c]);
      else *d = (T)0;
    }
    fft_places<PLACE_CONV, VPT, true, LGHI, LGLO, TW_TABLE>(buf, lg, 0, ltx, TX, stw, lg, ld, mid, out);
  } else if (a.mode == COLS_FWD) {
    auto outp = [=](int c, int p, C v) {
      if (c < ncol) base[(size_t)p * lstride + c] = v;
    };
    fft_places<PLACE_FWD, VPT, true, LGHI, LGLO, TW_TABLE>(buf, lg, 0, ltx, TX, stw, lg, ld, mid, outp);
  } else {
    auto ldi = [=](int c, int p0, auto lgs, auto cnt, C* v) {
#pragma unroll
      for (int r = 0; r < decltype(cnt)::v; ++r)
        v[r] = c < ncol ? cswap(base[(size_t)(p0 + (r << decltype(lgs)::v)) * lstride + c]) : cmake<C>((T)0, (T)0);
    };
    fft_places<PLACE_INV, VPT, true, LGHI, LGLO, TW_TABLE>(buf, lg, 0, ltx, TX, stw, lg, ldi, mid, out);
  }
}

// the tile width of column block bx: the plan's, narrowed for a partial
// last tile to the smallest power of two that holds its columns (each
// column's transform is the same at any width)
__device__ __forceinline__ int block_ltx(int ltx, int bx, int ncols) {
  const int left = ncols - (bx << ltx);
  while (ltx > 0 && (1 << (ltx - 1)) >= left) --ltx;
  return ltx;
}

// body_cols for the full tiles of the widest width of lengths 2^LG ..
// 2^LGHI as compile-time shapes, else with runtime shapes
template <typename T, int THREADS, int VPT, int LGLO, int LGHI, int LG>
__device__ __forceinline__ void body_cols_fixed(const ColsArgs<T>& a, int bx, int by) {
  if constexpr (LG <= LGHI) {
    constexpr int W = widest_ltx(THREADS, VPT, LG);
    if (a.lg == LG && a.ltx == W && ((bx + 1) << W) <= a.H) {
      body_cols_at<T, THREADS, VPT, LGLO, LGHI>(a, bx << W, by, LG, W);
      return;
    }
    body_cols_fixed<T, THREADS, VPT, LGLO, LGHI, LG + 1>(a, bx, by);
  } else {
    body_cols_at<T, THREADS, VPT, LGLO, LGHI>(a, bx << a.ltx, by, a.lg, block_ltx(a.ltx, bx, a.H));
  }
}

// FP64: fixed-point lines (fix_passes.cuh)
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_cols(const ColsArgs<double>& a, int bx, int by);

template <typename T, int THREADS, int VPT, int LGLO = 4, int LGHI = clog2(THREADS * VPT)>
__device__ __forceinline__ void body_cols(const ColsArgs<T>& a, int bx, int by) {
  if constexpr (sizeof(T) == 8) fx_body_cols<THREADS, VPT, LGLO, LGHI>(a, bx, by);
  else body_cols_fixed<T, THREADS, VPT, LGLO, LGHI, (LGLO > kFixedLgMin ? LGLO : kFixedLgMin)>(a, bx, by);
}

template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_cols(ColsArgs<T> a) {
  pdl_wait();
  body_cols<T, THREADS, VPT, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}

// ---------------------------------------------------------------------------
// Operator last pass: complex-to-real inverse FFT along the last axis,
// restriction to the first n entries and to Omega, and the epilogue
//   out = cm * (M x) + cx * x + cb * b          (x = the apply's input)
// optionally also written as float (out32), and per-CTA partial sums of
// out . dotw (dotw nullable; dotw == out gives ||out||^2).
template <typename T>
struct RowsInvArgs {
  const typename Cplx<T>::type* S;
  const uint8_t* mask;
  const PcgState* st;
  T* out;                  // nullable
  float* out32;            // nullable
  const T* x;              // nullable
  const T* b;              // nullable
  const T* dotw;           // nullable; if equals out, squares
  double* partials;        // nullable: one per CTA
  double cm, cx, cb;
  int rows, n, H, lg, lgmax;
  int rows_per_plane, plane_stride;
  int dot_self;            // 1: partial = sum out^2
  int fin;                 // FIN_NONE or FIN_PQ (the last CTA sets fst->pq, fst->alpha)
  int nparts;              // CTAs of the pass (partials to sum)
  PcgState* fst;
  T* outm;                 // nullable: M x itself (restricted to Omega)
  const FxW* ftw;          // FP64: twiddles as fixed-point constants
};

template <typename T, int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void body_rows_inv_at(const RowsInvArgs<T>& a, int bx, int by, const int lg) {
  typedef typename Cplx<T>::type C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SBuf<C> buf{reinterpret_cast<C*>(smem_raw)};
  __shared__ double red[32];
  if (a.st && a.st->done) return;
  const int L = 1 << lg;
  const int ls = L;
  const int NL = (VPT * THREADS) / L;
  const int pair0 = bx * NL;
  const int npairs = (a.rows + 1) / 2;
  const int nl = NL == 1 ? 1 : min(NL, npairs - pair0);
  // Z[k] = Xa[k] + i Xb[k];  Z[L-k] = conj(Xa[k]) + i conj(Xb[k]) for the
  // row pair (ra, rb) = (2p, 2p + 1) of line q
  const SpecRows spec(2 * pair0, a.rows_per_plane, a.plane_stride, a.H);
  auto put = [&](int q, int k, C xa, C xb) {
    const SBuf<C> lb = buf.at(q * ls);
    lb[k] = cmake<C>(xa.x - xb.y, xa.y + xb.x);
    if (k > 0 && k < a.H - 1) lb[L - k] = cmake<C>(xa.x + xb.y, xb.x - xa.y);
  };
  // all lines of the CTA in one index space, U spectrum pairs in flight per
  // thread; k = L/2 afterwards
  const int hL = L >> 1;
  const int tot = nl * hL;
  constexpr int U = 4;
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    C xa[U], xb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int dr = 2 * (e >> (lg - 1)), k = e & (hL - 1);
      xa[u] = xb[u] = cmake<C>((T)0, (T)0);
      if (e < tot) {
        xa[u] = a.S[spec(dr) + k];
        if (2 * pair0 + dr + 1 < a.rows) xb[u] = a.S[spec(dr + 1) + k];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      if (e < tot) put(e >> (lg - 1), e & (hL - 1), xa[u], xb[u]);
    }
  }
  for (int q = threadIdx.x; q < nl; q += THREADS) {
    const bool hb = 2 * (pair0 + q) + 1 < a.rows;
    put(q, hL, a.S[spec(2 * q) + hL], hb ? a.S[spec(2 * q + 1) + hL] : cmake<C>((T)0, (T)0));
  }
  __syncthreads();
  const C* const calc = nullptr;   // twiddles are computed
  fft_smem<VPT, false, LGHI, LGLO>(buf, lg, ls, 0, nl, calc, a.lgmax, true);
  DotAcc<T> part;
  const T* FL_RESTRICT xin = (a.cx != 0.0) ? a.x : nullptr;
  const T* FL_RESTRICT bin = (a.cb != 0.0) ? a.b : nullptr;
  const T* FL_RESTRICT win = a.dot_self ? nullptr : a.dotw;
  T* FL_RESTRICT out = a.out;
  float* FL_RESTRICT out32 = a.out32;
  const T cm = (T)a.cm, cx = (T)a.cx, cb = (T)a.cb;
#pragma unroll 2
  for (int e = threadIdx.x; e < tot; e += THREADS) {
    const int q = e >> (lg - 1), j = e & (hL - 1);
    if (j >= a.n) continue;
    const int row = 2 * (pair0 + q);
    const C z = buf[q * ls + j];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (half && row + 1 >= a.rows) break;
      const size_t idx = ((size_t)row + half) * a.n + j;
      const bool off = a.mask && !a.mask[idx];
      const T mx = off ? (T)0 : (half ? z.y : z.x);
      if (a.outm) a.outm[idx] = mx;
      T v = mx * cm;
      if (xin) v += cx * xin[idx];
      if (bin) v += cb * bin[idx];
      if (off) v = (T)0;
      if (out) out[idx] = v;
      if (out32) out32[idx] = (float)v;
      if (a.partials) part.add(win ? v * win[idx] : v * v);
    }
  }
  if (a.partials) {
    const double s = part.cta_total(red);
    if (threadIdx.x == 0) a.partials[bx] = s;
    if (a.fin == FIN_PQ && arrive_last(&a.fst->arrive, a.nparts)) {
      const double pq = cta_sum_partials(a.partials, a.nparts, red);
      if (threadIdx.x == 0) {
        a.fst->pq = pq;
        a.fst->alpha = a.fst->rz / pq;
      }
    }
  }
}

// body_rows_inv with the line length 2^LG .. 2^LGHI as a compile-time
// constant (the lengths below 2^kFixedLgMin at run time)
template <typename T, int THREADS, int VPT, int LGLO, int LGHI, int LG>
__device__ __forceinline__ void body_rows_inv_fixed(const RowsInvArgs<T>& a, int bx, int by) {
  if constexpr (LG <= LGHI) {
    if (a.lg == LG) {
      body_rows_inv_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, by, LG);
      return;
    }
    body_rows_inv_fixed<T, THREADS, VPT, LGLO, LGHI, LG + 1>(a, bx, by);
  } else if constexpr (LGLO < kFixedLgMin) {
    body_rows_inv_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, by, a.lg);
  }
}

// FP64: fixed-point lines (fix_passes.cuh)
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_rows_inv(const RowsInvArgs<double>& a, int bx);

template <typename T, int THREADS, int VPT, int LGLO = 4, int LGHI = clog2(THREADS * VPT)>
__device__ __forceinline__ void body_rows_inv(const RowsInvArgs<T>& a, int bx, int by) {
  if constexpr (sizeof(T) == 8) fx_body_rows_inv<THREADS, VPT, LGLO, LGHI>(a, bx);
  else body_rows_inv_fixed<T, THREADS, VPT, LGLO, LGHI, (LGLO > kFixedLgMin ? LGLO : kFixedLgMin)>(a, bx, by);
}

template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_rows_inv(RowsInvArgs<T> a) {
  pdl_wait();
  body_rows_inv<T, THREADS, VPT, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}

// ---------------------------------------------------------------------------
// Preconditioner: DST-I along the last axis (rows of length n), by chirp-z.
// DPRE_UPDATE fuses the CG update before the transform:
//   alpha = rz / sum(pq partials); x += alpha p; r -= alpha q,
// writing x and r and per-CTA partials of ||r||^2.  The transformed row
// is multiplied by `post` (per-axis DST normalisation) and written to
// `out`; with `dotw` set, per-CTA partials of out . dotw are written.
template <typename T>
struct DstRowsArgs {
  const T* in;             // DPRE_NONE: input rows
  T* out;
  // FP32, n + 1 prime, lines of up to 2^kRowTableLg points: the stages' twiddle
  // tables (row_table_power) of the plans with 16 and with 8 values per thread
  const typename Cplx<T>::type* rtw;
  const typename Cplx<T>::type* rtw8;
  const typename Cplx<T>::type* chirp;   // c_{j+1}, j = 0..n-1
  // FFT_L of conj(c_m) embedded circularly, / L, in the order (row_place) of the
  // stage plans with 16 and with 8 values per thread
  const typename Cplx<T>::type* bhat;
  const typename Cplx<T>::type* bhat8;
  PcgState* st;            // DPRE_UPDATE: alpha from here; FIN_STEP: updated
  // DPRE_UPDATE
  T* x; T* r; const T* p; const T* q;
  double* rr_part;         // per-CTA ||r||^2 (after update)
  const T* dotw; double* dot_part;
  double post;
  int rows, n, lg, lgmax;
  int pre;
  // FIN_STEP (with dotw = r): the last CTA sums rr_in (rr_count partials of
  // the DPRE_UPDATE pass) and its own r.z partials and takes the CG step
  int fin;
  int nparts;
  const double* rr_in; int rr_count;
  // nullable: Omega inside the box (occluded domain).  The first pass zeroes
  // its DPRE_NONE input outside Omega (mask_in), the last pass its output
  // (mask_out): the box solve restricted to Omega, R B^{-1} R^T.
  const uint8_t* mask_in;
  const uint8_t* mask_out;
  int odd;                 // n + 1 = L/2: two rows per complex line (body_dst_rows_odd_at)
  // FP32, n + 1 prime: the orders of Rader's convolution (body_dst_rows_prime_at);
  // lg and bhat are then that convolution's
  const short* perm;
  // nullable (last pass): added to the transformed value before the output
  // mask, out = mask_out ? (B^{-1} in + add) : 0 (the second half of the
  // capacitance solve on an occluded domain)
  const T* add;
  // FP64: twiddles, chirp and chirp kernel as fixed-point constants, the
  // chirp kernel divided by 2^bexp
  const FxW* ftw;
  const FxW* fchirp;
  const FxW* fbhat;
  int bexp;
};

// u_j + i v_j of the prime-length sines from x_j and x_{p-j} (for j > M the
// signs are those of the odd continuation)
template <typename C, typename T>
__device__ __forceinline__ C rader_fold(T xj, T xm, int j) {
  const T s = xj + xm;
  return cmake<C>(xj - xm, (j & 1) ? s : -s);
}

// The partial sums of a DST row pass, and in its last CTA the CG step.
template <typename T>
__device__ __forceinline__ void dst_rows_finish(const DstRowsArgs<T>& a, int bx, DotAcc<T>& rr, DotAcc<T>& dp,
                                                double* red) {
  if (a.pre == DPRE_UPDATE) {
    const double s = rr.cta_total(red);
    if (threadIdx.x == 0) a.rr_part[bx] = s;
  }
  if (a.dotw) {
    const double s = dp.cta_total(red);
    if (threadIdx.x == 0) a.dot_part[bx] = s;
    if (a.fin == FIN_STEP && arrive_last(&a.st->arrive, a.nparts)) {
      const double rrv = cta_sum_partials(a.rr_in, a.rr_count, red);
      const double rz = cta_sum_partials(a.dot_part, a.nparts, red);
      if (threadIdx.x == 0) pcg_step(a.st, rrv, rz);
    }
  }
}

template <typename T, int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void body_dst_rows_at(const DstRowsArgs<T>& a, int bx, int by, const int lg) {
  typedef typename Cplx<T>::type C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SBuf<C> buf{reinterpret_cast<C*>(smem_raw)};
  __shared__ double red[32];
  if (a.st && a.st->done) return;
  const int L = 1 << lg;
  const int ls = L;
  const int NL = (VPT * THREADS) / L;
  const int row0 = bx * NL;
  const int nl = min(NL, a.rows - row0);
  // Both transforms in place (fft_places), the first stage's legs from global
  // memory with all loads before the first use, the sine coefficients from
  // the last stage's registers.  Against autosort stages with the rows staged
  // first: preconditioner 1024^2 32.0 -> 29.5 us, 700 x 1001 27.7 -> 24.9, 200^2
  // 14.6 -> 9.9 (one wave or less, bound by its loads and one CTA's chain).
  DotAcc<T> rr, dp;
  const bool update = a.pre == DPRE_UPDATE;
  const T al = update ? (T)a.st->alpha : (T)0;
  const C* FL_RESTRICT chirp = a.chirp;
  const C* FL_RESTRICT bhat = VPT == 8 ? a.bhat8 : a.bhat;
  const int n = a.n;
  auto ld = [&](int q, int n0, auto lgs, auto cnt, C* v) {
    constexpr int N = decltype(cnt)::v, LGS = decltype(lgs)::v;
    const size_t row = (size_t)(row0 + q) * n;
    T xo[N], ro[N], po[N], qo[N];
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int j = n0 + (r << LGS);
      xo[r] = ro[r] = po[r] = qo[r] = (T)0;
      if (j < n) {
        if (update) {
          xo[r] = a.x[row + j];
          ro[r] = a.r[row + j];
          po[r] = a.p[row + j];
          qo[r] = a.q[row + j];
        } else if (!a.mask_in || a.mask_in[row + j]) {
          ro[r] = a.in[row + j];
        }
      }
    }
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int j = n0 + (r << LGS);
      v[r] = cmake<C>((T)0, (T)0);
      if (j < n) {
        T rn = ro[r];
        if (update) {
          rn = ro[r] - al * qo[r];
          a.x[row + j] = xo[r] + al * po[r];
          a.r[row + j] = rn;
          rr.add(rn * rn);
        }
        v[r] = cscale(chirp[j], rn);
      }
    }
  };
  auto mid = [=](int q, int, int p, C v) -> C { return cswap(cmul(v, bhat[p])); };
  {
    const T post = (T)a.post;
    T* FL_RESTRICT outp = a.out;
    const T* FL_RESTRICT dw = a.dotw;
    const uint8_t* FL_RESTRICT mask = a.mask_out;
    const T* FL_RESTRICT add = a.add;
    // v is swapped: Im(chirp conv) of the value itself
    auto out = [=, &dp](int q, int k, C v) {
      if (k < n) {
        const size_t idx = (size_t)(row0 + q) * n + k;
        const C c = chirp[k];
        const T o = (!mask || mask[idx]) ? (c.x * v.x + c.y * v.y) * post + (add ? add[idx] : (T)0) : (T)0;
        outp[idx] = o;
        if (dw) dp.add(o * dw[idx]);
      }
    };
    const C* const calc = nullptr;   // twiddles are computed
    fft_places<PLACE_CONV, VPT, false, LGHI, LGLO, TW_CALC>(buf, lg, ls, 0, nl, calc, a.lgmax, ld, mid, out);
  }
  dst_rows_finish(a, bx, rr, dp, red);
}

// body_dst_rows with the line length 2^LG .. 2^LGHI as a compile-time
// constant (the lengths below 2^kFixedLgMin at run time)
template <typename T, int THREADS, int VPT, int LGLO, int LGHI, int LG>
__device__ __forceinline__ void body_dst_rows_fixed(const DstRowsArgs<T>& a, int bx, int by) {
  if constexpr (LG <= LGHI) {
    if (a.lg == LG) {
      body_dst_rows_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, by, LG);
      return;
    }
    body_dst_rows_fixed<T, THREADS, VPT, LGLO, LGHI, LG + 1>(a, bx, by);
  } else if constexpr (LGLO < kFixedLgMin) {
    body_dst_rows_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, by, a.lg);
  }
}

// The same where n + 1 is half the line length (n = 2^k - 1, the paper's grids;
// then L = 2 (n + 1)): the odd extension z_{L-j} = -z_j of z = a + i b, two rows
// of sines in one transform of length L, Z_k = -2 i sum_j z_j sin(pi jk/(n+1)).
// The rounding of the pair is that of its larger row.
// One transform per two rows instead of four (a chirp convolution per row):
// preconditioner 1023^2 33.4 -> 22.2 us, 255^3 966 -> 484 us (with the other
// changes since), FP64 511^2 59 -> 38 us.
template <typename T, int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void body_dst_rows_odd_at(const DstRowsArgs<T>& a, int bx, const int lg) {
  typedef typename Cplx<T>::type C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SBuf<C> buf{reinterpret_cast<C*>(smem_raw)};
  __shared__ double red[32];
  if (a.st && a.st->done) return;
  const int L = 1 << lg, hL = L >> 1;
  const int ls = L;
  const int NL = (VPT * THREADS) / L;
  const int pair0 = bx * NL;
  const int nl = NL == 1 ? 1 : min(NL, (a.rows + 1) / 2 - pair0);
  const int n = a.n;
  const bool update = a.pre == DPRE_UPDATE;
  const T al = update ? (T)a.st->alpha : (T)0;
  DotAcc<T> rr, dp;
  const int tot = nl * hL;
  constexpr int U = 2;   // pairs in flight per thread
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    T xo[2 * U], ro[2 * U], po[2 * U], qo[2 * U];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const int e = e0 + (u >> 1) * THREADS;
      const int row = 2 * (pair0 + (e >> (lg - 1))) + (u & 1), i = e & (hL - 1);
      xo[u] = ro[u] = po[u] = qo[u] = (T)0;
      if (e < tot && i > 0 && row < a.rows) {
        const size_t idx = (size_t)row * n + i - 1;
        if (update) {
          xo[u] = a.x[idx];
          ro[u] = a.r[idx];
          po[u] = a.p[idx];
          qo[u] = a.q[idx];
        } else if (!a.mask_in || a.mask_in[idx]) {
          ro[u] = a.in[idx];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const int e = e0 + (u >> 1) * THREADS;
      const int row = 2 * (pair0 + (e >> (lg - 1))) + (u & 1), i = e & (hL - 1);
      if (update && e < tot && i > 0 && row < a.rows) {
        const size_t idx = (size_t)row * n + i - 1;
        ro[u] -= al * qo[u];
        a.x[idx] = xo[u] + al * po[u];
        a.r[idx] = ro[u];
        rr.add(ro[u] * ro[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      if (e < tot) {
        const int q = e >> (lg - 1), i = e & (hL - 1);
        const C z = cmake<C>(ro[2 * u], ro[2 * u + 1]);
        buf[q * ls + i] = z;                                           // i = 0: zero
        buf[q * ls + (i > 0 ? L - i : hL)] = cmake<C>(-z.x, -z.y);     // and at L/2
      }
    }
  }
  __syncthreads();
  {
    const T post = (T)(0.5 * a.post);
    T* FL_RESTRICT outp = a.out;
    const T* FL_RESTRICT dw = a.dotw;
    const uint8_t* FL_RESTRICT mask = a.mask_out;
    const T* FL_RESTRICT add = a.add;
    const int rows = a.rows;
    auto ld = [=](int q, int k) -> C { return buf[q * ls + k]; };
    auto epi = [=, &dp](int q, int k, C v) {
      if (k < 1 || k > n) return;
      const T s[2] = {-v.y * post, v.x * post};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = 2 * (pair0 + q) + h;
        if (row >= rows) break;
        const size_t idx = (size_t)row * n + k - 1;
        const T o = (!mask || mask[idx]) ? s[h] + (add ? add[idx] : (T)0) : (T)0;
        outp[idx] = o;
        if (dw) dp.add(o * dw[idx]);
      }
    };
    const C* const calc = nullptr;   // twiddles are computed
    fft_io<VPT, false, false, LGHI, LGLO>(buf, lg, ls, 0, nl, calc, a.lgmax, false, ld, true, epi, false);
  }
  dst_rows_finish(a, bx, rr, dp, red);
}

template <typename T, int THREADS, int VPT, int LGLO, int LGHI, int LG>
__device__ __forceinline__ void body_dst_rows_odd_fixed(const DstRowsArgs<T>& a, int bx) {
  if constexpr (LG <= LGHI) {
    if (a.lg == LG) {
      body_dst_rows_odd_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, LG);
      return;
    }
    body_dst_rows_odd_fixed<T, THREADS, VPT, LGLO, LGHI, LG + 1>(a, bx);
  } else if constexpr (LGLO < kFixedLgMin) {
    body_dst_rows_odd_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, a.lg);
  }
}

// The same where p = n + 1 is an odd prime (192, 256, 640, 768 points), by a
// convolution of half the length.  With u_j = x_j - x_{p-j}, v_j = (-1)^{j+1}
// (x_j + x_{p-j}) and M = n/2, the sines are S_{2m} = sum_{j=1..M} u_j
// sin(2 pi jm/p) and S_{p-2m} the same of v, and for a generator g of the
// residues modulo p (Rader, Proc. IEEE 56, 1968) the substitution j = g^a, m =
// g^-b makes both the convolution with the real sequence sin(2 pi g^-d / p): one
// complex transform pair of length L >= 2M - 1 carries u + i v, no chirp.  perm:
// g^a mod p for a < M, then for b < M the index 2m (m = +-g^-b in 1..M),
// negative where the sign is.  The rows go through shared memory in their own
// order, so global reads and writes are one contiguous run per CTA.
// By chirp convolutions and so (CUDA graphs): preconditioner 256^3 588 and 292
// us, 192^3 324 and 152, 130^3 155 and 69, 768^2 24.4 and 18.3; few CTAs, one
// chain: 256^2 9.9 and 10.9, 192^2 9.4 and 10.7.  The twiddle tables (TW_ROWS) are
// 7 us of 256^3, 2 of 192^3 and 0.3 of 256^2.
template <typename T, int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void body_dst_rows_prime_at(const DstRowsArgs<T>& a, int bx, const int lg) {
  typedef typename Cplx<T>::type C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SBuf<C> buf{reinterpret_cast<C*>(smem_raw)};
  __shared__ double red[32];
  if (a.st && a.st->done) return;
  const int L = 1 << lg;
  const int ls = L;
  const int NL = (VPT * THREADS) / L;
  const int row0 = bx * NL;
  const int nl = min(NL, a.rows - row0);
  const int n = a.n, M = n >> 1;
  // the stages' twiddles, then the CTA's rows
  C* stw = reinterpret_cast<C*>(smem_raw + sbuf_elems((long long)NL * L) * sizeof(C));
  const int ntw = row_table_len(lg);
  T* xs = reinterpret_cast<T*>(stw + ntw);
  {
    const C* FL_RESTRICT rtw = VPT == 8 ? a.rtw8 : a.rtw;
    for (int m = threadIdx.x; m < ntw; m += THREADS) cp_async<sizeof(C)>(&stw[m], &rtw[m]);
  }
  const size_t base = (size_t)row0 * n;
  const int tot = nl * n;
  constexpr int U = 4;   // elements in flight per thread
  DotAcc<T> rr, dp;
  const bool update = a.pre == DPRE_UPDATE;
  const T al = update ? (T)a.st->alpha : (T)0;
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    T xo[U], ro[U], po[U], qo[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const size_t idx = base + e;
      xo[u] = ro[u] = po[u] = qo[u] = (T)0;
      if (e < tot) {
        if (update) {
          xo[u] = a.x[idx];
          ro[u] = a.r[idx];
          po[u] = a.p[idx];
          qo[u] = a.q[idx];
        } else if (!a.mask_in || a.mask_in[idx]) {
          ro[u] = a.in[idx];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      if (e < tot) {
        if (update) {
          const size_t idx = base + e;
          ro[u] -= al * qo[u];
          a.x[idx] = xo[u] + al * po[u];
          a.r[idx] = ro[u];
          rr.add(ro[u] * ro[u]);
        }
        xs[e] = ro[u];
      }
    }
  }
  cp_async_wait_all();
  __syncthreads();
  {
    const short* FL_RESTRICT perm = a.perm;
    const C* FL_RESTRICT bhat = VPT == 8 ? a.bhat8 : a.bhat;
    const T post = (T)a.post;
    auto ld = [=](int q, int n0, auto lgs, auto cnt, C* v) {
      constexpr int N = decltype(cnt)::v, LGS = decltype(lgs)::v;
      const T* x = xs + q * n;
#pragma unroll
      for (int r = 0; r < N; ++r) {
        const int i = n0 + (r << LGS);
        v[r] = cmake<C>((T)0, (T)0);
        if (i < M) {
          const int j = perm[i];
          v[r] = rader_fold<C>(x[j - 1], x[n - j], j);
        }
      }
    };
    auto mid = [=](int, int, int p, C v) -> C { return cswap(cmul(v, bhat[p])); };
    // every row was read before the first stage's barrier (one thread holds
    // the whole row where there is one stage only)
    auto out = [=](int q, int k, C v) {
      if (k < M) {
        const int m = perm[M + k], i = abs(m);
        const T s = m < 0 ? -post : post;
        xs[q * n + i - 1] = v.y * s;   // v is swapped
        xs[q * n + n - i] = v.x * s;
      }
    };
    fft_places<PLACE_CONV, VPT, false, LGHI, LGLO, TW_ROWS>(buf, lg, ls, 0, nl, stw, lg, ld, mid, out);
  }
  __syncthreads();
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    T ad[U], dw[U];
    bool in[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const size_t idx = base + e;
      in[u] = e < tot && (!a.mask_out || a.mask_out[idx]);
      ad[u] = in[u] && a.add ? a.add[idx] : (T)0;
      dw[u] = e < tot && a.dotw ? a.dotw[idx] : (T)0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      if (e < tot) {
        const T o = in[u] ? xs[e] + ad[u] : (T)0;
        a.out[base + e] = o;
        if (a.dotw) dp.add(o * dw[u]);
      }
    }
  }
  dst_rows_finish(a, bx, rr, dp, red);
}

template <typename T, int THREADS, int VPT, int LGLO, int LGHI, int LG>
__device__ __forceinline__ void body_dst_rows_prime_fixed(const DstRowsArgs<T>& a, int bx) {
  if constexpr (LG <= LGHI) {
    if (a.lg == LG) {
      body_dst_rows_prime_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, LG);
      return;
    }
    body_dst_rows_prime_fixed<T, THREADS, VPT, LGLO, LGHI, LG + 1>(a, bx);
  } else if constexpr (LGLO < kFixedLgMin) {
    body_dst_rows_prime_at<T, THREADS, VPT, LGLO, LGHI>(a, bx, a.lg);
  }
}

// FP64: fixed-point lines (fix_passes.cuh)
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_dst_rows(const DstRowsArgs<double>& a, int bx);
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_dst_rows_odd(const DstRowsArgs<double>& a, int bx);

// by a chirp convolution per row, for a.odd or (FP32) for a.perm
enum { DST_CHIRP = 0, DST_ODD = 1, DST_PRIME = 2 };
template <typename T, int THREADS, int VPT, int FORM, int LGLO = 4, int LGHI = clog2(THREADS * VPT)>
__device__ __forceinline__ void body_dst_rows_as(const DstRowsArgs<T>& a, int bx, int by) {
  constexpr int LG0 = LGLO > kFixedLgMin ? LGLO : kFixedLgMin;
  if constexpr (sizeof(T) == 8) {
    if constexpr (FORM == DST_ODD) fx_body_dst_rows_odd<THREADS, VPT, LGLO, LGHI>(a, bx);
    else fx_body_dst_rows<THREADS, VPT, LGLO, LGHI>(a, bx);
  } else {
    if constexpr (FORM == DST_ODD) body_dst_rows_odd_fixed<T, THREADS, VPT, LGLO, LGHI, LG0>(a, bx);
    else if constexpr (FORM == DST_PRIME) body_dst_rows_prime_fixed<T, THREADS, VPT, LGLO, LGHI, LG0>(a, bx);
    else body_dst_rows_fixed<T, THREADS, VPT, LGLO, LGHI, LG0>(a, bx, by);
  }
}

template <typename T, int THREADS, int VPT, int LGLO = 4, int LGHI = clog2(THREADS * VPT)>
__device__ __forceinline__ void body_dst_rows(const DstRowsArgs<T>& a, int bx, int by) {
  if constexpr (sizeof(T) == 4) {
    if (a.perm) {
      body_dst_rows_as<T, THREADS, VPT, DST_PRIME, LGLO, LGHI>(a, bx, by);
      return;
    }
  }
  if (a.odd) body_dst_rows_as<T, THREADS, VPT, DST_ODD, LGLO, LGHI>(a, bx, by);
  else body_dst_rows_as<T, THREADS, VPT, DST_CHIRP, LGLO, LGHI>(a, bx, by);
}

template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_dst_rows(DstRowsArgs<T> a) {
  pdl_wait();
  body_dst_rows_as<T, THREADS, VPT, DST_CHIRP, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}
template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_dst_rows_odd(DstRowsArgs<T> a) {
  pdl_wait();
  body_dst_rows_as<T, THREADS, VPT, DST_ODD, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}
template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_dst_rows_prime(DstRowsArgs<T> a) {
  pdl_wait();
  body_dst_rows_as<T, THREADS, VPT, DST_PRIME, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}

// ---------------------------------------------------------------------------
// Preconditioner strided pass: DST-I along a slow axis for a tile of TX
// consecutive columns of a real field; line element r of column c at outer
// index o is v[o * ostride + r * lstride + c0 + c] (3D: the middle axis).
template <typename T>
struct DstColsArgs {
  T* v;
  const typename Cplx<T>::type* ptw;   // FP32: the stages' twiddle tables
  const typename Cplx<T>::type* chirp;
  const typename Cplx<T>::type* bhat;
  const PcgState* st;
  double post;
  int n, ncols, lg, lgmax;
  long long ostride, lstride;
  int ltx;
  const short* perm;       // as in DstRowsArgs
  const FxW* ftw;          // FP64: as in DstRowsArgs
  const FxW* fchirp;
  const FxW* fbhat;
  int bexp;
};

template <typename T, int THREADS, int VPT, bool PRIME, int LGLO, int LGHI>
__device__ __forceinline__ void body_dst_cols_at(const DstColsArgs<T>& a, int c0, int by, const int lg,
                                                 const int ltx) {
  typedef typename Cplx<T>::type C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SBuf<C> buf{reinterpret_cast<C*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int L = 1 << lg;
  const int TX = 1 << ltx;
  const int o = by;
  const int ncol = min(TX, a.ncols - c0);
  T* base = a.v + (size_t)o * a.ostride + c0;
  // the stages' twiddles in shared memory (as in body_cols_at)
  C* stw = reinterpret_cast<C*>(smem_raw + sbuf_elems((long long)TX * L) * sizeof(C));
  for (int m = threadIdx.x; m < place_table_len(lg); m += THREADS) cp_async<sizeof(C)>(&stw[m], &a.ptw[m]);
  const int n = a.n;
  const long long lstride = a.lstride;
  const C* FL_RESTRICT chirp = a.chirp;
  const C* FL_RESTRICT bhat = a.bhat;
  const T post = (T)a.post;
  const short* FL_RESTRICT perm = a.perm;
  const int M = n >> 1;
  auto ld = [=](int c, int n0, auto lgs, auto cnt, C* v) {
    constexpr int N = decltype(cnt)::v, LGS = decltype(lgs)::v;
    if constexpr (PRIME) {
      // both rows of a fold once, each a contiguous run of the tile's columns
      T x[N], y[N];
      int j[N];
#pragma unroll
      for (int r = 0; r < N; ++r) {
        const int i = n0 + (r << LGS);
        j[r] = i < M ? perm[i] : 0;
        const bool in = c < ncol && i < M;
        x[r] = in ? base[(size_t)(j[r] - 1) * lstride + c] : (T)0;
        y[r] = in ? base[(size_t)(n - j[r]) * lstride + c] : (T)0;
      }
#pragma unroll
      for (int r = 0; r < N; ++r) v[r] = rader_fold<C>(x[r], y[r], j[r]);
      return;
    }
    T x[N];
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int j = n0 + (r << LGS);
      x[r] = (c < ncol && j < n) ? base[(size_t)j * lstride + c] : (T)0;
    }
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int j = n0 + (r << LGS);
      v[r] = j < n ? cscale(chirp[j], x[r]) : cmake<C>((T)0, (T)0);
    }
  };
  auto mid = [=](int c, int, int p, C v) -> C { return cswap(cmul(v, bhat[p])); };
  auto out = [=](int c, int k, C v) {
    if constexpr (PRIME) {
      if (c < ncol && k < M) {
        const int m = perm[M + k], i = abs(m);
        const T s = m < 0 ? -post : post;
        base[(size_t)(i - 1) * lstride + c] = v.y * s;   // v is swapped
        base[(size_t)(n - i) * lstride + c] = v.x * s;
      }
    } else if (c < ncol && k < n) {
      const C w = chirp[k];   // v is swapped
      base[(size_t)k * lstride + c] = (w.x * v.x + w.y * v.y) * post;
    }
  };
  fft_places<PLACE_CONV, VPT, true, LGHI, LGLO, TW_TABLE>(buf, lg, 0, ltx, TX, stw, lg, ld, mid, out);
}

template <typename T, int THREADS, int VPT, bool PRIME, int LGLO, int LGHI, int LG>
__device__ __forceinline__ void body_dst_cols_fixed(const DstColsArgs<T>& a, int bx, int by) {
  if constexpr (LG <= LGHI) {
    constexpr int W = widest_ltx(THREADS, VPT, LG);
    if (a.lg == LG && a.ltx == W && ((bx + 1) << W) <= a.ncols) {
      body_dst_cols_at<T, THREADS, VPT, PRIME, LGLO, LGHI>(a, bx << W, by, LG, W);
      return;
    }
    body_dst_cols_fixed<T, THREADS, VPT, PRIME, LGLO, LGHI, LG + 1>(a, bx, by);
  } else {
    body_dst_cols_at<T, THREADS, VPT, PRIME, LGLO, LGHI>(a, bx << a.ltx, by, a.lg, block_ltx(a.ltx, bx, a.ncols));
  }
}

// FP64: fixed-point lines (fix_passes.cuh)
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_dst_cols(const DstColsArgs<double>& a, int bx, int by);

template <typename T, int THREADS, int VPT, bool PRIME, int LGLO = 4, int LGHI = clog2(THREADS * VPT)>
__device__ __forceinline__ void body_dst_cols_as(const DstColsArgs<T>& a, int bx, int by) {
  if constexpr (sizeof(T) == 8) fx_body_dst_cols<THREADS, VPT, LGLO, LGHI>(a, bx, by);
  else
    body_dst_cols_fixed<T, THREADS, VPT, PRIME, LGLO, LGHI, (LGLO > kFixedLgMin ? LGLO : kFixedLgMin)>(a, bx, by);
}

template <typename T, int THREADS, int VPT, int LGLO = 4, int LGHI = clog2(THREADS * VPT)>
__device__ __forceinline__ void body_dst_cols(const DstColsArgs<T>& a, int bx, int by) {
  if constexpr (sizeof(T) == 4) {
    if (a.perm) {
      body_dst_cols_as<T, THREADS, VPT, true, LGLO, LGHI>(a, bx, by);
      return;
    }
  }
  body_dst_cols_as<T, THREADS, VPT, false, LGLO, LGHI>(a, bx, by);
}

template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_dst_cols(DstColsArgs<T> a) {
  pdl_wait();
  body_dst_cols_as<T, THREADS, VPT, false, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}
template <typename T, int THREADS, int VPT, int LGLO = 4>
__global__ void __launch_bounds__(THREADS, min_ctas(THREADS, LGLO)) k_dst_cols_prime(DstColsArgs<T> a) {
  pdl_wait();
  body_dst_cols_as<T, THREADS, VPT, true, LGLO>(a, blockIdx.x, blockIdx.y);
  pdl_release();
}

}  // namespace fl

#include "fix_passes.cuh"

namespace fl {

// ---------------------------------------------------------------------------
// Preconditioner solve along axis 0, after the DST-I along the other axes.
// Mode c of the other axes leaves, along axis 0, the tridiagonal system
//   (shift + scale mu_c) z_i + scale cA (2 z_i - z_{i-1} - z_{i+1}) = t_i,
// z_{-1} = z_n = 0 (mu_c: eigenvalue of C h^d L over the other axes, cA =
// c (-a) the stencil weight), i.e. scale cA T_d z = t with
// T_d = tridiag(-1, d, -1), d = 2 + e, e = (shift + scale mu_c)/(scale cA).
// With r = 2 / (d + sqrt(d^2 - 4)) in (0, 1), the root of r^2 - d r + 1 = 0,
// and S the down-shift,
//   T_d = (1/r) (I - r S)(I - r S^T) + r e_0 e_0^T,
// so T_d^{-1} t is two first-order recurrences and a rank-one
// (Sherman-Morrison) correction:
//   y_i = t_i + r y_{i-1},  w_i = y_i + r w_{i+1},  x = r w,
//   z = x - gamma v,  v_i = (r^{i+1} - r^{2n+1-i}) / (1 - r^2),
//   gamma = r x_0 / (1 + r v_0).
// This is the same solve the DST-I along axis 0 would give, in O(n) work.
// Each column runs as kTriSeg segments of m <= kTriM rows, one thread each;
// the segment carries (factor R = r^m) are a linear-recurrence scan across
// the 32 lanes of one warp per column.
//
// FP64 is bound by the FP64 pipe (1.7 operations per clock and SM): eight
// operations per value, one exp2 per segment, and four columns per CTA, so
// that a 2D plan of 512 columns has 128 CTAs (eight columns and twelve
// operations with two exp2 per thread: 36.9 us at 511^2, now 15.8 us, both
// between events).
// FP32 is bound by the latency of its one load and store phase.
template <typename T> constexpr int kTriCols = sizeof(T) == 8 ? 4 : 8;   // columns per CTA: 32-byte row pieces
constexpr int kTriSeg = 32;    // segments per column (one warp lane each)
constexpr int kTriM = 32;      // max rows per segment: n <= 1024
template <typename T> constexpr int kTriTab = sizeof(T) == 8 ? 5 : 4;   // table entries per column

// Per-column constants, data-independent (FP64, once per shift and scale):
// tab[0] = r (rounded to T; every other entry is formed from this r),
// tab[1] = r^m, tab[2] = log2(r), tab[3] = K, with
// gamma / (1 - r^2) = K w_0 (w_0 = r^{-1} x_0), and in FP64 tab[4] = r^e,
// e = 2n + 2 - m S for the S = ceil(n/m) segments that hold rows.
template <typename T>
__global__ void k_tri_table(T* tab, const T* mu_col, const T* mu_outer, int ncols, int n_inner,
                            double shift, double scale, double cA, int n, int m, int diag) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncols) return;
  const double mu = (double)mu_col[c % n_inner] + (mu_outer ? (double)mu_outer[c / n_inner] : 0.0);
  T* o = tab + kTriTab<T> * c;
  if (diag) {
    // no stencil along axis 0 (a 1D problem): z = t / (shift + scale mu)
    o[0] = (T)(1.0 / (shift + scale * mu));
    for (int i = 1; i < kTriTab<T>; ++i) o[i] = (T)0;
    return;
  }
  const double e = (shift + scale * mu) / (scale * cA);
  const T rt = (T)(2.0 / (2.0 + e + sqrt(e * (e + 4.0))));
  const double r = (double)rt;
  const double lr = log1p(-(1.0 - r));
  const double omr2 = (1.0 - r) * (1.0 + r);
  const double v0 = (r - exp((2.0 * n + 1.0) * lr)) / omr2;
  o[0] = rt;
  o[1] = (T)exp((double)m * lr);
  o[2] = (T)(lr * 1.4426950408889634073599246810018921);
  o[3] = (T)(r * r / ((1.0 + r * v0) * omr2));
  if constexpr (sizeof(T) == 8) o[4] = (T)exp((2.0 * n + 2.0 - (double)m * ((n + m - 1) / m)) * lr);
}

template <typename T>
struct TriArgs {
  T* v;                  // in: coefficients t; out: z (in place); row stride ncols
  const PcgState* st;
  const T* tab;          // k_tri_table for this shift and scale
  double inv_sc;         // 1 / (scale cA)
  int n;                 // rows along axis 0
  int ncols;             // columns: product of the other axes
  int m;                 // rows per segment, ceil(n / kTriSeg)
  int diag;              // 1D problem (n = 1, no stencil along axis 0): z = t * tab[0]
};

__device__ __forceinline__ float tri_exp2(float x) { return exp2f(x); }
__device__ __forceinline__ double tri_exp2(double x) { return exp2(x); }

// Inclusive scan of b_s = E_s + R b_{s-1} over the lanes (up: s = lane;
// down: s counted from lane 31).
template <typename T>
__device__ __forceinline__ T lane_scan(T b, T R, bool up) {
  const int lane = threadIdx.x & 31;
  T Rd = R;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T o = up ? __shfl_up_sync(0xffffffffu, b, d) : __shfl_down_sync(0xffffffffu, b, d);
    if (up ? lane >= d : lane + d < 32) b += Rd * o;
    Rd *= Rd;
  }
  return b;
}

// TC columns per CTA of TC * kTriSeg threads (warp w scans column w), up to M
// rows per segment.  FP32.
template <typename T, int TC, int M>
__device__ __forceinline__ void body_tri_cols_f32(const TriArgs<T>& a, int bx) {
  __shared__ T s_e[kTriSeg][TC + 1];   // segment end values (forward, backward)
  __shared__ T s_c[kTriSeg][TC + 1];   // carries into each segment
  __shared__ T s_w0[TC];
  if (a.st && a.st->done) return;
  if (a.diag) {
    const int dc = bx * TC + (int)threadIdx.x;
    if ((int)threadIdx.x < TC && dc < a.ncols) a.v[dc] *= a.tab[kTriTab<T> * dc];
    return;
  }
  const int c = threadIdx.x % TC, s = threadIdx.x / TC;
  const int col = bx * TC + c;
  const bool act = col < a.ncols;
  const int n = a.n, m = a.m, i0 = s * m;
  T* FL_RESTRICT vc = a.v + col;
  const size_t ld = (size_t)a.ncols;
  T y[M];
#pragma unroll
  for (int j = 0; j < M; ++j)
    y[j] = (act && j < m && i0 + j < n) ? vc[(size_t)(i0 + j) * ld] : (T)0;
  T r = (T)0, R = (T)0, l2r = (T)0, K = (T)0;
  if (act) {
    r = a.tab[kTriTab<T> * col];
    R = a.tab[kTriTab<T> * col + 1];
    l2r = a.tab[kTriTab<T> * col + 2];
    K = a.tab[kTriTab<T> * col + 3];
  }
  // scan lanes: warp w scans column w, lane = segment
  const int wc = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wcol = bx * TC + wc;
  const T wR = wcol < a.ncols ? a.tab[kTriTab<T> * wcol + 1] : (T)0;
  // forward recurrence within the segment
  {
    T acc = (T)0;
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < m) {
        acc = y[j] + r * acc;
        y[j] = acc;
      }
    s_e[s][c] = acc;
  }
  __syncthreads();
  {
    const T b = lane_scan(s_e[lane][wc], wR, true);
    const T ex = __shfl_up_sync(0xffffffffu, b, 1);
    s_c[lane][wc] = lane > 0 ? ex : (T)0;
  }
  __syncthreads();
  {
    const T cin = s_c[s][c];
    T pw = r;
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < m) {
        y[j] = (i0 + j < n) ? y[j] + pw * cin : (T)0;
        pw *= r;
      }
  }
  // backward recurrence within the segment
  {
    T acc = (T)0;
#pragma unroll
    for (int j = M - 1; j >= 0; --j)
      if (j < m) {
        acc = y[j] + r * acc;
        y[j] = acc;
      }
    s_e[s][c] = acc;
  }
  __syncthreads();
  {
    const T b = lane_scan(s_e[lane][wc], wR, false);
    const T ex = __shfl_down_sync(0xffffffffu, b, 1);
    s_c[lane][wc] = lane < 31 ? ex : (T)0;
    if (lane == 0) s_w0[wc] = b;   // w_0 of the column
  }
  __syncthreads();
  if (!act || i0 >= n) return;
  const T g = K * s_w0[c];
  const T inv_sc = (T)a.inv_sc;
  // z_i = (r w_i - g (r^{i+1} - r^{2n+1-i})) / (scale cA), w_i = w_local + r^{m-j} cin
  {
    T p = tri_exp2(l2r * (T)(i0 + 1));
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < m) {
        y[j] = r * y[j] - g * p;
        p *= r;
      }
  }
  {
    const T cin = s_c[s][c];
    T pw = r * r;
    T qv = tri_exp2(l2r * (T)(2 * n + 2 - i0 - m));
#pragma unroll
    for (int j = M - 1; j >= 0; --j)
      if (j < m) {
        y[j] = (y[j] + pw * cin + g * qv) * inv_sc;
        pw *= r;
        qv *= r;
      }
  }
#pragma unroll
  for (int j = 0; j < M; ++j)
    if (j < m && i0 + j < n) vc[(size_t)(i0 + j) * ld] = y[j];
}

// FP64: one exp2 per segment, eight operations per value.
template <typename T, int TC, int M>
__device__ __forceinline__ void body_tri_cols_f64(const TriArgs<T>& a, int bx) {
  __shared__ T s_e[kTriSeg][TC + 1];   // segment end values (forward, backward)
  __shared__ T s_c[kTriSeg][TC + 1];   // carries into each segment
  __shared__ T s_p[kTriSeg][TC + 1];   // r^(m s)
  __shared__ T s_w0[TC];
  if (a.st && a.st->done) return;
  if (a.diag) {
    const int dc = bx * TC + (int)threadIdx.x;
    if ((int)threadIdx.x < TC && dc < a.ncols) a.v[dc] *= a.tab[kTriTab<T> * dc];
    return;
  }
  const int c = threadIdx.x % TC, s = threadIdx.x / TC;
  const int col = bx * TC + c;
  const bool act = col < a.ncols;
  const int n = a.n, m = a.m, i0 = s * m;
  T* FL_RESTRICT vc = a.v + col;
  const size_t ld = (size_t)a.ncols;
  T y[M];
#pragma unroll
  for (int j = 0; j < M; ++j)
    y[j] = (act && j < m && i0 + j < n) ? vc[(size_t)(i0 + j) * ld] : (T)0;
  T r = (T)0, K = (T)0, qe = (T)0;
  if (act) {
    r = a.tab[kTriTab<T> * col];
    K = a.tab[kTriTab<T> * col + 3];
    qe = a.tab[kTriTab<T> * col + 4];
  }
  // scan lanes: warp w scans column w, lane = segment
  const int wc = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wcol = bx * TC + wc;
  const T wR = wcol < a.ncols ? a.tab[kTriTab<T> * wcol + 1] : (T)0;
  // (log2 r is -infinity where r rounds to nothing beside 1)
  s_p[lane][wc] = lane == 0 ? (T)1 : (wcol < a.ncols ? tri_exp2(a.tab[kTriTab<T> * wcol + 2] * (T)(lane * m)) : (T)0);
  // forward recurrence within the segment
  {
    T acc = (T)0;
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < m) {
        acc = y[j] + r * acc;
        y[j] = acc;
      }
    s_e[s][c] = acc;
  }
  __syncthreads();
  {
    const T b = lane_scan(s_e[lane][wc], wR, true);
    const T ex = __shfl_up_sync(0xffffffffu, b, 1);
    s_c[lane][wc] = lane > 0 ? ex : (T)0;
  }
  __syncthreads();
  {
    T t = r * s_c[s][c];
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < m) {
        y[j] = (i0 + j < n) ? y[j] + t : (T)0;
        t *= r;
      }
  }
  // backward recurrence within the segment
  {
    T acc = (T)0;
#pragma unroll
    for (int j = M - 1; j >= 0; --j)
      if (j < m) {
        acc = y[j] + r * acc;
        y[j] = acc;
      }
    s_e[s][c] = acc;
  }
  __syncthreads();
  {
    const T b = lane_scan(s_e[lane][wc], wR, false);
    const T ex = __shfl_down_sync(0xffffffffu, b, 1);
    s_c[lane][wc] = lane < 31 ? ex : (T)0;
    if (lane == 0) s_w0[wc] = b;   // w_0 of the column
  }
  __syncthreads();
  if (!act || i0 >= n) return;
  const T inv_sc = (T)a.inv_sc;
  const T g = K * s_w0[c];
  // z_i = (r w_i - g (r^{i+1} - r^{2n+1-i})) / (scale cA), w_i = w_local + r^{m-j} cin:
  // one term falling like r^j and one like r^{m-1-j}
  {
    const T ri = r * inv_sc;
    T t = -g * (r * s_p[s][c]) * inv_sc;
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < m) {
        y[j] = ri * y[j] + t;
        t *= r;
      }
  }
  {
    const int last = (n + m - 1) / m - 1;
    T t = (r * r * s_c[s][c] + g * (qe * s_p[last - s][c])) * inv_sc;
#pragma unroll
    for (int j = M - 1; j >= 0; --j)
      if (j < m) {
        y[j] += t;
        t *= r;
      }
  }
#pragma unroll
  for (int j = 0; j < M; ++j)
    if (j < m && i0 + j < n) vc[(size_t)(i0 + j) * ld] = y[j];
}

// The body for m <= M rows per segment: with M = 32 throughout, a 3D plan of
// 256^3 (m = 8) spent most of its instructions on rows that are not there
// and held one CTA per SM (149 us, now 42 us); 24 where 32 would leave a
// quarter of them empty (preconditioner 640^2 17.76 -> 17.45 us, 768^2 18.56 ->
// 18.16, 700 x 1001 25.07 -> 24.86), in single launches only: the batched and the
// persistent kernels hold every variant in one body, and take 32 there.
template <typename T, int TC, int M>
__device__ __forceinline__ void body_tri_cols_m(const TriArgs<T>& a, int bx) {
  if constexpr (sizeof(T) == 8) body_tri_cols_f64<T, TC, M>(a, bx);
  else body_tri_cols_f32<T, TC, M>(a, bx);
}

template <typename T, int TC = kTriCols<T>>
__device__ __forceinline__ void body_tri_cols(const TriArgs<T>& a, int bx) {
  if (a.m <= 8) body_tri_cols_m<T, TC, 8>(a, bx);
  else if (a.m <= 16) body_tri_cols_m<T, TC, 16>(a, bx);
  else body_tri_cols_m<T, TC, kTriM>(a, bx);
}

template <typename T, int M>
__global__ void __launch_bounds__(kTriCols<T> * kTriSeg) k_tri_cols(TriArgs<T> a) {
  pdl_wait();
  body_tri_cols_m<T, kTriCols<T>, M>(a, blockIdx.x);
  pdl_release();
}

}  // namespace fl
