// The FP64 passes (operator apply and preconditioner DSTs) on 64-bit
// fixed-point lines: shared-memory FFT stages on Fx values and the pass
// bodies that kernels.cuh's FP64 instantiations run.  Inputs and outputs are
// FP64 arrays; see fix_core.cuh for the arithmetic.
//
// A pass stages its FP64 tile in shared memory as it is, finds each line's
// largest exponent (the key below), converts in the first stage's loads and
// converts back in the last stage's stores.  The inverse transform is the
// forward one with the real and imaginary parts swapped on the way in and
// out.  Lines have exponents of their own, so that results do not depend on
// the tile width.
//
// The FP64 forms of these passes were bound by the FP64 pipe (82 % busy at
// 1.7 operations per clock and SM).  These are bound by the integer pipes
// (math-pipe throttle is the largest stall, issue 0.5 to 0.64 per cycle);
// FP64 instructions are left in the epilogues only (two to six per output).
// Measured on one GB300 in CUDA graphs, FP64 form -> this one: applies 64^2 154
// -> 39 us, 512^2 208 -> 57 us, 1024^2 507 -> 139 us, 256^3 13.0 -> 3.1 ms;
// preconditioner solves (with the tridiagonal pass's change) 147 -> 34, 200 ->
// 60, 710 -> 166 us and 16.9 -> 3.5 ms.
#pragma once

namespace fl {

// Exponent key of an FP64 value: upper word of |v|, nonzero for every v != 0.
__device__ __forceinline__ unsigned fx_key(double v) {
  const unsigned lo = (unsigned)__double2loint(v);
  return ((unsigned)__double2hiint(v) & 0x7fffffffu) | (lo < 1u ? lo : 1u);
}
// exponent field of a line with largest key `key`; a line of zeros takes
// that of 1.0, so that its exponent stays in the normal range
__device__ __forceinline__ int fx_line_field(unsigned key) {
  return key == 0u ? 1023 : max((int)(key >> 20), 1);
}

// FP64 values that may leave the normal range, and the lines with non-finite
// inputs
static __device__ __noinline__ double fx_to_wide(long long f, int X) {
  if (X > kFxBad / 2) return __longlong_as_double(0x7ff8000000000000ll);
  return ldexp((double)f, X);
}
__device__ __forceinline__ double fx_to(long long f, int X) {
  return fx_x_normal(X) ? fx_to_normal(f, X) : fx_to_wide(f, X);
}

// Record the magnitude bits m of line `line` (every thread of the warp calls
// it; m = 0 from threads without a butterfly).  IL: lanes 2^ltx apart share a
// line; else runs of 2^LGRUN lanes (a whole warp from 32 up).
template <bool IL, int LGRUN>
__device__ __forceinline__ void fx_note(unsigned* mx, int line, unsigned m, int ltx) {
  const int lane = threadIdx.x & 31;
  if constexpr (IL) {
    for (int o = 16; o >> ltx; o >>= 1) m |= __shfl_xor_sync(0xffffffffu, m, o);
    if ((lane >> ltx) == 0 && m) atomicOr(mx + line, m);
  } else if constexpr (LGRUN >= 5) {
    m = __reduce_or_sync(0xffffffffu, m);
    if (lane == 0 && m) atomicOr(mx + line, m);
  } else {
#pragma unroll
    for (int o = (1 << LGRUN) >> 1; o > 0; o >>= 1) m |= __shfl_xor_sync(0xffffffffu, m, o);
    if ((lane & ((1 << LGRUN) - 1)) == 0 && m) atomicOr(mx + line, m);
  }
}

// One stage (see stage_ct): legs are shifted up by their line's headroom
// (bits recorded by the stage before), divided by 8 and summed.
// load(line, index, c) gives the first stage's legs, already divided by 8
// (c: the line's word of slot 0); epi(line, index, value, X, ctx)
// takes the last stage's outputs and returns their magnitude bits.
template <int R, int VPT, bool IL, int LG, int NS, int ST, int MODE, bool HALF, bool HOUT, typename Load,
          typename Epi>
__device__ __forceinline__ void fx_stage(SBuf<Fx> buf, int ls, int ltx, int nlines, const FxW* FL_RESTRICT tw,
                                         int lgmax, unsigned* mx, int cap, unsigned* mx_out, Load& load,
                                         Epi& epi, bool sync_io) {
  typedef FftPlan<LG, VPT> P;
  constexpr int NB = VPT / R;
  constexpr int LR = LogR<R>::v;
  constexpr int LGLR = LG - LR;
  constexpr int RUN = 1 << LGLR;
  const int total = IL ? (RUN << ltx) : (nlines << LGLR);
  const int rd_stride = IL ? sbuf_phys(RUN << ltx) : sbuf_phys(RUN);
  const int wr_stride = IL ? sbuf_phys(NS << ltx) : sbuf_phys(NS);
  Fx v[NB][R];
  int line_of[NB], out0[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int g = threadIdx.x + b * blockDim.x;
    out0[b] = -1;
    line_of[b] = 0;
    if (g < total) {
      const int line = IL ? (g & ((1 << ltx) - 1)) : (g >> LGLR);
      const int j = IL ? (g >> ltx) : (g & (RUN - 1));
      const int k = j & (NS - 1);
      const unsigned c = mx[ST * cap + line];
      if constexpr (MODE == STAGE_FIRST) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          v[b][r] = (HALF && 2 * r >= R) ? Fx{0, 0} : load(line, j + r * RUN, c);
      } else {
        const int sh = fx_headroom(c);
        const int l0 = IL ? ((j << ltx) + line) : (line * ls + j);
        if ((IL ? ((RUN << ltx) & 15) : (RUN & 15)) == 0) {
          const Fx* p0 = buf.p + sbuf_phys(l0);
#pragma unroll
          for (int r = 0; r < R; ++r) v[b][r] = fx_shl(p0[r * rd_stride], sh);
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) v[b][r] = fx_shl(buf[l0 + (IL ? ((r * RUN) << ltx) : r * RUN)], sh);
        }
        const int step = k << (lgmax - clog2(NS * R));
        v[b][0] = fx_shr<kFxShift>(v[b][0]);
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = fx_mul(v[b][r], tw[r * step]);
      }
      fx_dft<R>(v[b]);
      line_of[b] = line;
      out0[b] = (j - k) * R + k;
    }
  }
  if (MODE == STAGE_MID || sync_io) __syncthreads();
  unsigned m = 0u;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (out0[b] >= 0) {
      if constexpr (MODE == STAGE_LAST) {
        // exponent change over the transform, X of this line relative to its
        // input
        int X = kFxShift;
#pragma unroll
        for (int s = 1; s < P::S; ++s) X += kFxShift - fx_headroom(mx[s * cap + line_of[b]]);
        epi.begin(line_of[b], X, mx[line_of[b]]);
        // HOUT: only the lower half of the line is wanted
#pragma unroll
        for (int r = 0; r < (HOUT ? R / 2 : R); ++r) m |= epi(line_of[b], out0[b] + r * NS, v[b][r]);
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) m |= fx_mag(v[b][r].x) | fx_mag(v[b][r].y);
        const int d0 = IL ? ((out0[b] << ltx) + line_of[b]) : (line_of[b] * ls + out0[b]);
        if (!IL && NS == 1) {
          Fx* p0 = buf.p + sbuf_phys(d0);
#pragma unroll
          for (int r = 0; r < R; ++r) p0[r] = v[b][r];
        } else if ((IL ? ((NS << ltx) & 15) : (NS & 15)) == 0) {
          Fx* p0 = buf.p + sbuf_phys(d0);
#pragma unroll
          for (int r = 0; r < R; ++r) p0[r * wr_stride] = v[b][r];
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) buf[d0 + (IL ? ((r * NS) << ltx) : r * NS)] = v[b][r];
        }
      }
    }
    // interleaved: a thread's butterflies are all of one line
    if (!IL || b == NB - 1) {
      if (MODE != STAGE_LAST) fx_note<IL, LGLR>(mx + (ST + 1) * cap, IL ? (int)(threadIdx.x & ((1 << ltx) - 1)) : line_of[b], m, ltx);
      else if (Epi::kNote) fx_note<IL, LGLR>(mx_out, IL ? (int)(threadIdx.x & ((1 << ltx) - 1)) : line_of[b], m, ltx);
      m = 0u;
    }
  }
  if constexpr (MODE != STAGE_LAST) __syncthreads();
}

template <int LG, int VPT, bool IL, bool HALF, bool HOUT, int ST, typename Load, typename Epi>
__device__ __forceinline__ void fx_stages(SBuf<Fx> buf, int ls, int ltx, int nlines, const FxW* FL_RESTRICT tw,
                                          int lgmax, unsigned* mx, int cap, unsigned* mx_out, Load& load,
                                          bool sync_load, Epi& epi, bool sync_epi) {
  typedef FftPlan<LG, VPT> P;
  constexpr int R = P::radix(ST);
  constexpr int MODE = ST == 0 ? STAGE_FIRST : (ST == P::S - 1 ? STAGE_LAST : STAGE_MID);
  fx_stage<R, VPT, IL, LG, P::ns(ST), ST, MODE, HALF, HOUT>(buf, ls, ltx, nlines, tw, lgmax, mx, cap, mx_out,
                                                            load, epi,
                                                            MODE == STAGE_FIRST ? sync_load : sync_epi);
  if constexpr (ST + 1 < P::S)
    fx_stages<LG, VPT, IL, HALF, HOUT, ST + 1>(buf, ls, ltx, nlines, tw, lgmax, mx, cap, mx_out, load, sync_load,
                                               epi, sync_epi);
}

// A transform of `nlines` lines of length 2^lg.  mx: P::S slots of `cap`
// words; slot 0 holds the input's word per line (an exponent key or
// magnitude bits, as load takes it), the others start at zero.  Magnitude
// bits of the outputs are recorded in mx_out where epi asks for it.  The
// caller separates the writes of slot 0 from the call by a barrier.
template <int LG, int VPT, bool IL, bool HALF, bool HOUT, typename Load, typename Epi>
__device__ __forceinline__ void fx_fft_ct(SBuf<Fx> buf, int ls, int ltx, int nlines, const FxW* FL_RESTRICT tw,
                                          int lgmax, unsigned* mx, int cap, unsigned* mx_out, Load load,
                                          bool sync_load, Epi epi, bool sync_epi) {
  static_assert(FftPlan<LG, VPT>::S >= 2, "a first and a last stage");
  fx_stages<LG, VPT, IL, HALF, HOUT, 0>(buf, ls, ltx, nlines, tw, lgmax, mx, cap, mx_out, load, sync_load, epi,
                                        sync_epi);
}

#define FL_FX_LEN(LGV)                                                                                  \
  if constexpr (LGV >= LGLO && LGV <= LGHI) {                                                           \
    if (lg == LGV) {                                                                                    \
      fx_fft_ct<LGV, VPT, IL, HALF, HOUT>(buf, ls, ltx, nlines, tw, lgmax, mx, cap, mx_out, load,       \
                                          sync_load, epi, sync_epi);                                    \
      return;                                                                                           \
    }                                                                                                   \
  }
template <int VPT, bool IL, bool HALF, bool HOUT, int LGLO, int LGHI, typename Load, typename Epi>
__device__ __forceinline__ void fx_fft(SBuf<Fx> buf, int lg, int ls, int ltx, int nlines,
                                       const FxW* FL_RESTRICT tw, int lgmax, unsigned* mx, int cap,
                                       unsigned* mx_out, Load load, bool sync_load, Epi epi, bool sync_epi) {
  FL_FX_LEN(13)
  FL_FX_LEN(12)
  FL_FX_LEN(11)
  FL_FX_LEN(10)
  FL_FX_LEN(9)
  FL_FX_LEN(8)
  FL_FX_LEN(7)
  FL_FX_LEN(6)
  FL_FX_LEN(5)
  FL_FX_LEN(4)
}
#undef FL_FX_LEN

// Words of line bookkeeping of a CTA of THREADS x VPT values: per transform
// S slots of one word per line, at most 2 x VALUES/16 (length 16: two slots;
// the longer lengths have fewer lines).
constexpr int fx_words(int threads, int vpt, int lglo) {
  return lglo > 4 ? 8 : threads * vpt / 8;
}
template <int N>
__device__ __forceinline__ void fx_zero(unsigned* w) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) w[i] = 0u;
}

// --- loads and epilogues ----------------------------------------------------------

// FP64 complex values staged as they are
struct FxLoadRaw {
  SBuf<Fx> buf;
  int ls, ltx;
  bool il, swap;
  __device__ __forceinline__ Fx operator()(int q, int k, unsigned key) const {
    const Fx w = il ? buf[(k << ltx) + q] : buf[q * ls + k];
    const int E = fx_line_field(key);
    const Fx v = Fx{fx_from<kFxShift>(__longlong_as_double(w.x), E), fx_from<kFxShift>(__longlong_as_double(w.y), E)};
    return swap ? fx_swap(v) : v;
  }
};
// fixed-point values of an earlier transform; swapped for the inverse
struct FxLoadFix {
  SBuf<Fx> buf;
  int ls, ltx;
  bool il;
  __device__ __forceinline__ Fx operator()(int q, int k, unsigned m) const {
    const Fx v = il ? buf[(k << ltx) + q] : buf[q * ls + k];
    return fx_swap(fx_shr<kFxShift>(fx_shl(v, fx_headroom(m))));
  }
};
// FP64 real values (in .x of the staged element) times the chirp
struct FxLoadChirp {
  SBuf<Fx> buf;
  const FxW* FL_RESTRICT chirp;
  int ls, ltx, n;
  bool il;
  __device__ __forceinline__ Fx operator()(int q, int k, unsigned key) const {
    if (k >= n) return Fx{0, 0};
    const Fx w = il ? buf[(k << ltx) + q] : buf[q * ls + k];
    const long long x = fx_from<0>(__longlong_as_double(w.x), fx_line_field(key));
    const FxW c = chirp[k];
    return Fx{fx_mul_real(x, FxR{c.xh, c.xl}), fx_mul_real(x, FxR{c.yh, c.yl})};
  }
};
// outputs back into the buffer, the line's exponent into xs
struct FxStore {
  static constexpr bool kNote = false;
  SBuf<Fx> buf;
  int ls;
  int* xs;
  __device__ __forceinline__ void begin(int q, int X, unsigned key) { xs[q] = fx_x0(fx_line_field(key)) + X; }
  __device__ __forceinline__ unsigned operator()(int q, int k, Fx v) {
    buf[q * ls + k] = v;
    return 0u;
  }
};
// outputs times a per-index complex constant (the chirp kernel's transform),
// back into the buffer
struct FxMulStore {
  static constexpr bool kNote = true;
  SBuf<Fx> buf;
  const FxW* FL_RESTRICT w;
  int* xs;
  int ls, ltx, wexp;
  bool il;
  __device__ __forceinline__ void begin(int q, int X, unsigned key) { xs[q] = fx_x0(fx_line_field(key)) + X + wexp + kFxShift; }
  __device__ __forceinline__ unsigned operator()(int q, int k, Fx v) {
    v = fx_mul(v, w[k]);
    if (il) buf[(k << ltx) + q] = v;
    else buf[q * ls + k] = v;
    return fx_mag(v.x) | fx_mag(v.y);
  }
};
// outputs times the kernel symbol (rows 0..L/2 staged in shared memory)
struct FxSymStore {
  static constexpr bool kNote = true;
  SBuf<Fx> buf;
  const FxR* sig;
  int* xs;
  int ltx, L, wexp;
  __device__ __forceinline__ void begin(int q, int X, unsigned key) { xs[q] = fx_x0(fx_line_field(key)) + X + wexp + kFxShift; }
  __device__ __forceinline__ unsigned operator()(int q, int k, Fx v) {
    v = fx_mul_real(v, sig[(min(k, L - k) << ltx) + q]);
    buf[(k << ltx) + q] = v;
    return fx_mag(v.x) | fx_mag(v.y);
  }
};
// strided-pass outputs to global memory as FP64
struct FxOut {
  static constexpr bool kNote = false;
  double2* base;
  long long lstride;
  const int* xs;     // exponent of the transform's input (second transform), or null: an FP64 input
  int ncol, rows_out;
  bool swap;
  int X;
  __device__ __forceinline__ void begin(int q, int dX, unsigned w) {
    // second transform: its input was shifted up by the headroom of w
    X = xs ? xs[q] + dX - fx_headroom(w) : fx_x0(fx_line_field(w)) + dX;
  }
  __device__ __forceinline__ unsigned operator()(int c, int k, Fx v) {
    if (c < ncol && k < rows_out) {
      if (swap) v = fx_swap(v);
      double2 o;
      o.x = fx_to(v.x, X);
      o.y = fx_to(v.y, X);
      base[(size_t)k * lstride + c] = o;
    }
    return 0u;
  }
};

// --- operator pass 1 (see body_rows_fwd_at) ---------------------------------------
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_rows_fwd(const RowsFwdArgs<double>& a, int bx) {
  constexpr int W = fx_words(THREADS, VPT, LGLO);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_mx[W];
  __shared__ int s_x[W];
  const SBuf<Fx> buf{reinterpret_cast<Fx*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int lg = a.lg, L = 1 << lg, ls = L;
  const int NL = (VPT * THREADS) >> lg;
  const int pair0 = bx * NL;
  const int npairs = (a.rows + 1) / 2;
  const int nl = NL == 1 ? 1 : min(NL, npairs - pair0);
  fx_zero<W>(s_mx);
  __syncthreads();
  const double beta = (a.pre == PRE_PUPDATE) ? a.st->beta : 0.0;
  constexpr int U = 4;
  const int hL = L >> 1;
  const int tot = nl * hL;
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    double va[U], vb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int q = e >> (lg - 1), j = e & (hL - 1);
      const int ra = 2 * (pair0 + q), rb = ra + 1;
      va[u] = 0.0;
      vb[u] = 0.0;
      if (e < tot && j < a.n) {
        const size_t ia = (size_t)ra * a.n + j, ib = (size_t)rb * a.n + j;
        const bool hb = rb < a.rows;
        if (a.pre == PRE_PUPDATE) {
          // beta == 0 (first iteration): p = z, without reading the old p
          va[u] = beta != 0.0 ? a.u[ia] + beta * a.p[ia] : a.u[ia];
          if (hb) vb[u] = beta != 0.0 ? a.u[ib] + beta * a.p[ib] : a.u[ib];
        } else if (a.pre == PRE_ACCUM) {
          va[u] = a.acc[ia] + (double)a.x32[ia];
          if (hb) vb[u] = a.acc[ib] + (double)a.x32[ib];
        } else {
          va[u] = a.u[ia];
          if (hb) vb[u] = a.u[ib];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int q = e >> (lg - 1), j = e & (hL - 1);
      const int ra = 2 * (pair0 + q), rb = ra + 1;
      double xa = va[u], xb = vb[u];
      if (e < tot && j < a.n) {
        const size_t ia = (size_t)ra * a.n + j, ib = (size_t)rb * a.n + j;
        const bool hb = rb < a.rows;
        if (a.pre == PRE_PUPDATE) {
          a.p[ia] = xa;
          if (hb) a.p[ib] = xb;
        } else if (a.pre == PRE_ACCUM) {
          a.acc[ia] = xa;
          if (hb) a.acc[ib] = xb;
        }
        if (a.mask) {
          if (!a.mask[ia]) xa = 0.0;
          if (hb && !a.mask[ib]) xb = 0.0;
        }
      }
      unsigned key = max(fx_key(xa), fx_key(xb));
      if (e < tot) buf[q * ls + j] = Fx{__double_as_longlong(xa), __double_as_longlong(xb)};
      if (hL >= 32) {
        // tot is a multiple of 32: whole warps, each on one line
        key = __reduce_max_sync(0xffffffffu, key);
        if (e < tot && (threadIdx.x & 31) == 0 && key) atomicMax(s_mx + q, key);
      } else if (e < tot && key) {
        atomicMax(s_mx + q, key);
      }
    }
  }
  __syncthreads();
  fx_fft<VPT, false, true, false, LGLO, LGHI>(buf, lg, ls, 0, nl, a.ftw, a.lgmax, s_mx, NL, s_mx + NL,
                                              FxLoadRaw{buf, ls, 0, false, false}, true,
                                              FxStore{buf, ls, s_x}, true);
  __syncthreads();
  // k = 0 also writes k = L/2
  const SpecRows spec(2 * pair0, a.rows_per_plane, a.plane_stride, a.H);
  for (int e = threadIdx.x; e < tot; e += THREADS) {
    const int q = e >> (lg - 1);
    const bool hb = 2 * (pair0 + q) + 1 < a.rows;
    double2* Sa = a.S + spec(2 * q);
    double2* Sb = a.S + spec(2 * q + 1);
    const SBuf<Fx> lb = buf.at(q * ls);
    const int X = s_x[q];
    for (int k = e & (hL - 1); k <= hL; k += hL) {
      const Fx z = lb[k], w = lb[(L - k) & (L - 1)];
      // halved before the sums, which could pass 2^63
      const long long zx = z.x >> 1, zy = z.y >> 1, wx = w.x >> 1, wy = w.y >> 1;
      Sa[k] = make_double2(fx_to(zx + wx, X), fx_to(zy - wy, X));
      if (hb) Sb[k] = make_double2(fx_to(zy + wy, X), fx_to(wx - zx, X));
      if (k > 0) break;
    }
  }
}

// --- operator strided pass (see body_cols_at) ---------------------------------------
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_cols(const ColsArgs<double>& a, int bx, int by) {
  constexpr int W = fx_words(THREADS, VPT, LGLO);
  constexpr int U = 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_mx[2 * W];
  __shared__ int s_x[1 << kMaxLtx];
  const SBuf<Fx> buf{reinterpret_cast<Fx*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int lg = a.lg, L = 1 << lg;
  const int kx0 = bx << a.ltx;
  const int ltx = block_ltx(a.ltx, bx, a.H);
  const int TX = 1 << ltx;
  const int o = by;
  const int ncol = min(TX, a.H - kx0);
  double2* base = a.S + (size_t)o * a.ostride + kx0;
  const int hL = L >> 1;
  // FWD and CONV: rows_in <= L/2, only the lower half of the tile is staged
  const int total = TX * (a.mode == COLS_INV ? L : hL);
  FxR* ssig = reinterpret_cast<FxR*>(smem_raw + sbuf_elems((long long)TX * L) * sizeof(Fx));
  const FxR* FL_RESTRICT sig = a.fsig + kx0;
  if (a.mode == COLS_CONV && a.Lo) sig += (size_t)min(o, a.Lo - o) * a.sig_outer;
  const int nsym = a.mode == COLS_CONV ? ((hL + 1) << ltx) : 0;
  for (int e = threadIdx.x; e < nsym; e += THREADS) {
    const int kk = e >> ltx, c = e & (TX - 1);
    if (c < ncol) cp_async<sizeof(FxR)>(&ssig[e], &sig[(size_t)kk * a.sig_line + c]);
    else ssig[e] = FxR{0, 0};
  }
  fx_zero<2 * W>(s_mx);
  __syncthreads();
  unsigned key = 0u;   // all of a thread's elements are of column threadIdx.x mod TX
  for (int e0 = threadIdx.x; e0 < total; e0 += THREADS * U) {
    double2 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int r = e >> ltx, c = e & (TX - 1);
      v[u] = make_double2(0.0, 0.0);
      if (e < total && r < a.rows_in && c < ncol) v[u] = base[(size_t)r * a.lstride + c];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      key = max(key, max(fx_key(v[u].x), fx_key(v[u].y)));
      if (e < total) buf[e] = Fx{__double_as_longlong(v[u].x), __double_as_longlong(v[u].y)};
    }
  }
  for (int s = 16; s >> ltx; s >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, s));
  if (((threadIdx.x & 31) >> ltx) == 0 && key) atomicMax(s_mx + (threadIdx.x & (TX - 1)), key);
  cp_async_wait_all();
  __syncthreads();
  const int cap = TX;
  unsigned* mx2 = s_mx + W;
  if (a.mode == COLS_CONV) {
    fx_fft<VPT, true, true, false, LGLO, LGHI>(buf, lg, 0, ltx, TX, a.ftw, a.lgmax, s_mx, cap, mx2,
                                               FxLoadRaw{buf, 0, ltx, true, false}, true,
                                               FxSymStore{buf, ssig, s_x, ltx, L, a.sig_exp}, true);
    __syncthreads();
    fx_fft<VPT, true, false, true, LGLO, LGHI>(buf, lg, 0, ltx, TX, a.ftw, a.lgmax, mx2, cap, mx2 + cap,
                                               FxLoadFix{buf, 0, ltx, true}, true,
                                               FxOut{base, a.lstride, s_x, ncol, a.rows_out, true, 0}, false);
  } else if (a.mode == COLS_FWD) {
    fx_fft<VPT, true, true, false, LGLO, LGHI>(buf, lg, 0, ltx, TX, a.ftw, a.lgmax, s_mx, cap, mx2,
                                               FxLoadRaw{buf, 0, ltx, true, false}, true,
                                               FxOut{base, a.lstride, nullptr, ncol, a.rows_out, false, 0}, false);
  } else {
    fx_fft<VPT, true, false, true, LGLO, LGHI>(buf, lg, 0, ltx, TX, a.ftw, a.lgmax, s_mx, cap, mx2,
                                               FxLoadRaw{buf, 0, ltx, true, true}, true,
                                               FxOut{base, a.lstride, nullptr, ncol, a.rows_out, true, 0}, false);
  }
}

// the lower half of the line holds the n <= L/2 values kept; the exponent
// change of the transform goes to dx
struct FxRowsInvEpi {
  static constexpr bool kNote = false;
  SBuf<Fx> buf;
  int ls;
  unsigned* dx;
  __device__ __forceinline__ void begin(int q, int X, unsigned m) { dx[q] = (unsigned)(X - fx_headroom(m)); }
  __device__ __forceinline__ unsigned operator()(int q, int k, Fx v) {
    buf[q * ls + k] = v;
    return 0u;
  }
};

// --- operator last pass (see body_rows_inv_at) ---------------------------------------
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_rows_inv(const RowsInvArgs<double>& a, int bx) {
  constexpr int W = fx_words(THREADS, VPT, LGLO);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_mx[W];
  __shared__ unsigned s_key[W];
  __shared__ int s_x[W];
  __shared__ double red[32];
  const SBuf<Fx> buf{reinterpret_cast<Fx*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int lg = a.lg, L = 1 << lg, ls = L, hL = L >> 1;
  const int NL = (VPT * THREADS) >> lg;
  const int pair0 = bx * NL;
  const int npairs = (a.rows + 1) / 2;
  const int nl = NL == 1 ? 1 : min(NL, npairs - pair0);
  fx_zero<W>(s_mx);
  fx_zero<W>(s_key);
  __syncthreads();
  const SpecRows spec(2 * pair0, a.rows_per_plane, a.plane_stride, a.H);
  // Staged as they are: xa[k] at k and xb[k] at L - k for 0 < k < L/2; at
  // k = 0 and L/2 the sum xa + i xb itself (both by the thread of k = 0).
  const int tot = nl * hL;
  constexpr int U = 4;
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    double2 va[U], vb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int dr = 2 * (e >> (lg - 1)), k = e & (hL - 1);
      va[u] = vb[u] = make_double2(0.0, 0.0);
      if (e < tot) {
        va[u] = a.S[spec(dr) + k];
        if (2 * pair0 + dr + 1 < a.rows) vb[u] = a.S[spec(dr + 1) + k];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int q = e >> (lg - 1), k = e & (hL - 1);
      unsigned key = 0u;
      if (e < tot) {
        const SBuf<Fx> lb = buf.at(q * ls);
        double2 xa = va[u], xb = vb[u];
        if (k == 0) {
          const double2 ya = a.S[spec(2 * q) + hL];
          const double2 yb = 2 * (pair0 + q) + 1 < a.rows ? a.S[spec(2 * q + 1) + hL] : make_double2(0.0, 0.0);
          xa = make_double2(xa.x - xb.y, xa.y + xb.x);
          xb = make_double2(ya.x - yb.y, ya.y + yb.x);
        }
        key = max(max(fx_key(xa.x), fx_key(xa.y)), max(fx_key(xb.x), fx_key(xb.y)));
        lb[k] = Fx{__double_as_longlong(xa.x), __double_as_longlong(xa.y)};
        lb[k == 0 ? hL : L - k] = Fx{__double_as_longlong(xb.x), __double_as_longlong(xb.y)};
      }
      if (hL >= 32) {
        key = __reduce_max_sync(0xffffffffu, key);
        if (e < tot && (threadIdx.x & 31) == 0 && key) atomicMax(s_key + q, key);
      } else if (key) {
        atomicMax(s_key + q, key);
      }
    }
  }
  __syncthreads();
  // Z[k] = xa[k] + i xb[k], Z[L-k] = conj xa[k] + i conj xb[k], in place
  // (each pair of places by one thread); inputs below 2^61, sums below 2^62
  for (int e = threadIdx.x; e < tot; e += THREADS) {
    const int q = e >> (lg - 1), k = e & (hL - 1);
    const SBuf<Fx> lb = buf.at(q * ls);
    const int E = fx_line_field(s_key[q]);
    const int k2 = k == 0 ? hL : L - k;
    const Fx ra = lb[k], rb = lb[k2];
    Fx z = Fx{fx_from<1>(__longlong_as_double(ra.x), E), fx_from<1>(__longlong_as_double(ra.y), E)};
    Fx zc = Fx{fx_from<1>(__longlong_as_double(rb.x), E), fx_from<1>(__longlong_as_double(rb.y), E)};
    if (k > 0) {
      const Fx xa = z, xb = zc;
      z = Fx{xa.x - xb.y, xa.y + xb.x};
      zc = Fx{xa.x + xb.y, xb.x - xa.y};
    } else {
      s_x[q] = fx_x0(E) + 1;
    }
    lb[k] = z;
    lb[k2] = zc;
    unsigned m = fx_mag(z.x) | fx_mag(z.y) | fx_mag(zc.x) | fx_mag(zc.y);
    if (hL >= 32) {
      m = __reduce_or_sync(0xffffffffu, m);
      if ((threadIdx.x & 31) == 0 && m) atomicOr(s_mx + q, m);
    } else if (m) {
      atomicOr(s_mx + q, m);
    }
  }
  __syncthreads();
  fx_fft<VPT, false, false, true, LGLO, LGHI>(buf, lg, ls, 0, nl, a.ftw, a.lgmax, s_mx, NL, s_mx + NL,
                                              FxLoadFix{buf, ls, 0, false}, true, FxRowsInvEpi{buf, ls, s_key}, true);
  __syncthreads();
  DotAcc<double> part;
  const double* FL_RESTRICT xin = (a.cx != 0.0) ? a.x : nullptr;
  const double* FL_RESTRICT bin = (a.cb != 0.0) ? a.b : nullptr;
  const double* FL_RESTRICT win = a.dot_self ? nullptr : a.dotw;
  double* FL_RESTRICT out = a.out;
  float* FL_RESTRICT out32 = a.out32;
  const double cm = a.cm, cx = a.cx, cb = a.cb;
#pragma unroll 2
  for (int e = threadIdx.x; e < tot; e += THREADS) {
    const int q = e >> (lg - 1), j = e & (hL - 1);
    if (j >= a.n) continue;
    const int row = 2 * (pair0 + q);
    const int X = s_x[q] + (int)s_key[q];
    const Fx z = buf[q * ls + j];   // swapped: .y is the real part (row a), .x the imaginary (row b)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (half && row + 1 >= a.rows) break;
      const size_t idx = ((size_t)row + half) * a.n + j;
      const bool off = a.mask && !a.mask[idx];
      const double mx = off ? 0.0 : fx_to(half ? z.x : z.y, X);
      if (a.outm) a.outm[idx] = mx;
      double v = cm == 1.0 ? mx : mx * cm;
      if (xin) v += cx * xin[idx];
      if (bin) v += cb * bin[idx];
      if (off) v = 0.0;
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

// sine coefficients Im(c_k v) of a row, with their dot product
struct FxDstRowsEpi {
  static constexpr bool kNote = false;
  const DstRowsArgs<double>& a;
  const int* xs;
  DotAcc<double>& dp;
  int row0, X;
  __device__ __forceinline__ void begin(int q, int dX, unsigned m) {
    X = xs[q] + dX - fx_headroom(m) + kFxShift;   // + kFxShift: the chirp product below
  }
  __device__ __forceinline__ unsigned operator()(int q, int k, Fx v) {
    if (k < a.n) {
      const size_t idx = (size_t)(row0 + q) * a.n + k;
      double o = 0.0;
      if (!a.mask_out || a.mask_out[idx]) {
        o = fx_to(fx_mul_im(fx_swap(v), a.fchirp[k]), X);
        if (a.post != 1.0) o *= a.post;
        if (a.add) o += a.add[idx];
      }
      a.out[idx] = o;
      if (a.dotw) dp.add(o * a.dotw[idx]);
    }
    return 0u;
  }
};

// --- preconditioner rows (see body_dst_rows_at) ---------------------------------------
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_dst_rows(const DstRowsArgs<double>& a, int bx) {
  constexpr int W = fx_words(THREADS, VPT, LGLO);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_mx[2 * W];
  __shared__ int s_x[W];
  __shared__ double red[32];
  const SBuf<Fx> buf{reinterpret_cast<Fx*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int lg = a.lg, L = 1 << lg, ls = L;
  const int NL = (VPT * THREADS) >> lg;
  const int row0 = bx * NL;
  const int nl = min(NL, a.rows - row0);
  fx_zero<2 * W>(s_mx);
  __syncthreads();
  DotAcc<double> rr;
  const int hL = L >> 1;
  const int tot = nl * hL;
  const bool update = a.pre == DPRE_UPDATE;
  const double al = update ? a.st->alpha : 0.0;
  constexpr int U = 4;
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    double xo[U], ro[U], po[U], qo[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int q = e >> (lg - 1), j = e & (hL - 1);
      xo[u] = ro[u] = po[u] = qo[u] = 0.0;
      if (e < tot && j < a.n) {
        const size_t idx = (size_t)(row0 + q) * a.n + j;
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
      const int q = e >> (lg - 1), j = e & (hL - 1);
      double v = ro[u];
      if (update && e < tot && j < a.n) {
        const size_t idx = (size_t)(row0 + q) * a.n + j;
        v = ro[u] - al * qo[u];
        a.x[idx] = xo[u] + al * po[u];
        a.r[idx] = v;
        rr.add(v * v);
      }
      unsigned key = fx_key(v);
      if (e < tot) buf[q * ls + j].x = __double_as_longlong(v);
      if (hL >= 32) {
        key = __reduce_max_sync(0xffffffffu, key);
        if (e < tot && (threadIdx.x & 31) == 0 && key) atomicMax(s_mx + q, key);
      } else if (e < tot && key) {
        atomicMax(s_mx + q, key);
      }
    }
  }
  __syncthreads();
  unsigned* mx2 = s_mx + W;
  fx_fft<VPT, false, true, false, LGLO, LGHI>(buf, lg, ls, 0, nl, a.ftw, a.lgmax, s_mx, NL, mx2,
                                              FxLoadChirp{buf, a.fchirp, ls, 0, a.n, false}, true,
                                              FxMulStore{buf, a.fbhat, s_x, ls, 0, a.bexp, false}, true);
  __syncthreads();
  DotAcc<double> dp;
  fx_fft<VPT, false, false, true, LGLO, LGHI>(buf, lg, ls, 0, nl, a.ftw, a.lgmax, mx2, NL, mx2 + NL,
                                              FxLoadFix{buf, ls, 0, false}, true, FxDstRowsEpi{a, s_x, dp, row0, 0}, false);
  dst_rows_finish(a, bx, rr, dp, red);
}

// sine coefficients of a pair of rows: Z = -2 i (S_a + i S_b)
struct FxDstOddEpi {
  static constexpr bool kNote = false;
  const DstRowsArgs<double>& a;
  DotAcc<double>& dp;
  int pair0, X;
  __device__ __forceinline__ void begin(int q, int dX, unsigned key) { X = fx_x0(fx_line_field(key)) + dX - 1; }
  __device__ __forceinline__ unsigned operator()(int q, int k, Fx v) {
    if (k < 1 || k > a.n) return 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = 2 * (pair0 + q) + h;
      if (row >= a.rows) break;
      const size_t idx = (size_t)row * a.n + k - 1;
      double o = 0.0;
      if (!a.mask_out || a.mask_out[idx]) {
        o = fx_to(h ? v.x : -v.y, X);
        if (a.post != 1.0) o *= a.post;
        if (a.add) o += a.add[idx];
      }
      a.out[idx] = o;
      if (a.dotw) dp.add(o * a.dotw[idx]);
    }
    return 0u;
  }
};

// --- preconditioner rows, n + 1 = L/2 (see body_dst_rows_odd_at) -----------------------
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_dst_rows_odd(const DstRowsArgs<double>& a, int bx) {
  constexpr int W = fx_words(THREADS, VPT, LGLO);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_mx[W];
  __shared__ double red[32];
  const SBuf<Fx> buf{reinterpret_cast<Fx*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int lg = a.lg, L = 1 << lg, ls = L, hL = L >> 1;
  const int NL = (VPT * THREADS) >> lg;
  const int pair0 = bx * NL;
  const int nl = NL == 1 ? 1 : min(NL, (a.rows + 1) / 2 - pair0);
  fx_zero<W>(s_mx);
  __syncthreads();
  DotAcc<double> rr, dp;
  const int tot = nl * hL;
  const bool update = a.pre == DPRE_UPDATE;
  const double al = update ? a.st->alpha : 0.0;
  constexpr int U = 2;   // pairs in flight per thread
  for (int e0 = threadIdx.x; e0 < tot; e0 += THREADS * U) {
    double xo[2 * U], ro[2 * U], po[2 * U], qo[2 * U];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const int e = e0 + (u >> 1) * THREADS;
      const int row = 2 * (pair0 + (e >> (lg - 1))) + (u & 1), i = e & (hL - 1);
      xo[u] = ro[u] = po[u] = qo[u] = 0.0;
      if (e < tot && i > 0 && row < a.rows) {
        const size_t idx = (size_t)row * a.n + i - 1;
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
        const size_t idx = (size_t)row * a.n + i - 1;
        ro[u] -= al * qo[u];
        a.x[idx] = xo[u] + al * po[u];
        a.r[idx] = ro[u];
        rr.add(ro[u] * ro[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int q = e >> (lg - 1), i = e & (hL - 1);
      const double va = ro[2 * u], vb = ro[2 * u + 1];
      unsigned key = max(fx_key(va), fx_key(vb));
      if (e < tot) {
        buf[q * ls + i] = Fx{__double_as_longlong(va), __double_as_longlong(vb)};   // i = 0: zero, and at L/2
        buf[q * ls + (i > 0 ? L - i : hL)] = Fx{__double_as_longlong(-va), __double_as_longlong(-vb)};
      }
      if (hL >= 32) {
        key = __reduce_max_sync(0xffffffffu, key);
        if (e < tot && (threadIdx.x & 31) == 0 && key) atomicMax(s_mx + q, key);
      } else if (e < tot && key) {
        atomicMax(s_mx + q, key);
      }
    }
  }
  __syncthreads();
  fx_fft<VPT, false, false, true, LGLO, LGHI>(buf, lg, ls, 0, nl, a.ftw, a.lgmax, s_mx, NL, s_mx + NL,
                                              FxLoadRaw{buf, ls, 0, false, false}, true,
                                              FxDstOddEpi{a, dp, pair0, 0}, false);
  dst_rows_finish(a, bx, rr, dp, red);
}

// sine coefficients of a column tile
struct FxDstColsEpi {
  static constexpr bool kNote = false;
  const DstColsArgs<double>& a;
  double* base;
  const int* xs;
  int ncol, X;
  __device__ __forceinline__ void begin(int q, int dX, unsigned m) {
    X = xs[q] + dX - fx_headroom(m) + kFxShift;   // + kFxShift: the chirp product below
  }
  __device__ __forceinline__ unsigned operator()(int c, int k, Fx v) {
    if (c < ncol && k < a.n) {
      double o = fx_to(fx_mul_im(fx_swap(v), a.fchirp[k]), X);
      if (a.post != 1.0) o *= a.post;
      base[(size_t)k * a.lstride + c] = o;
    }
    return 0u;
  }
};

// --- preconditioner strided pass (see body_dst_cols_at) -------------------------------
template <int THREADS, int VPT, int LGLO, int LGHI>
__device__ __forceinline__ void fx_body_dst_cols(const DstColsArgs<double>& a, int bx, int by) {
  constexpr int W = fx_words(THREADS, VPT, LGLO);
  constexpr int U = 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_mx[2 * W];
  __shared__ int s_x[1 << kMaxLtx];
  const SBuf<Fx> buf{reinterpret_cast<Fx*>(smem_raw)};
  if (a.st && a.st->done) return;
  const int lg = a.lg, L = 1 << lg;
  const int c0 = bx << a.ltx;
  const int ltx = block_ltx(a.ltx, bx, a.ncols);
  const int TX = 1 << ltx;
  const int ncol = min(TX, a.ncols - c0);
  double* base = a.v + (size_t)by * a.ostride + c0;
  const int total = TX * (L >> 1);
  fx_zero<2 * W>(s_mx);
  __syncthreads();
  unsigned key = 0u;
  for (int e0 = threadIdx.x; e0 < total; e0 += THREADS * U) {
    double v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      const int r = e >> ltx, c = e & (TX - 1);
      v[u] = 0.0;
      if (e < total && r < a.n && c < ncol) v[u] = base[(size_t)r * a.lstride + c];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * THREADS;
      key = max(key, fx_key(v[u]));
      if (e < total) buf[e].x = __double_as_longlong(v[u]);
    }
  }
  for (int s = 16; s >> ltx; s >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, s));
  if (((threadIdx.x & 31) >> ltx) == 0 && key) atomicMax(s_mx + (threadIdx.x & (TX - 1)), key);
  __syncthreads();
  unsigned* mx2 = s_mx + W;
  fx_fft<VPT, true, true, false, LGLO, LGHI>(buf, lg, 0, ltx, TX, a.ftw, a.lgmax, s_mx, TX, mx2,
                                             FxLoadChirp{buf, a.fchirp, 0, ltx, a.n, true}, true,
                                             FxMulStore{buf, a.fbhat, s_x, 0, ltx, a.bexp, true}, true);
  __syncthreads();
  fx_fft<VPT, true, false, true, LGLO, LGHI>(buf, lg, 0, ltx, TX, a.ftw, a.lgmax, mx2, TX, mx2 + TX,
                                             FxLoadFix{buf, 0, ltx, true}, true, FxDstColsEpi{a, base, s_x, ncol, 0}, false);
}

}  // namespace fl
