// 64-bit fixed-point complex arithmetic and its shared-memory FFT: what the
// FP64 passes transform with.
//
// GB300 issues 1.7 FP64 operations per clock and SM, but 61 32 x 32 ->
// 64-bit multiply-adds (IMAD.WIDE, with a 64-bit addend) and 126 32-bit
// additions (all measured).  A complex addition is 4 integer instructions
// instead of 2 FP64 ones, a complex multiplication about 20 (12 of them
// IMAD.WIDE) instead of 4: a radix-8 butterfly with its twiddles takes a
// tenth of the time on the integer pipes.
//
// Numbers.  A line of the transform is block floating point: every component
// is a signed 64-bit integer f, the value is f 2^X with one exponent X per
// line.  Loads from FP64 take X from the line's largest exponent; each stage
// records the bits its outputs use (the OR of their magnitudes' upper words,
// per line) and the next stage first shifts the line left by the headroom
// that is left, so that a stage always works near the top of the 64 bits.
// All moduli stay below 2^62.5: a stage divides its inputs by 8 (in the
// twiddle multiplication itself) before summing up to 8 of them.  Rounding
// therefore enters at about 2^-60 of the line's largest value per stage,
// below the 2^-53 of every single FP64 operation that it replaces.  Relative
// 2-norm errors of one transform against extended precision, lines of 16 ..
// 8192 values, six kinds of data: up to 4e-17, 7e-17 once the outputs are
// rounded to FP64; FP64 radix-2 arithmetic up to 2.7e-16.
//
// The error is absolute, one size for the whole line: a value below about 2^-8
// of its line's largest keeps fewer than 53 bits of its own (an FP64 transform
// spreads its rounding over the line in the same way, but reads such a value
// exactly).  The same holds for constants that share an exponent: the kernel
// symbol (one for the array) and the chirp spectra (one per axis); and for the
// two rows that share a complex line, of the operator's passes and of the odd
// extension.
//
// Twiddles, chirps and the kernel symbol are constants w, |w| <= 1, with 61
// fraction bits, split as w 2^61 = h 2^32 + l, |l| < 2^31.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define FL_HD __host__ __device__ __forceinline__
#else
#define FL_HD inline
#endif

namespace fl {

struct alignas(16) Fx { long long x, y; };
// a complex constant: (h 2^32 + l) / 2^61 per component
struct alignas(16) FxW { int xh, xl, yh, yl; };
// a real constant
struct alignas(8) FxR { int h, l; };

constexpr int kFxFrac = 61;       // fraction bits of the constants
constexpr int kFxShift = 64 - kFxFrac;   // a product is divided by 2^kFxShift = 8
// X of a line whose FP64 input holds an infinity or a NaN: its outputs are NaN
constexpr int kFxBad = 1 << 20;

// v = hi 2^32 + lo with lo in [-2^31, 2^31)
FL_HD int fx_hi(long long v) { return (int)(v >> 32) + (int)((unsigned)v >> 31); }
FL_HD int fx_lo(long long v) { return (int)v; }
FL_HD long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }

// the split of a constant (-2^31 is left out of the low half: it is negated)
FL_HD constexpr FxR fx_real(long long q) {
  const int h = (int)((q + (1ll << 31)) >> 32);
  const long long l = q - ((long long)h << 32);
  return FxR{h, l == -(1ll << 31) ? (int)(l + 1) : (int)l};
}

// upper word of |v| (one below for negative v): the OR of these over a line
// has the bit length of its largest component
FL_HD unsigned fx_mag(long long v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h >> 31));
}
FL_HD int fx_clz(unsigned v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}
// left shift that brings components with magnitude bits m below 2^62
FL_HD int fx_headroom(unsigned m) {
  const int s = fx_clz(m) - 2;
  return s > 0 ? s : 0;
}
FL_HD long long fx_shl(long long v, int s) { return (long long)((unsigned long long)v << s); }
FL_HD Fx fx_shl(Fx v, int s) { return Fx{fx_shl(v.x, s), fx_shl(v.y, s)}; }
// v / 2^S rounded to nearest
template <int S> FL_HD long long fx_shr(long long v) { return S > 0 ? (v + (1ll << (S > 0 ? S - 1 : 0))) >> S : v; }
template <int S> FL_HD Fx fx_shr(Fx v) { return Fx{fx_shr<S>(v.x), fx_shr<S>(v.y)}; }

FL_HD Fx fx_add(Fx a, Fx b) { return Fx{a.x + b.x, a.y + b.y}; }
FL_HD Fx fx_sub(Fx a, Fx b) { return Fx{a.x - b.x, a.y - b.y}; }
FL_HD Fx fx_swap(Fx a) { return Fx{a.y, a.x}; }

// v w / 8.  With v = vh 2^32 + vl the product is H 2^64 + M 2^32 + vl wl,
// H = vh wh, M = vh wl + vl wh, so that v w 2^61 / 2^64 = H + M / 2^32: the
// upper word of M is the addend of H's first multiply-add.  |v| < 2^62.5
// keeps M within 2^63.  The constant in M's sum rounds it to nearest (zero
// gives zero); the dropped vl wl / 2^64 is below half a unit.
constexpr long long kFxRound = 1ll << 31;
FL_HD long long fx_carry(long long M) { return (long long)(int)(M >> 32); }

FL_HD Fx fx_mul(Fx v, FxW w) {
  const int xh = fx_hi(v.x), xl = fx_lo(v.x), yh = fx_hi(v.y), yl = fx_lo(v.y);
  const long long mx = fx_mad(xh, w.xl, fx_mad(xl, w.xh, fx_mad(yh, -w.yl, fx_mad(yl, -w.yh, kFxRound))));
  const long long my = fx_mad(xh, w.yl, fx_mad(xl, w.yh, fx_mad(yh, w.xl, fx_mad(yl, w.xh, kFxRound))));
  return Fx{fx_mad(xh, w.xh, fx_mad(yh, -w.yh, fx_carry(mx))), fx_mad(xh, w.yh, fx_mad(yh, w.xh, fx_carry(my)))};
}
// imaginary part of v w / 8
FL_HD long long fx_mul_im(Fx v, FxW w) {
  const int xh = fx_hi(v.x), xl = fx_lo(v.x), yh = fx_hi(v.y), yl = fx_lo(v.y);
  const long long m = fx_mad(xh, w.yl, fx_mad(xl, w.yh, fx_mad(yh, w.xl, fx_mad(yl, w.xh, kFxRound))));
  return fx_mad(xh, w.yh, fx_mad(yh, w.xh, fx_carry(m)));
}
// v times a real constant / 8
FL_HD long long fx_mul_real(long long v, FxR w) {
  const int h = fx_hi(v), l = fx_lo(v);
  return fx_mad(h, w.h, fx_carry(fx_mad(h, w.l, fx_mad(l, w.h, kFxRound))));
}
FL_HD Fx fx_mul_real(Fx v, FxR w) { return Fx{fx_mul_real(v.x, w), fx_mul_real(v.y, w)}; }

// --- butterflies (forward) ----------------------------------------------------

// v sqrt(1/2) = v - v (1 - sqrt(1/2)), the constant with 64 fraction bits
// (below 1/2, so that its upper half fits 32 signed bits)
constexpr unsigned long long kFx1mH = 5402926248376769404ull;
FL_HD long long fx_half(long long v) {
  constexpr FxR w = fx_real((long long)kFx1mH);
  const int h = fx_hi(v), l = fx_lo(v);
  return v - fx_mad(h, w.h, fx_carry(fx_mad(h, w.l, fx_mad(l, w.h, kFxRound))));
}
// v exp(-i pi / 4) and v exp(-3 i pi / 4)
FL_HD Fx fx_rot45(Fx v) { return Fx{fx_half(v.x + v.y), fx_half(v.y - v.x)}; }
FL_HD Fx fx_rot135(Fx v) { return Fx{fx_half(v.y - v.x), -fx_half(v.x + v.y)}; }
FL_HD Fx fx_mi(Fx v) { return Fx{v.y, -v.x}; }

FL_HD void fx_dft2(Fx* v) {
  const Fx a = v[0], b = v[1];
  v[0] = fx_add(a, b);
  v[1] = fx_sub(a, b);
}
FL_HD void fx_dft4(Fx* v) {
  const Fx t0 = fx_add(v[0], v[2]), t1 = fx_sub(v[0], v[2]);
  const Fx t2 = fx_add(v[1], v[3]), t3 = fx_sub(v[1], v[3]);
  v[0] = fx_add(t0, t2);
  v[2] = fx_sub(t0, t2);
  v[1] = Fx{t1.x + t3.y, t1.y - t3.x};
  v[3] = Fx{t1.x - t3.y, t1.y + t3.x};
}
FL_HD void fx_dft8(Fx* v) {
  Fx e[4] = {v[0], v[2], v[4], v[6]};
  Fx o[4] = {v[1], v[3], v[5], v[7]};
  fx_dft4(e);
  fx_dft4(o);
  o[1] = fx_rot45(o[1]);
  o[2] = fx_mi(o[2]);
  o[3] = fx_rot135(o[3]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = fx_add(e[k], o[k]);
    v[k + 4] = fx_sub(e[k], o[k]);
  }
}
template <int R> FL_HD void fx_dft(Fx* v) {
  static_assert(R <= 8, "stages of at most 8 legs");
  if constexpr (R == 2) fx_dft2(v);
  else if constexpr (R == 4) fx_dft4(v);
  else fx_dft8(v);
}

// --- FP64 in and out --------------------------------------------------------------

FL_HD long long fx_bits(double d) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(d);
#else
  long long b;
  __builtin_memcpy(&b, &d, 8);
  return b;
#endif
}
FL_HD double fx_from_bits(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}
// exponent field of a double (0: zero or subnormal, 2047: not finite)
FL_HD int fx_field(double d) { return (int)(fx_bits(d) >> 52) & 0x7ff; }

// d on a line whose largest exponent field is E, below 2^(62 - LR).  The
// value is f 2^X with X = fx_x0(E) + LR.
template <int LR> FL_HD long long fx_from(double d, int E) {
  const long long b = fx_bits(d);
  const int e = (int)(b >> 52) & 0x7ff;
  // fraction with its hidden bit at 2^62; subnormals have none and exponent 1
  const unsigned long long m = ((unsigned long long)b << 10 & 0x3ffffffffffffc00ull) | (e ? 1ull << 62 : 0ull);
  int s = (E > 1 ? E : 1) - (e ? e : 1) + 1 + LR;
  if (s > 63) s = 63;
  const long long f = (long long)(m >> s);
  return b < 0 ? -f : f;
}
FL_HD int fx_x0(int E) { return E == 0x7ff ? kFxBad : (E > 1 ? E : 1) - 1084; }

// f 2^X rounded to nearest (ties up in magnitude) where no result can leave
// the normal range, 2 - 1023 <= X <= 2046 - 1088
FL_HD bool fx_x_normal(int X) { return X >= -1021 && X <= 958; }
FL_HD double fx_to_normal(long long f, int X) {
  const unsigned long long a = f < 0 ? 0ull - (unsigned long long)f : (unsigned long long)f;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  const unsigned long long n = a << (lz & 63);
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1ull);   // 53 bits, the top one hidden
  const long long field = X + (63 - lz) + 1022;
  const long long b = (long long)(((unsigned long long)field << 52) + m);
  return a ? fx_from_bits(f < 0 ? (long long)((unsigned long long)b | (1ull << 63)) : b) : 0.0;
}

}  // namespace fl
