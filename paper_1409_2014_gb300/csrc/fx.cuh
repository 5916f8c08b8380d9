// fx.cuh -- the FP64 transforms in 64-bit block fixed point.
//
// GB300 issues FP64 instructions at 1/64 of its FP32 rate: one warp-wide FP64
// addition occupies an SM's FP64 pipe for 20 cycles (measured), a 64-bit
// integer addition the integer pipes for 0.76, and a 32 x 32 + 64 bit
// multiply-add for about one.  The FFTs of the FP64 plans, which are additions
// for the most part, therefore run on 64-bit integers: one complex
// multiplication by a table factor costs 16 cycles instead of 75, one addition
// 0.76 instead of 20, a radix-16 butterfly with its twiddles about 460 instead
// of 4200 cycles per warp.
//
// Block fixed point: the values of one transform share one exponent E, value =
// v 2^E.  Before each radix-16 stage the values are shifted left as far as the
// largest component allows (|component| < 2^61), and the stage's twiddle
// multiplication carries the factor 1/16: complex magnitudes enter a butterfly
// below 2^57.5 and leave it below 2^61.5, with no overflow in any partial sum
// (a partial sum of a DFT is a DFT of fewer terms).  The quantum is then at
// most 2^-56 of the block's largest component at every stage (the shift looks at
// the high words and recovers up to 29 bits at a time): a fixed 1/16 per stage
// would cost localised data, which do not grow in the first stages, four bits
// each (measured: 5 times the FP64 transforms' error).
//
// As in floating point, errors are relative to the norm of a transform's input,
// not to single elements; their constant grows with the ratio of a block's
// largest component to its root mean square, 3-5 for noise, up to sqrt(N) for a
// single wave.  Against the same passes in FP64 arithmetic (standard solver and
// linear flow, lengths 32-4096, noise, smooth densities, single waves), relative
// to max |m| ||rho||, the errors are 0.5-1.0 times as large and at most 1.1 times
// on the blocks with the largest ratio; where a multiplier damps the whole input
// (by 2^-8 and more) they can be three times as large relative to the small result.
//
// Multiplication: x = xh 2^32 + xl with both halves signed (xl in [-2^31,
// 2^31)), the constant as w 2^k = h + l 2^-32 in two signed 32-bit halves;
//   x w 2^(k-32) = xh h + 2^-32 (xh l + xl h) + 2^-64 xl l,
// the last term (at most 1/4 of the quantum) dropped, the middle one rounded.
#pragma once

#include "common.cuh"

namespace dsnu {

using i64 = long long;

struct alignas(16) fxc {  // fixed-point complex value
  i64 x, y;
};
struct alignas(16) fxw {  // constant w 2^k: re = rh + rl 2^-32, im = ih + il 2^-32 (|rl|, |il| < 2^31)
  int rh, rl, ih, il;
};
struct alignas(8) fxr {  // real constant in the same form
  int h, l;
};

// k of the tables: the twiddles carry 1/16, the multiplier and the deconvolution
// factors 1/2
constexpr int kFxTwBits = 28, kFxMultBits = 31, kFxDeconBits = 31;

// Exponents of all-zero transforms, and of ones with an infinity or a NaN.
constexpr int kFxZero = -(1 << 20), kFxBad = 1 << 20;
// The exponent of a multiplier's column whose entries are not all finite: added to
// those of any transform it gives one above kFxBad.
constexpr int kFxMultBad = 2 * kFxBad;

__device__ __forceinline__ fxc fx_mk(i64 x, i64 y) { fxc c; c.x = x; c.y = y; return c; }
__device__ __forceinline__ fxc operator+(fxc a, fxc b) { return fx_mk(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ fxc operator-(fxc a, fxc b) { return fx_mk(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ fxc fx_swap(fxc a) { return fx_mk(a.y, a.x); }

__device__ __forceinline__ i64 fx_mad(int a, int b, i64 c) {
  i64 d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ i64 fx_mulw(int a, int b) {
  i64 d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ void fx_split(i64 x, int& h, int& l) {
  l = int(x);
  h = int(x >> 32) + int(unsigned(l) >> 31);
}
__device__ __forceinline__ i64 fx_hi(i64 q) { return i64(int(q >> 32)); }
constexpr i64 kFxHalf = i64(1) << 31;

// x c 2^(k-32)
__device__ __forceinline__ i64 fx_mulr(i64 x, int h, int l) {
  int xh, xl;
  fx_split(x, xh, xl);
  return fx_mad(xh, h, fx_hi(fx_mad(xl, h, fx_mad(xh, l, kFxHalf))));
}
__device__ __forceinline__ i64 fx_mulr(i64 x, fxr c) { return fx_mulr(x, c.h, c.l); }
// a w 2^(k-32) and a conj(w) 2^(k-32)
__device__ __forceinline__ fxc fx_mul(fxc a, fxw w) {
  int xh, xl, yh, yl;
  fx_split(a.x, xh, xl);
  fx_split(a.y, yh, yl);
  const int nh = -w.ih, nl = -w.il;
  const i64 q = fx_mad(yl, nh, fx_mad(yh, nl, fx_mad(xl, w.rh, fx_mad(xh, w.rl, kFxHalf))));
  const i64 r = fx_mad(yl, w.rh, fx_mad(yh, w.rl, fx_mad(xl, w.ih, fx_mad(xh, w.il, kFxHalf))));
  return fx_mk(fx_mad(yh, nh, fx_mad(xh, w.rh, fx_hi(q))), fx_mad(yh, w.rh, fx_mad(xh, w.ih, fx_hi(r))));
}
__device__ __forceinline__ fxw fx_conj(fxw w) {
  w.ih = -w.ih;
  w.il = -w.il;
  return w;
}
// v 2^-s rounded (s > 0 a constant)
template <int S>
__device__ __forceinline__ i64 fx_shr(i64 v) { return (v + (i64(1) << (S - 1))) >> S; }
template <int S>
__device__ __forceinline__ fxc fx_shr(fxc a) { return fx_mk(fx_shr<S>(a.x), fx_shr<S>(a.y)); }
__device__ __forceinline__ fxc fx_shl(fxc a, int s) { return fx_mk(a.x << s, a.y << s); }
// v 2^s, rounded when s < 0 (s uniform over a group)
__device__ __forceinline__ fxc fx_scale2(fxc a, int s) {
  if (s >= 0) return fx_shl(a, s);
  const int r = min(-s, 63) - 1;
  return fx_mk(((a.x >> r) + 1) >> 1, ((a.y >> r) + 1) >> 1);
}

// a e^{-2 pi i m/16} / 2 (m = 1, 2, 3, 5, 6, 7): cos(pi/8), sin(pi/8) and
// sqrt(1/2) times 2^31 as h + l 2^-32
constexpr int kFxC1h = 1984016189, kFxC1l = -902489949;
constexpr int kFxS1h = 821806413, kFxS1l = 1565705635;
constexpr int kFxR2h = 1518500250, kFxR2l = -51432894;
template <int M16>
__device__ __forceinline__ fxc fx_rot16h(fxc a) {
  if constexpr (M16 == 2) {
    return fx_mk(fx_mulr(a.x + a.y, kFxR2h, kFxR2l), fx_mulr(a.y - a.x, kFxR2h, kFxR2l));
  } else if constexpr (M16 == 6) {
    return fx_mk(fx_mulr(a.y - a.x, kFxR2h, kFxR2l), fx_mulr(a.x + a.y, -kFxR2h, -kFxR2l));
  } else {
    constexpr int ch = (M16 == 1) ? kFxC1h : (M16 == 3) ? kFxS1h : (M16 == 5) ? -kFxS1h : -kFxC1h;
    constexpr int cl = (M16 == 1) ? kFxC1l : (M16 == 3) ? kFxS1l : (M16 == 5) ? -kFxS1l : -kFxC1l;
    constexpr int sh = (M16 == 1 || M16 == 7) ? kFxS1h : kFxC1h;
    constexpr int sl = (M16 == 1 || M16 == 7) ? kFxS1l : kFxC1l;
    fxw w;  // cos - i sin
    w.rh = ch;
    w.rl = cl;
    w.ih = -sh;
    w.il = -sl;
    return fx_mul(a, w);
  }
}

// In-place forward DFT of v[0..RAD) (natural order in and out), as dft_rec.
template <int RAD>
__device__ __forceinline__ void fx_dft(fxc (&v)[RAD]) {
  if constexpr (RAD == 2) {
    const fxc a = v[0], b = v[1];
    v[0] = a + b;
    v[1] = a - b;
  } else if constexpr (RAD > 2) {
    constexpr int H = RAD / 2, step = 16 / RAD;
    fxc e[H], o[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    fx_dft<H>(e);
    fx_dft<H>(o);
#define DSNU_FXTW(K)                                                             \
  if constexpr ((K) < H) {                                                       \
    constexpr int RK = ((K) * step) & 15;                                        \
    if constexpr (RK == 0) {                                                     \
      v[(K)] = e[(K)] + o[(K)];                                                  \
      v[(K) + H] = e[(K)] - o[(K)];                                              \
    } else if constexpr (RK == 4) {                                              \
      v[(K)] = fx_mk(e[(K)].x + o[(K)].y, e[(K)].y - o[(K)].x);                  \
      v[(K) + H] = fx_mk(e[(K)].x - o[(K)].y, e[(K)].y + o[(K)].x);              \
    } else {                                                                     \
      const fxc h = fx_rot16h<RK>(o[(K)]); /* half of the rotated value */       \
      v[(K)] = fx_mk(e[(K)].x + h.x + h.x, e[(K)].y + h.y + h.y);                \
      v[(K) + H] = fx_mk(e[(K)].x - h.x - h.x, e[(K)].y - h.y - h.y);            \
    }                                                                            \
  }
    DSNU_FXTW(0) DSNU_FXTW(1) DSNU_FXTW(2) DSNU_FXTW(3) DSNU_FXTW(4) DSNU_FXTW(5) DSNU_FXTW(6) DSNU_FXTW(7)
#undef DSNU_FXTW
  }
}

// ---------------------------------------------------------------------------
// Scaling.  fx_mag collects (by OR) the magnitudes' high words of a thread's
// values; after the OR over the transform's group, every |v| < 2^(64 - clz).
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned fx_mag(unsigned m, i64 v) {
  const int h = int(v >> 32);
  return m | unsigned(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned fx_mag(unsigned m, fxc a) { return fx_mag(fx_mag(m, a.x), a.y); }
template <int E>
__device__ __forceinline__ unsigned fx_mag(const fxc (&a)[E]) {
  // (three-operand minimum and maximum: one instruction per two values each,
  // against four; 2 % of a pass.  -1: no negative value)
  int hi = 0, lo = -1;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    hi = __vimax3_s32(hi, int(a[i].x >> 32), int(a[i].y >> 32));
    lo = __vimin3_s32(lo, int(a[i].x >> 32), int(a[i].y >> 32));
  }
  return unsigned(hi) | unsigned(~lo);
}

// Barrier of the P adjacent threads (a power of two) that work on one transform
// or pair of transforms: a named barrier, or the warp's (the CTAs of smaller
// groups have one warp).
template <int P>
__device__ __forceinline__ void fx_sync() {
  if constexpr (P > 32) asm volatile("bar.sync %0, %1;" ::"r"(1 + int(threadIdx.x) / P), "n"(P) : "memory");
  else __syncwarp();
}

// OR (or maximum) over P adjacent threads, in two halves around a barrier of
// theirs: fx_post gives the warp's part, fx_read collects the group's.  P <= 32:
// the group lies in one warp and fx_read needs no barrier.  `red`: one word per
// warp of the CTA.
template <int P, bool MAX = false>
__device__ __forceinline__ unsigned fx_post(unsigned m, unsigned* red) {
  if constexpr (P < 32) {
#pragma unroll
    for (int s = 1; s < P; s <<= 1) {
      const unsigned o = __shfl_xor_sync(0xffffffffu, m, s);
      m = MAX ? max(m, o) : (m | o);
    }
  } else {
    m = MAX ? __reduce_max_sync(0xffffffffu, m) : __reduce_or_sync(0xffffffffu, m);
    if (P > 32 && (threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  }
  return m;
}
template <int P, bool MAX = false>
__device__ __forceinline__ unsigned fx_read(unsigned m, const unsigned* red) {
  if constexpr (P > 32) {
    constexpr int W = P / 32;
    const unsigned* r = red + (threadIdx.x / P) * W;
    m = r[0];
#pragma unroll
    for (int i = 1; i < W; ++i) m = MAX ? max(m, r[i]) : (m | r[i]);
  }
  return m;
}
// Left shift that brings magnitudes OR-ed to m just below 2^T (0 where one is
// above: a component of a complex value whose magnitude is below 2^(T + 1/2)).
template <int T>
__device__ __forceinline__ int fx_norm_shift(unsigned m) { return max(__clz(int(m)) - (64 - T), 0); }

// Right shift that brings magnitudes OR-ed to m below 2^T.
template <int T>
__device__ __forceinline__ int fx_excess(unsigned m) { return max(64 - T - __clz(int(m)), 0); }

// ---------------------------------------------------------------------------
// Values per thread, the radix of the stages: 16, or 8 for the short transforms,
// whose passes do not fill the GPU: twice the threads, each with less than half
// the instructions in a row (FP64 solves with 8 against 16 values: 128^2 66 -> 49
// us, 512^2 92 -> 86, 1024 x 256 88 -> 76, 1024^2 equal, 2048^2 534 -> 639).
constexpr int kFxE8Max = 10;  // log2 of the longest transform with 8 values per thread
template <int LOG2N>
struct FxRad {
  static constexpr int LE = (LOG2N <= kFxE8Max) ? 3 : 4, E = 1 << LE;
  static constexpr int FULL = LOG2N / LE, LR = LOG2N - LE * FULL;  // radix-E stages, log2 of the last one's radix
  // stage twiddles (e^{-2 pi i r k/(NS RAD)}, r = 1 .. RAD - 1, k < NS, stage by stage)
  __host__ __device__ static constexpr int stw() {
    int n = 0;
    for (int s = 1; s < FULL; ++s) n += (E - 1) << (LE * s);
    return n + (LR > 0 ? ((1 << LR) - 1) << (LE * FULL) : 0);
  }
  static constexpr int STW = stw() > 0 ? stw() : 1;
};
inline int fx_log2_radix(int log2n) { return log2n <= kFxE8Max ? 3 : 4; }

// Length-N DFT by a group of G = N/E threads, E values per thread (the index
// order and buffer layout of block_fft_regs with E for 16).  P threads share one scale and
// one barrier: G, or 2 G where the lanes of two transforms interleave.  Groups
// with barriers of their own drift apart: while one multiplies (on the FMA pipe),
// another adds (on the ALU) -- in step, all warps of an SM wait for the same pipe
// (FP64 column pass at 4096^2 977 -> 912 us).  One transform per thread keeps it at 128 registers and one
// copy of the radix-16 code for all stages (the loop below): two transforms per
// thread at 8 warps per SM, the stages unrolled, came to 200 KB of code and ran
// twice as long (column pass at 4096^2 1405 us).
// Returns the exponent that the result gained.  red: 2 words per warp.
template <int LOG2N, int P>
__device__ __forceinline__ int fx_fft(fxc (&v)[FxRad<LOG2N>::E], fxc* buf, int t, const fxw* __restrict__ stw,
                                      unsigned* red) {
  using FR = FxRad<LOG2N>;
  constexpr int N = 1 << LOG2N, LE = FR::LE, E = FR::E, G = N / E, FULL = FR::FULL, LR = FR::LR;
  int ex = 0;
  // leave stage s (radix E, NS = E^s): exchange, and scale for the next one
  auto exchange = [&](int s) {
    const int ns = 1 << (LE * s), k = t & (ns - 1);
    const int base = (t - k) * E + k;
    unsigned* rd = red + (s & 1) * (blockDim.x >> 5);
    const unsigned m0 = fx_post<P>(fx_mag(v), rd);
    fx_sync<P>();  // every load of this buffer done (in place)
    if constexpr (E == 16) {  // (pad16 is linear over the stride)
      const int b0 = pad16(base), st = (s == 0) ? 1 : ns + (ns >> 4);
#pragma unroll
      for (int r = 0; r < E; ++r) buf[b0 + r * st] = v[r];
    } else {
#pragma unroll
      for (int r = 0; r < E; ++r) buf[pad16(base + r * ns)] = v[r];
    }
    fx_sync<P>();
    const int sh = fx_norm_shift<61>(fx_read<P>(m0, rd));
    ex += 4 - sh;
    return sh;
  };
#pragma unroll 1
  for (int s = 0;; ++s) {
    fx_dft<E>(v);
    if (s == FULL - 1) break;
    const int sh = exchange(s);
    const int ns = E << (LE * s);
    const fxw* tw = stw + (ns - E) + (t & (ns - 1));  // (E - 1)(E + .. + ns/E) = ns - E entries before
    v[0] = fx_shr<4>(fx_shl(buf[pad16(t)], sh));
#pragma unroll
    for (int r = 1; r < E; ++r) v[r] = fx_mul(fx_shl(buf[pad16(t + r * G)], sh), tw[(r - 1) * ns]);
  }
  if constexpr (LR > 0) {
    constexpr int RAD = 1 << LR, NS = 1 << (LE * FULL), PER = E / RAD, NB = N / RAD;
    const int sh = exchange(FULL - 1);
    fxc o[E];
#pragma unroll
    for (int b = 0; b < PER; ++b) {
      const int j = t + b * G;
      const fxw* tw = stw + (NS - E) + (j & (NS - 1));
      fxc u[RAD];
      u[0] = fx_shr<4>(fx_shl(buf[pad16(j)], sh));
#pragma unroll
      for (int r = 1; r < RAD; ++r) u[r] = fx_mul(fx_shl(buf[pad16(j + r * NB)], sh), tw[(r - 1) * NS]);
      fx_dft<RAD>(u);
#pragma unroll
      for (int r = 0; r < RAD; ++r) o[b + r * PER] = u[r];
    }
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = o[m];
  }
  return ex;
}
// The unnormalised inverse e^{+2 pi i nk/N}: real and imaginary parts
// exchanged before and after (register renaming).
template <int LOG2N, int P>
__device__ __forceinline__ int fx_ifft(fxc (&v)[FxRad<LOG2N>::E], fxc* buf, int t, const fxw* __restrict__ stw,
                                       unsigned* red) {
#pragma unroll
  for (int m = 0; m < FxRad<LOG2N>::E; ++m) v[m] = fx_swap(v[m]);
  const int ex = fx_fft<LOG2N, P>(v, buf, t, stw, red);
#pragma unroll
  for (int m = 0; m < FxRad<LOG2N>::E; ++m) v[m] = fx_swap(v[m]);
  return ex;
}

// FP64 -> fixed, |v| <= 2^62, relative to the exponent field efm >= 1 of the
// transform's largest component: d = v 2^(efm - kFxBias), rounded to nearest.
constexpr int kFxBias = 1084;
__device__ __forceinline__ i64 fx_from_f64(double d, int efm) {
  const int hi = __double2hiint(d);
  const int ef = (hi >> 20) & 0x7FF;
  const unsigned mh = (unsigned(hi) & 0xFFFFFu) | (ef ? 0x100000u : 0u);
  const i64 m = i64(((unsigned long long)mh << 32) | unsigned(__double2loint(d))) << 10;
  const int r = min(efm - max(ef, 1), 62);
  const i64 v = ((m >> r) + 1) >> 1;
  return hi < 0 ? -v : v;
}

// v 2^e as FP64 (round to nearest).  The conversion runs on the FP64 pipe,
// which is otherwise idle here; the exponent is added to its bit pattern.
static __device__ __noinline__ double fx_scale_slow(double d, int e) { return scalbn(d, e); }
__device__ __forceinline__ double fx_scale(double d, int e) {
  const int hi = __double2hiint(d);
  const int ne = ((hi >> 20) & 0x7FF) + e;
  const bool slow = unsigned(ne - 1) >= 0x7FEu || e != max(min(e, 4000), -4000);
  double r = __hiloint2double(int(unsigned(hi) + unsigned(e) * 0x100000u), __double2loint(d));
  if (d == 0.0) r = d;
  else if (slow) r = fx_scale_slow(d, e);
  return r;
}
__device__ __forceinline__ double fx_to_f64(i64 v, int e) { return fx_scale(__ll2double_rn(v), e); }

// ---------------------------------------------------------------------------
// Launch geometry of the passes with one transform per group (standard solver,
// linear flow): two groups per CTA for the long transforms (16 warps per SM),
// one warp's worth for the short ones (a small grid spreads over the SMs).
template <int LOG2N>
struct FxOne {
  static constexpr int N = 1 << LOG2N, E = FxRad<LOG2N>::E;
  static constexpr int G = N / E;
  static constexpr int PER = (G >= 64) ? 2 : (G >= 32) ? 1 : 32 / G;
  static constexpr int T = PER * G;
  static constexpr int MINB = (E == 16 ? 512 : 768) / T;
  static constexpr int FB = fft_buf_elems(N);
  static constexpr int STW = FxRad<LOG2N>::STW;
  static constexpr int W = T / 32, RED = 5 * W;
  static constexpr size_t smem = size_t(STW + PER * FB) * 16 + ((RED * 4 + 15) & ~15);
};

__device__ __forceinline__ fxr fx_ldr(const fxr* __restrict__ p) {
  const int2 v = __ldg(reinterpret_cast<const int2*>(p));
  fxr r;
  r.h = v.x;
  r.l = v.y;
  return r;
}
__device__ __forceinline__ fxw fx_ldw(const fxw* __restrict__ p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  fxw w;
  w.rh = v.x;
  w.rl = v.y;
  w.ih = v.z;
  w.il = v.w;
  return w;
}
__device__ __forceinline__ void fx_copy(fxw* __restrict__ dst, const fxw* __restrict__ src, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    *reinterpret_cast<int4*>(dst + i) = __ldg(reinterpret_cast<const int4*>(src + i));
}

// Collects into mx the largest high word of FP64 values (bit 0 set too for a
// subnormal below 2^-1042): its exponent field for fx_from_f64, 0 only when all
// are zero, >= 0x7FF00000 when one is infinite or a NaN.
__device__ __forceinline__ unsigned fx_top(unsigned mx, double d) {
  mx = max(mx, unsigned(__double2hiint(d)) & 0x7FFFFFFFu);
  return __double2loint(d) != 0 ? (mx | 1u) : mx;
}
constexpr unsigned kFxInf = 0x7FF00000u;
__device__ __forceinline__ int fx_efm(unsigned mx) { return max(int(mx >> 20), 1); }
// Exponent to store for a transform whose inputs had fx_top mx.
__device__ __forceinline__ int fx_exp(unsigned mx, int e) { return mx >= kFxInf ? kFxBad : mx == 0u ? kFxZero : e; }

// Maximum of n exponents over the CTA (every thread calls it; contains barriers).
__device__ __forceinline__ int fx_cta_max(const int* e, int n, unsigned* red) {
  int m = kFxZero;
  for (int i = threadIdx.x; i < n; i += blockDim.x) m = max(m, e[i]);
  m = __reduce_max_sync(0xffffffffu, m);
  __syncthreads();  // earlier reads of `red`
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = unsigned(m);
  __syncthreads();
  int r = int(red[0]);
  for (int w = 1; w < int(blockDim.x >> 5); ++w) r = max(r, int(red[w]));
  return r;
}

// a 2^-s rounded to nearest, s >= 1 (a shift alone rounds down: its mean error
// of half a quantum adds up over a transform to a spike at index 0).
__device__ __forceinline__ i64 fx_sra(i64 v, int s) { return ((v >> (s - 1)) + 1) >> 1; }
__device__ __forceinline__ fxc fx_sra(fxc a, int s) { return fx_mk(fx_sra(a.x, s), fx_sra(a.y, s)); }
// Right shift that aligns a value of exponent e to exponent emax + HEAD (values
// are stored below 2^63 and become smaller than 2^(63 - HEAD)).
template <int HEAD>
__device__ __forceinline__ int fx_align(int emax, int e) { return min(emax - e + HEAD, 63); }

// Alignment shifts, a byte each, packed by four.
template <int E>
__device__ __forceinline__ void fx_pack(unsigned (&pk)[(E + 3) / 4], int i, int s) {
  if ((i & 3) == 0) pk[i >> 2] = 0;
  pk[i >> 2] |= unsigned(s) << (8 * (i & 3));
}
template <int W>
__device__ __forceinline__ int fx_byte(const unsigned (&pk)[W], int i) {
  return int((pk[i >> 2] >> (8 * (i & 3))) & 0xFFu);
}

}  // namespace dsnu
