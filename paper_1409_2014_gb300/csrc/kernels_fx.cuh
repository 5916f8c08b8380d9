// kernels_fx.cuh -- the FFT passes of the FP64 plans, in 64-bit block fixed
// point (fx.cuh).
//
// The passes, their order and the row-tiled buffers A and B are those of
// kernels.cuh; here
//   * A and B hold fixed-point values.  The row pass scales each row by its
//     own exponent (rexp[iy]); the column passes align a column's rows to the
//     largest of them, scale the column to its own largest component, and write
//     it with its own exponent (cexp, bexp); the inverse row pass aligns the
//     columns and scales each row again.
//   * the deconvolution factor d_y of a row is a factor of the whole row, so
//     it multiplies the band columns (forward and inverse), not the rows;
//     z = rho + i rho d_x / 2^k, k per row so that both parts fill the format
//     (B's rows then have exponents of their own, rexpb).
//   * an infinity or a NaN in a row makes its exponent kFxBad, which travels
//     with the maxima: every result is then NaN.
//   * for real input the transposed pipeline (every complex constant
//     conjugated) computes the complex conjugate of each intermediate and the
//     same real result, so dsnu_solve_adjoint runs these same kernels.
// A pair of groups of G = N/E threads (E values per thread, 16 or 8) works on one
// row or column: group h = 0 runs the even, h = 1 the odd chain (even and odd frequencies, or output
// points).  Inputs are loaded, converted and aligned once, each thread taking
// E/2 of them, and handed to both chains through shared memory.  A CTA
// holds one pair, or as many as fill a warp, so that a small grid spreads over
// as many SMs as it has rows.
#pragma once

#include "fx.cuh"
#include "kernels.cuh"

namespace dsnu {

template <int LOG2N>
struct FxGeo {
  static constexpr int N = 1 << LOG2N, M = 2 * N, E = FxRad<LOG2N>::E;
  static constexpr int G = N / E, P = 2 * G;          // threads per chain, per pair
  static constexpr int PER = (P >= 32) ? 1 : 32 / P;  // pairs per CTA
  static constexpr int T = PER * P;
  static constexpr int MINB = (E == 16 ? 512 : 768) / T;  // 16 warps per SM, 24 with 8 values per thread
  static constexpr int FB = fft_buf_elems(N);
  static constexpr int STW = FxRad<LOG2N>::STW;
  static constexpr int W = T / 32, RED = 5 * W;       // words of the reductions: two for the FFT, three more
  static constexpr size_t smem = size_t(STW + PER * 2 * FB) * 16 + (((RED + 4 * PER) * 4 + 15) & ~15);
  // inverse rows: a byte of alignment shift per column of A, and one of B
  static constexpr size_t smem_row_inv(int Q) { return smem + ((N + 1 + 15) & ~15) + ((Q + 1 + 15) & ~15); }
};

// Plan tables of one axis.
struct FxAxis {
  const fxw* stw;    // stage twiddles e^{-2 pi i rk/(NS RAD)} 2^kFxTwBits
  const fxw* wm;     // e^{-2 pi i n/M} 2^kFxTwBits, n < N/2
  const fxr* dec;    // d / 2^kd 2^kFxDeconBits
};

struct FxOff {
  size_t A, B, Bband, Sband, rexp, rexpb, cexp, bexp;
};

struct FxMult {
  const fxr* m1;     // m1 2^-mexp[q] 2^kFxMultBits, row of ldm entries per column
  const int* mexp;   // NULL: 0
  int ldm;
};

// e^{-2 pi i n/M} at n = t + G m, m < E
template <int E>
__device__ __forceinline__ fxw fx_wm(const fxw* __restrict__ wm, int t, int m, int G) {
  fxw w = fx_ldw(wm + t + G * (m & (E / 2 - 1)));
  if (m >= E / 2) {  // e^{-2 pi i (n' + N/2)/M} = -i e^{-2 pi i n'/M}
    const fxw v = w;
    w.rh = v.ih;
    w.rl = v.il;
    w.ih = -v.rh;
    w.il = -v.rl;
  }
  return w;
}
// Threads that share a scale and barriers: the chain's G, or both chains' where they
// fit one warp (one reduction instruction; no warps to drift apart).
__host__ __device__ constexpr int fx_share(int G) { return 2 * G <= 32 ? 2 * G : G; }

// The chains' inputs from the staged values z (|component| < 2^61 after the
// shift s): z/16 for the even one, z e^{-2 pi i n/M}/16 for the odd one.
// (A barrier of the CTA: the chains' buffers are free for their exchanges after it.)
template <int G, int E>
__device__ __forceinline__ void fx_chain_in(fxc (&v)[E], const fxc* st, int s, int h, int t, const fxw* wm) {
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = st[pad16(t + G * m)];
  __syncthreads();
  if (h == 0) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = fx_shr<4>(fx_shl(v[m], s));
  } else {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = fx_mul(fx_shl(v[m], s), fx_wm<E>(wm, t, m, G));
  }
}
// The column sum e(n) + e^{+2 pi i n/M} o(n) of the two chains' results, each of
// exponent ex with its magnitudes m (fx_post over the chain, red), at
// n = t + G (m + h E/2), m < E/2: each chain hands the other half of its values
// over (in its own buffer) and multiplies half of the odd ones.  exs: two words of
// the pair.  Returns the sum's exponent (values below 2^59.5).
template <int G, int E>
__device__ __forceinline__ int fx_chain_out(fxc (&v)[E], fxc* buf_e, fxc* buf_o, unsigned mag, const unsigned* red,
                                            int ex, int* exs, int h, int t, const fxw* wm) {
  fx_sync<fx_share(G)>();  // (the chain's last loads of its buffer are done; `red` is complete)
  const int s = fx_norm_shift<62>(fx_read<fx_share(G)>(mag, red));
  if (t == 0) exs[h] = ex - s;
  if (h == 0) {
#pragma unroll
    for (int m = E / 2; m < E; ++m) buf_e[pad16(t + G * m)] = fx_shl(v[m], s);
  } else {
#pragma unroll
    for (int m = 0; m < E / 2; ++m) buf_o[pad16(t + G * m)] = fx_shl(v[m], s);
  }
  __syncthreads();
  // the chains' exponents differ by little: the smaller one's values are aligned
  const int xe = exs[0], xo = exs[1], x = max(xe, xo);
  const int de = min(x - xe, 59), dd = min(x - xo, 62);
#pragma unroll
  for (int m = 0; m < E / 2; ++m) {
    const fxc e = h ? buf_e[pad16(t + G * (m + E / 2))] : fx_shl(v[m], s);
    const fxc o = h ? fx_shl(v[m + E / 2], s) : buf_o[pad16(t + G * m)];
    const fxw w = h ? fx_wm<E>(wm, t, m + E / 2, G) : fx_wm<E>(wm, t, m, G);
    fxc p = fx_mul(o, fx_conj(w));
    if (dd > 0) p = fx_sra(p, dd);
    v[m] = fx_sra(e, 4 + de) + p;
  }
  return x + 4;
}

// Into L2 ahead of its use.
__device__ __forceinline__ void fx_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Common prologue of the passes: the CTA's tables, buffers and thread roles.
#define DSNU_FX_SETUP(AX)                                                  \
  using GG = FxGeo<LOG2N>;                                                 \
  using TL = Tile<double>;                                                 \
  constexpr int N = GG::N, E = GG::E, H = E / 2, G = GG::G, P = GG::P;     \
  constexpr int PER = GG::PER, W = GG::W;                                  \
  extern __shared__ __align__(16) unsigned char smem_raw[];                \
  fxw* stw = reinterpret_cast<fxw*>(smem_raw);                             \
  fxc* sm = reinterpret_cast<fxc*>(stw + GG::STW);                         \
  unsigned* red = reinterpret_cast<unsigned*>(sm + PER * 2 * GG::FB);      \
  fx_copy(stw, (AX).stw, FxRad<LOG2N>::stw());                             \
  const int pr = threadIdx.x / P, tp = threadIdx.x - pr * P;               \
  const int h = tp / G, t = tp - h * G;                                    \
  fxc* buf_e = sm + (2 * pr) * GG::FB;                                     \
  fxc* buf_o = buf_e + GG::FB;                                             \
  fxc* buf = h ? buf_o : buf_e;                                            \
  int* exs = reinterpret_cast<int*>(red + GG::RED) + 2 * pr;               \
  (void)exs;                                                               \
  __syncthreads();                                                         \
  grid_dep_wait();

// ---------------------------------------------------------------------------
// Forward row pass (k_row_fwd in fixed point).
template <int LOG2N>
__global__ void __launch_bounds__(FxGeo<LOG2N>::T, FxGeo<LOG2N>::MINB)
k_fx_row_fwd(Members mem, FxOff off, int ldqA, int ldqB, int Q, int ny, FxAxis ax, int kd) {
  DSNU_FX_SETUP(ax)
  const int items = (ny + PER - 1) / PER;
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, row = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    const bool valid = row < ny;
    double x[H];
    fxr d[H];
    unsigned mx = 0, md = 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      x[i] = valid ? __ldg(mb.rho + size_t(row) * N + tp + P * i) : 0.0;
      d[i] = fx_ldr(ax.dec + tp + P * i);
      mx = fx_top(mx, x[i]);
      md = max(md, ((unsigned(__double2hiint(x[i])) >> 20) & 0x7FFu) + 32u - unsigned(__clz(d[i].h)));
    }
    mx = fx_post<P, true>(mx, red + 2 * W);
    md = fx_post<P, true>(md, red + 3 * W);
    __syncthreads();
    mx = fx_read<P, true>(mx, red + 2 * W);
    md = fx_read<P, true>(md, red + 3 * W);
    const int efm = fx_efm(mx);
    // the smallest k with |rho d_x| <= 2^k max |rho| by the exponents (|rho| <
    // 2^(ef + 1), d_x/2^kd < 2^(1 - clz h)): z = rho + i rho d_x/2^k
    const int kr = min(max(int(md) - 32 + kd + 1 - efm, 0), kd);
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const i64 v = fx_from_f64(x[i], efm);
      buf_e[pad16(tp + P * i)] = fx_mk(fx_shr<1>(v), fx_mulr(v, d[i]) << (kd - kr));  // <= 2^61
    }
    __syncthreads();
    fxc v[E];
    // the next row into L2 while this one is transformed
    if (row + int(gridDim.x) * PER < ny && (tp & 15) == 0)
#pragma unroll
      for (int i = 0; i < H; ++i) fx_prefetch(mb.rho + size_t(row + int(gridDim.x) * PER) * N + tp + P * i);
    fx_chain_in<G, E>(v, buf_e, 0, h, t, ax.wm);
    // exponent of the chain: from_f64 (efm - kFxBias), the five bits, the stages
    const int xh = efm - kFxBias + 5 + fx_fft<LOG2N, fx_share(G)>(v, buf, t, stw, red);
    const unsigned mag = fx_post<fx_share(G)>(fx_mag(v), red + 4 * W);
    fx_sync<fx_share(G)>();  // (and the last stage's loads are done)
    if (t == 0) {
      exs[h] = xh - fx_norm_shift<62>(fx_read<fx_share(G)>(mag, red + 4 * W));  // sums of two: below 2^63
      exs[2 * PER + h] = xh;
    }
#pragma unroll
    for (int m = 0; m < E; ++m) buf[pad16(t + G * m)] = v[m];
    __syncthreads();
    // A = (Z(q) + conj Z(M - q))/2 and B = (Z(q) - conj Z(M - q))/2i as sums, both
    // chains brought to one exponent
    const int xc = max(exs[0], exs[1]), s1 = exs[2 * PER + (tp & 1)] - xc;
    if (tp == 0 && valid) {
      const int ea = xc - 1;
      ws_ptr<int>(mb, off.rexp)[row] = fx_exp(mx, ea);
      ws_ptr<int>(mb, off.rexpb)[row] = fx_exp(mx, ea + kr);
    }
    if (valid) {
      fxc* Ar = ws_ptr<fxc>(mb, off.A) + TL::at(row, 0, ldqA);
      fxc* Br = ws_ptr<fxc>(mb, off.B) + TL::at(row, 0, ldqB);
#pragma unroll
      for (int i = 0; i < H + 1; ++i) {
        const int q = tp + P * i;
        if (i == H && q > N) break;
        const int k = q >> 1;
        const fxc zq = (q & 1) ? buf_o[pad16(k)] : buf_e[pad16(k & (N - 1))];
        const fxc zm = (q & 1) ? buf_o[pad16(N - 1 - k)] : buf_e[pad16((N - k) & (N - 1))];
        Ar[q * TL::TR] = fx_scale2(fx_mk(zq.x + zm.x, zq.y - zm.y), s1);
        if (q <= Q) Br[q * TL::TR] = fx_scale2(fx_mk(zq.y + zm.y, zm.x - zq.x), s1);
      }
    }
  }
}

// Alignment shifts of the rows tp + P i that a thread stages.  Returns the rows'
// largest exponent.
template <int P, int H>
__device__ __forceinline__ int fx_row_shifts(const int* rexp, int ny, int tp, unsigned* red,
                                             unsigned (&pk)[(H + 3) / 4]) {
  const int emax = fx_cta_max(rexp, ny, red);
#pragma unroll
  for (int i = 0; i < H; ++i) fx_pack<H>(pk, i, fx_align<2>(emax, rexp[tp + P * i]));
  return emax;
}

// ---------------------------------------------------------------------------
// Column pass of I1 (k_col_main in fixed point).  FULL: the multiplier row has
// an entry for each of the M natural frequencies (multipliers with a sin 2theta
// term), else for a = |qbar| <= N only; both parity-split.
template <int LOG2N, bool FULL>
__global__ void __launch_bounds__(FxGeo<LOG2N>::T, FxGeo<LOG2N>::MINB)
k_fx_col_main(Members mem, FxOff off, int ldqA, int ncols, FxAxis ay, FxMult mt) {
  DSNU_FX_SETUP(ay)
  constexpr int MH = FULL ? N : N / 2 + 1;  // even entries
  const int items = (ncols + PER - 1) / PER;
  int cur = -1, emax = 0;
  unsigned pk[(H + 3) / 4] = {};
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, col = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    if (mi != cur) {
      emax = fx_row_shifts<P, H>(ws_ptr<int>(mb, off.rexp), N, tp, red + 4 * W, pk);
      cur = mi;
    }
    fxc* __restrict__ A = ws_ptr<fxc>(mb, off.A);
    const bool valid = col < ncols;
    fxc v[E];
    unsigned mag = 0;
#pragma unroll
    for (int i = 0; i < H; ++i) v[i] = valid ? A[TL::at(tp + P * i, col, ldqA)] : fx_mk(0, 0);
#pragma unroll
    for (int i = 0; i < H; ++i) {
      v[i] = fx_sra(v[i], fx_byte(pk, i));
      mag = fx_mag(mag, v[i]);
    }
    mag = fx_post<P>(mag, red + 2 * W);
    __syncthreads();  // (and the previous item's reads of the buffers are done)
#pragma unroll
    for (int i = 0; i < H; ++i) buf_e[pad16(tp + P * i)] = v[i];
    __syncthreads();
    const int s0 = fx_norm_shift<61>(fx_read<P>(mag, red + 2 * W));
    // the next column and its multipliers into L2 while this one is transformed
    if (col + int(gridDim.x) * PER < ncols) {
      const int nc = col + int(gridDim.x) * PER;
      if ((tp & 1) == 0)
#pragma unroll
        for (int i = 0; i < H; ++i) fx_prefetch(A + TL::at(tp + P * i, nc, ldqA));
      for (int i = tp * 16; i < mt.ldm; i += P * 16) fx_prefetch(mt.m1 + size_t(nc) * mt.ldm + i);
    }
    fx_chain_in<G, E>(v, buf_e, s0, h, t, ay.wm);
    // the chain's exponent: the rows', s0, /16, stages, multiplier (its own and /2), d, stages
    int ex = emax + 2 - s0 + 4;
    ex += fx_fft<LOG2N, fx_share(G)>(v, buf, t, stw, red) + (mt.mexp && valid ? mt.mexp[col] : 0) + 1;
    const fxr* mg = mt.m1 + size_t(valid ? col : 0) * mt.ldm + (h ? MH : 0);
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int k = t + G * m;  // row q = 2 k + h: |qbar| / 2 rounded down
      const fxr c = fx_ldr(mg + (FULL ? k : (m < H ? k : N - h - k)));
      v[m] = fx_mk(fx_mulr(v[m].x, c), fx_mulr(v[m].y, c));
    }
    // room for the inverse's first stage by the products' own size, however small
    // they are against the multiplier's bound: a fixed 1/32 there cost a column
    // whose spectrum sits where the multiplier is small up to three bits against
    // FP64 arithmetic (half Laplacian of a smooth density, length 4096: 5.1 eps of
    // max |m| ||rho||, FP64 0.84, this 0.86).  The products themselves are rounded
    // at 2^-61 of the values' largest times the column's bound of |m|.
    mag = fx_post<fx_share(G)>(fx_mag(v), red + 2 * W);
    fx_sync<fx_share(G)>();
    const int d = fx_excess<57>(fx_read<fx_share(G)>(mag, red + 2 * W));
    ex += d;
    if constexpr (E == 16) {  // (d is 0 for tiny products only; without the branch 4096^2 2022 us, with it 2031)
      const i64 half = (i64(1) << d) >> 1;
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = fx_mk((v[m].x + half) >> d, (v[m].y + half) >> d);
    } else if (d > 0) {  // (512^2 73.4 us, without the branch 74.1)
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = fx_sra(v[m], d);
    }
    ex += fx_ifft<LOG2N, fx_share(G)>(v, buf, t, stw, red);
    mag = fx_post<fx_share(G)>(fx_mag(v), red + 3 * W);
    ex = fx_chain_out<G, E>(v, buf_e, buf_o, mag, red + 3 * W, ex, exs, h, t, ay.wm);
    if (valid) {
#pragma unroll
      for (int m = 0; m < H; ++m) A[TL::at(t + G * (m + H * h), col, ldqA)] = fx_shl(v[m], 3);  // < 2^59.5 before
      if (tp == 0) ws_ptr<int>(mb, off.cexp)[col] = (emax >= kFxBad) ? kFxBad : (emax <= kFxZero) ? kFxZero : ex - 3;
    }
  }
}

// ---------------------------------------------------------------------------
// Band columns of the type-2 spectrum (k_band_fwd in fixed point), written in
// FP64; kdy: the deconvolution factors' scale.
template <int LOG2N>
__global__ void __launch_bounds__(FxGeo<LOG2N>::T, FxGeo<LOG2N>::MINB)
k_fx_band_fwd(Members mem, FxOff off, int ldqB, int ncols, int ldq, int Q, FxAxis ay, int kdy) {
  DSNU_FX_SETUP(ay)
  constexpr int M = GG::M;
  const int items = (ncols + PER - 1) / PER;
  int cur = -1, emax = 0;
  unsigned pk[(H + 3) / 4] = {};
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, col = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    if (mi != cur) {
      emax = fx_row_shifts<P, H>(ws_ptr<int>(mb, off.rexpb), N, tp, red + 4 * W, pk);
      cur = mi;
    }
    const fxc* __restrict__ B = ws_ptr<fxc>(mb, off.B);
    double2* __restrict__ Bband = ws_ptr<double2>(mb, off.Bband);
    const bool valid = col < ncols;
    fxc v[E];
    unsigned mag = 0;
#pragma unroll
    for (int i = 0; i < H; ++i) v[i] = valid ? B[TL::at(tp + P * i, col, ldqB)] : fx_mk(0, 0);
#pragma unroll
    for (int i = 0; i < H; ++i) {
      v[i] = fx_sra(v[i], fx_byte(pk, i));
      mag = fx_mag(mag, v[i]);
    }
    mag = fx_post<P>(mag, red + 2 * W);
    __syncthreads();
    const int s0 = fx_norm_shift<61>(fx_read<P>(mag, red + 2 * W));
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const fxr d = fx_ldr(ay.dec + tp + P * i);  // d_y/2^kdy, and /2
      const fxc x = fx_shl(v[i], s0);
      buf_e[pad16(tp + P * i)] = fx_mk(fx_mulr(x.x, d), fx_mulr(x.y, d));
    }
    __syncthreads();
    fx_chain_in<G, E>(v, buf_e, 1, h, t, ay.wm);
    const int ex = emax + 2 - s0 + kdy + 4 + fx_fft<LOG2N, fx_share(G)>(v, buf, t, stw, red);
    if (valid) {
      const bool bad = emax >= kFxBad;
      const double nan = __longlong_as_double(0x7FF8000000000000ll);
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int q = 2 * (t + G * m) + h, sq = q < N ? q : q - M;
        if (sq >= -Q && sq <= Q)
          Bband[size_t(col) * ldq + sq + Q] =
              bad ? make_double2(nan, nan) : make_double2(fx_to_f64(v[m].x, ex), fx_to_f64(v[m].y, ex));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Inverse band columns (k_band_inv in fixed point) of the FP64 S, times d_y.
template <int LOG2N>
__global__ void __launch_bounds__(FxGeo<LOG2N>::T, FxGeo<LOG2N>::MINB)
k_fx_band_inv(Members mem, FxOff off, int ldq, int Q, int ncols, int ldqB, FxAxis ay, int kdy) {
  DSNU_FX_SETUP(ay)
  constexpr int M = GG::M;
  const int items = (ncols + PER - 1) / PER;
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, col = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    const double2* __restrict__ Sband = ws_ptr<double2>(mb, off.Sband);
    fxc* __restrict__ St = ws_ptr<fxc>(mb, off.B);
    const bool valid = col < ncols;
    fxc v[E];
    unsigned mx = 0;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int q = 2 * (t + G * m) + h, sq = q < N ? q : q - M;
      double2 a = make_double2(0.0, 0.0);
      if (valid && sq >= -Q && sq <= Q) a = Sband[size_t(col) * ldq + sq + Q];
      mx = fx_top(fx_top(mx, a.x), a.y);
      v[m] = fx_mk(__double_as_longlong(a.x), __double_as_longlong(a.y));
    }
    mx = fx_post<P, true>(mx, red + 2 * W);
    __syncthreads();
    mx = fx_read<P, true>(mx, red + 2 * W);
    const int efm = fx_efm(mx);
#pragma unroll
    for (int m = 0; m < E; ++m)
      v[m] = fx_shr<5>(fx_mk(fx_from_f64(__longlong_as_double(v[m].x), efm), fx_from_f64(__longlong_as_double(v[m].y), efm)));
    int ex = efm - kFxBias + 5 + fx_ifft<LOG2N, fx_share(G)>(v, buf, t, stw, red);
    const unsigned mag = fx_post<fx_share(G)>(fx_mag(v), red + 3 * W);
    ex = fx_chain_out<G, E>(v, buf_e, buf_o, mag, red + 3 * W, ex, exs, h, t, ay.wm);
    if (valid) {
#pragma unroll
      for (int m = 0; m < H; ++m) {
        const int n = t + G * (m + H * h);
        const fxr d = fx_ldr(ay.dec + n);
        St[TL::at(n, col, ldqB)] = fx_shl(fx_mk(fx_mulr(v[m].x, d), fx_mulr(v[m].y, d)), 4);  // < 2^58.5 before
      }
      if (tp == 0)
        ws_ptr<int>(mb, off.bexp)[col] = fx_exp(mx, ex + kdy + 1 - 4);
    }
  }
}

// ---------------------------------------------------------------------------
// Inverse row pass (k_row_inv in fixed point): with X = Y + i S and R = Y - i S,
//   T(2j) = IDFT_N[X(q) + conj R(N - q)](j),
//   T(2j+1) = IDFT_N[(X(q) - conj R(N - q)) e^{+2 pi i q/M}](j)
// (at q = 0 the second term is X(N)); Phi = (Re T + d_x Im T) 2^lscale.
template <int LOG2N>
__global__ void __launch_bounds__(FxGeo<LOG2N>::T, FxGeo<LOG2N>::MINB)
k_fx_row_inv(Members mem, FxOff off, int ldqA, int ldqB, int Q, int ny, FxAxis ax, int kd, int lscale) {
  DSNU_FX_SETUP(ax)
  unsigned char* sh_a = smem_raw + GG::smem;            // alignment shifts of the columns of A
  unsigned char* sh_b = sh_a + ((N + 1 + 15) & ~15);    // and of B
  const int items = (ny + PER - 1) / PER;
  int cur = -1, emax = 0;
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, row = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    if (mi != cur) {
      const int* ce = ws_ptr<int>(mb, off.cexp);
      const int* be = ws_ptr<int>(mb, off.bexp);
      emax = max(fx_cta_max(ce, N + 1, red + 4 * W), fx_cta_max(be, Q + 1, red + 4 * W));
      for (int q = threadIdx.x; q <= N; q += GG::T) sh_a[q] = (unsigned char)fx_align<4>(emax, ce[q]);
      for (int q = threadIdx.x; q <= Q; q += GG::T) sh_b[q] = (unsigned char)fx_align<4>(emax, be[q]);
      cur = mi;
      __syncthreads();
    }
    const bool valid = row < ny;
    const fxc* __restrict__ Ar = ws_ptr<fxc>(mb, off.A) + TL::at(valid ? row : 0, 0, ldqA);
    const fxc* __restrict__ Br = ws_ptr<fxc>(mb, off.B) + TL::at(valid ? row : 0, 0, ldqB);
    const fxc z = fx_mk(0, 0);
    fxc v[E];  // X in the first, R in the second half
    unsigned mag = 0;
    fxc yn = z;
#pragma unroll
    for (int i = 0; i < H; ++i) v[i] = valid ? Ar[(tp + P * i) * TL::TR] : z;
    if (valid && tp == 0) yn = Ar[N * TL::TR];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const int q = tp + P * i;
      const fxc y = fx_sra(v[i], sh_a[q]);
      const fxc s = (valid && q <= Q) ? fx_sra(Br[q * TL::TR], sh_b[q]) : z;
      v[i] = fx_mk(y.x - s.y, y.y + s.x);
      v[i + H] = fx_mk(y.x + s.y, y.y - s.x);
    }
    mag = fx_mag(v);
    if (tp == 0) {  // conj X(N) (Q < N: no band value) in the place of conj R(N - 0)
      yn = fx_sra(yn, sh_a[N]);
      yn.y = -yn.y;
      mag = fx_mag(mag, yn);
    }
    mag = fx_post<P>(mag, red + 2 * W);
    __syncthreads();  // (and the previous item's reads of the buffers are done)
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const int q = tp + P * i;
      buf_e[pad16(q)] = v[i];
      if (q != 0) buf_o[pad16(N - q)] = v[i + H];  // R(N - q) at q
    }
    if (tp == 0) buf_o[0] = yn;
    __syncthreads();
    const int s0 = fx_norm_shift<60>(fx_read<P>(mag, red + 2 * W));
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const fxc x = buf_e[pad16(t + G * m)], r = buf_o[pad16(t + G * m)];
      v[m] = h ? fx_mk(x.x - r.x, x.y + r.y) : fx_mk(x.x + r.x, x.y - r.y);
    }
    __syncthreads();  // the buffers are free for the chains' exchanges
    if (h == 0) {
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = fx_shr<4>(fx_shl(v[m], s0));
    } else {
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = fx_mul(fx_shl(v[m], s0), fx_conj(fx_wm<E>(ax.wm, t, m, G)));
    }
    const int ex = emax + 4 - s0 + 4 + kd + 1 + lscale + fx_ifft<LOG2N, fx_share(G)>(v, buf, t, stw, red);
    if (valid) {
      double* __restrict__ phi = mb.phi + size_t(row) * N + h;
      const bool bad = emax >= kFxBad;
      const i64 half = i64(1) << kd;
#pragma unroll
      for (int m = 0; m < H; ++m) {
        const int n = 2 * (t + G * m);
        // Re T 2^-(kd + 1) + Im T d_x/2^kd /2
        const i64 f = ((v[m].x + half) >> (kd + 1)) + fx_mulr(v[m].y, fx_ldr(ax.dec + n + h));
        phi[n] = bad ? __longlong_as_double(0x7FF8000000000000ll) : fx_to_f64(f, ex);
      }
    }
  }
}

#undef DSNU_FX_SETUP

}  // namespace dsnu
