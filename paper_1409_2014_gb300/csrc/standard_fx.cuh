// standard_fx.cuh -- the standard periodic FFT solver (standard.cuh) of the FP64
// plans in 64-bit block fixed point (fx.cuh): the same three passes and
// row-tiled half spectrum, each row pair and each column with its own exponent
// (as in kernels_fx.cuh), the multiplier from a plan table.  The operator is
// symmetric and its conjugated pipeline gives the same real result, so the
// adjoint runs these kernels too.
#pragma once

#include "kernels_fx.cuh"

namespace dsnu {

// Common prologue: the CTA's tables and buffers; groups of G threads, each with
// a scale of its own.
#define DSNU_FX_SETUP1(STWG)                                               \
  using GG = FxOne<LOG2N>;                                                 \
  using TL = Tile<double>;                                                 \
  constexpr int N = GG::N, E = GG::E, H = E / 2, G = GG::G, P = G;         \
  constexpr int PER = GG::PER, W = GG::W;                                  \
  extern __shared__ __align__(16) unsigned char smem_raw[];                \
  fxw* stw = reinterpret_cast<fxw*>(smem_raw);                             \
  fxc* sm = reinterpret_cast<fxc*>(stw + GG::STW);                         \
  unsigned* red = reinterpret_cast<unsigned*>(sm + PER * GG::FB);          \
  fx_copy(stw, STWG, FxRad<LOG2N>::stw());                                 \
  const int pr = threadIdx.x / G, t = threadIdx.x - pr * G;                \
  fxc* buf = sm + pr * GG::FB;                                             \
  __syncthreads();                                                         \
  grid_dep_wait();

template <int LOG2N>
__global__ void __launch_bounds__(FxOne<LOG2N>::T, FxOne<LOG2N>::MINB)
k_fx_std_row_fwd(Members mem, size_t offH, size_t offE, int ldq, int ny, const fxw* __restrict__ stw_g) {
  DSNU_FX_SETUP1(stw_g)
  const int pairs = ny / 2, items = (pairs + PER - 1) / PER;
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, pi = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    const bool valid = pi < pairs;
    const double* ra = mb.rho + size_t(valid ? 2 * pi : 0) * N;
    fxc v[E];
    unsigned mx = 0;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const double a = valid ? __ldg(ra + t + G * m) : 0.0, b = valid ? __ldg(ra + N + t + G * m) : 0.0;
      mx = fx_top(fx_top(mx, a), b);
      v[m] = fx_mk(__double_as_longlong(a), __double_as_longlong(b));
    }
    mx = fx_post<P, true>(mx, red + 2 * W);
    __syncthreads();
    mx = fx_read<P, true>(mx, red + 2 * W);
    const int efm = fx_efm(mx);
#pragma unroll
    for (int m = 0; m < E; ++m)
      v[m] = fx_shr<5>(fx_mk(fx_from_f64(__longlong_as_double(v[m].x), efm), fx_from_f64(__longlong_as_double(v[m].y), efm)));
    const int ef = fx_fft<LOG2N, P>(v, buf, t, stw, red);
    const unsigned mag = fx_post<P>(fx_mag(v), red + 3 * W);
    __syncthreads();
    const int s1 = fx_norm_shift<62>(fx_read<P>(mag, red + 3 * W));  // sums of two: below 2^63
#pragma unroll
    for (int m = 0; m < E; ++m) buf[pad16(t + G * m)] = v[m];
    __syncthreads();
    if (valid) {
      fxc* hs = ws_ptr<fxc>(mb, offH) + TL::at(2 * pi, 0, ldq);
#pragma unroll
      for (int i = 0; i < H + 1; ++i) {
        const int q = t + G * i;
        if (i == H && q > N / 2) break;
        const fxc zq = buf[pad16(q)], zm = buf[pad16((N - q) & (N - 1))];
        // X_a = (Z(q) + conj Z(N - q)) / 2,  X_b = (Z(q) - conj Z(N - q)) / (2i), as sums
        hs[q * TL::TR] = fx_shl(fx_mk(zq.x + zm.x, zq.y - zm.y), s1);
        hs[q * TL::TR + 1] = fx_shl(fx_mk(zq.y + zm.y, zm.x - zq.x), s1);
      }
      if (t == 0) ws_ptr<int>(mb, offE)[pi] = fx_exp(mx, efm - kFxBias + 5 + ef - 1 - s1);
    }
  }
}

// FULL: a multiplier row has an entry for each of the N frequencies, else for
// |qbar| <= N/2 only.
template <int LOG2N, bool FULL>
__global__ void __launch_bounds__(FxOne<LOG2N>::T, FxOne<LOG2N>::MINB)
k_fx_std_col(Members mem, size_t offH, size_t offE, size_t offC, int ldq, int ncols, const fxw* __restrict__ stw_g,
             FxMult mt) {
  DSNU_FX_SETUP1(stw_g)
  const int items = (ncols + PER - 1) / PER;
  int cur = -1, emax = 0;
  unsigned pk[(E + 3) / 4] = {};  // alignment shifts of the rows t + G m
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, col = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    if (mi != cur) {
      const int* re = ws_ptr<int>(mb, offE);
      emax = fx_cta_max(re, N / 2, red + 4 * W);
#pragma unroll
      for (int m = 0; m < E; ++m) fx_pack<E>(pk, m, fx_align<2>(emax, re[(t + G * m) >> 1]));
      cur = mi;
    }
    fxc* __restrict__ hs = ws_ptr<fxc>(mb, offH);
    const bool valid = col < ncols;
    fxc v[E];
    unsigned mag = 0;
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = valid ? hs[TL::at(t + G * m, col, ldq)] : fx_mk(0, 0);
#pragma unroll
    for (int m = 0; m < E; ++m) {
      v[m] = fx_sra(v[m], fx_byte(pk, m));
      mag = fx_mag(mag, v[m]);
    }
    mag = fx_post<P>(mag, red + 2 * W);
    __syncthreads();
    const int s0 = fx_norm_shift<61>(fx_read<P>(mag, red + 2 * W));
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = fx_shr<4>(fx_shl(v[m], s0));
    int ex = emax + 2 - s0 + 4 + (mt.mexp && valid ? mt.mexp[col] : 0) + 1;
#pragma unroll 1
    for (int inv = 0;; ++inv) {  // forward, then inverse (one copy of the transform's code)
      ex += fx_fft<LOG2N, P>(v, buf, t, stw, red);
      if (inv) {
        mag = fx_post<P>(fx_mag(v), red + 3 * W);
        __syncthreads();
        const int s = fx_norm_shift<62>(fx_read<P>(mag, red + 3 * W));
        ex -= s;
        if (valid) {
#pragma unroll
          for (int m = 0; m < E; ++m) hs[TL::at(t + G * m, col, ldq)] = fx_shl(fx_swap(v[m]), s);
          if (t == 0) ws_ptr<int>(mb, offC)[col] = (emax >= kFxBad) ? kFxBad : (emax <= kFxZero) ? kFxZero : ex;
        }
        break;
      }
      const fxr* mg = mt.m1 + size_t(valid ? col : 0) * mt.ldm;
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int q = t + G * m;
        const fxr c = fx_ldr(mg + (FULL || m < H ? q : N - q));
        v[m] = fx_mk(fx_mulr(v[m].y, c), fx_mulr(v[m].x, c));  // (components exchanged: the inverse transform)
      }
      // room for the inverse's first stage (as in k_fx_col_main)
      mag = fx_post<P>(fx_mag(v), red + 2 * W);
      __syncthreads();
      const int d = fx_excess<57>(fx_read<P>(mag, red + 2 * W));
      ex += d;
      if (d > 0)
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = fx_sra(v[m], d);
    }
  }
}

template <int LOG2N>
__global__ void __launch_bounds__(FxOne<LOG2N>::T, FxOne<LOG2N>::MINB)
k_fx_std_row_inv(Members mem, size_t offH, size_t offC, int ldq, int ny, const fxw* __restrict__ stw_g, int lscale) {
  DSNU_FX_SETUP1(stw_g)
  const int pairs = ny / 2, items = (pairs + PER - 1) / PER;
  int cur = -1, emax = 0;
  unsigned pk[(E + 3) / 4] = {};  // alignment shifts of the columns |qbar| of q = t + G m
#pragma unroll 1
  for (int it = blockIdx.x; it < items * mem.count; it += gridDim.x) {
    if (it + int(gridDim.x) >= items * mem.count) grid_dep_trigger();  // last item of this CTA
    const int mi = it / items, pi = (it - mi * items) * PER + pr;
    const Member mb = member_at(mem, mi);
    if (mi != cur) {
      const int* ce = ws_ptr<int>(mb, offC);
      emax = fx_cta_max(ce, N / 2 + 1, red + 4 * W);
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int q = t + G * m;
        fx_pack<E>(pk, m, fx_align<3>(emax, ce[q > N / 2 ? N - q : q]));
      }
      cur = mi;
    }
    const bool valid = pi < pairs;
    const fxc* __restrict__ hs = ws_ptr<fxc>(mb, offH) + TL::at(valid ? 2 * pi : 0, 0, ldq);
    fxc v[E];
    unsigned mag = 0;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int q = t + G * m, qq = q > N / 2 ? N - q : q;
      const int s = fx_byte(pk, m);
      fxc ya = fx_mk(0, 0), yb = ya;
      if (valid) {
        ya = fx_sra(hs[qq * TL::TR], s);
        yb = fx_sra(hs[qq * TL::TR + 1], s);
      }
      if (q > N / 2) {
        ya.y = -ya.y;
        yb.y = -yb.y;
      }
      v[m] = fx_mk(ya.x - yb.y, ya.y + yb.x);  // Y_a + i Y_b, below 2^61
      mag = fx_mag(mag, v[m]);
    }
    mag = fx_post<P>(mag, red + 2 * W);
    __syncthreads();
    const int s0 = fx_norm_shift<61>(fx_read<P>(mag, red + 2 * W));
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = fx_shr<4>(fx_shl(v[m], s0));
    const int ex = emax + 3 - s0 + 4 + lscale + fx_ifft<LOG2N, P>(v, buf, t, stw, red);
    if (valid) {
      const bool bad = emax >= kFxBad;
      const double nan = __longlong_as_double(0x7FF8000000000000ll);
      double* phi = mb.phi + size_t(2 * pi) * N;
#pragma unroll
      for (int m = 0; m < E; ++m) {
        phi[t + G * m] = bad ? nan : fx_to_f64(v[m].x, ex);
        phi[N + t + G * m] = bad ? nan : fx_to_f64(v[m].y, ex);
      }
    }
  }
}

}  // namespace dsnu
