// ds.cu -- split-step (time-splitting spectral) pieces of the DS time loop.
//
// Sec. 2.3 of the paper advances i u_t = -u_xx + alpha u_yy - 2 beta |u|^2 u
// - 4 beta Phi u (eq. DSII_exact) by composing
//   * the linear flow (eqs. 1st_tssp, 1st_tssp_more), exact in Fourier space on
//     the periodic N x N grid:  v_hat <- exp(-i tau (k_x^2 - alpha k_y^2)) v_hat;
//   * the nonlinear flow (eqs. 2nd_tssp, 2nd_tssp_more), pointwise with the
//     density and Phi frozen:  w <- w exp(i tau (2 beta |w|^2 + 4 beta Phi)).
// This file provides both flows on the GPU plus the pieces of their
// vector-Jacobian products; Phi itself comes from the potential solver.
// Complex fields are interleaved (re, im) [ny][nx]: complex64 for a DSNU_MIXED
// plan, complex128 for DSNU_FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "internal.h"
#include "kernels_fx.cuh"
#include "tables.h"

namespace dsnu {

// Geometry of the unpadded 2D transform (rows: length nx; columns: length ny).
template <typename R, int LOG2N>
struct GeoC2C {
  static constexpr int N = 1 << LOG2N;
  static constexpr int G = N / 16;
  static constexpr int FB = fft_buf_elems(N);
  static constexpr int PER = (G >= 256) ? 1 : 256 / G;  // rows per CTA
  static constexpr int T = PER * G;
  static constexpr int STW = fft_stage_tw_elems(LOG2N) > 0 ? fft_stage_tw_elems(LOG2N) : 1;
  static constexpr int STWP = (STW + 1) & ~1;
  static constexpr size_t smem = size_t(STWP + PER * FB) * sizeof(cpx<R>);
  // column pass: C adjacent columns, their threads interleaved (see the kernel),
  // SETS such sets per CTA; buffers 16/C elements apart modulo 16
  static constexpr int C = (G >= 256) ? 2 : 4;
  static constexpr int SETS = (C * G >= 256) ? 1 : 256 / (C * G);
  static constexpr int TC = SETS * C * G;
  static constexpr int RS = ((FB + 15) & ~15) + 16 / C;
  static constexpr size_t smem_cols = size_t(STWP + SETS * C * RS) * sizeof(cpx<R>);
};

// Length-nx DFT of every row of src into dst (which may be src; inv:
// unnormalised inverse).
template <typename R, int LOG2N>
__global__ void __launch_bounds__(GeoC2C<R, LOG2N>::T)
k_c2c_rows(const cpx<R>* src, cpx<R>* dst, int ny, const cpx<R>* __restrict__ stw_g, int inv) {
  using GG = GeoC2C<R, LOG2N>;
  constexpr int N = GG::N, G = GG::G, PER = GG::PER;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<R>* stw = reinterpret_cast<cpx<R>*>(smem_raw);
  cpx<R>* sm = stw + GG::STWP;
  copy_to_smem(stw, stw_g, GG::STW);
  const int tid = threadIdx.x;
  const int rr = tid / G, t = tid - rr * G;
  cpx<R>* buf = sm + rr * GG::FB;
  const int items = (ny + PER - 1) / PER;
  grid_dep_wait();
#pragma unroll 1
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    if (item + int(gridDim.x) >= items) grid_dep_trigger();  // last item of this CTA
    const int row = item * PER + rr;
    const bool valid = row < ny;
    cpx<R> v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = valid ? src[size_t(row) * N + t + G * m] : mk<R>(R(0), R(0));
    block_fft_regs<R, LOG2N>(v, buf, t, stw, inv != 0);
    if (valid) {
#pragma unroll
      for (int m = 0; m < 16; ++m) dst[size_t(row) * N + t + G * m] = v[m];
    }
  }
}

// Per column: DFT along y, multiply by px[col] py[k] * scale (conjugated when
// adj), inverse DFT along y; in place.  px, py: the separable linear-flow
// phases e^{-i tau k_x^2} and e^{+i tau alpha k_y^2} in FFT order.  Four adjacent
// columns (two at ny = 4096) go together with their threads interleaved lane by
// lane: every access moves whole 32-byte sectors (one column per group of
// threads moved 8 of each 32 bytes; linear flow of a 1024^2 complex64 field 33.9
// -> 20.7 us, 2048^2 90 -> 59, with the launches overlapped).
template <typename R, int LOG2N>
__global__ void __launch_bounds__(GeoC2C<R, LOG2N>::TC)
k_c2c_cols_phase(cpx<R>* __restrict__ u, int nx, const cpx<R>* __restrict__ stw_g,
                 const cpx<R>* __restrict__ px, const cpx<R>* __restrict__ py, R scale, int adj) {
  using GG = GeoC2C<R, LOG2N>;
  constexpr int G = GG::G, C = GG::C, SETS = GG::SETS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<R>* stw = reinterpret_cast<cpx<R>*>(smem_raw);
  cpx<R>* sm = stw + GG::STWP;
  copy_to_smem(stw, stw_g, GG::STW);
  const int set = threadIdx.x / (C * G), r = threadIdx.x - set * (C * G);
  const int cl = r % C, t = r / C;
  cpx<R>* buf = sm + (set * C + cl) * GG::RS;
  const int items = (nx / C + SETS - 1) / SETS;
  grid_dep_wait();
#pragma unroll 1
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    if (item + int(gridDim.x) >= items) grid_dep_trigger();  // last item of this CTA
    const int col = (item * SETS + set) * C + cl;
    const bool valid = col < nx;
    cpx<R> v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m)
      v[m] = valid ? u[size_t(t + G * m) * nx + col] : mk<R>(R(0), R(0));
    block_fft_regs<R, LOG2N>(v, buf, t, stw, false);
    cpx<R> pxc = valid ? px[col] : mk<R>(R(0), R(0));
    if (adj) pxc.y = -pxc.y;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      cpx<R> p = py[t + G * m];
      if (adj) p.y = -p.y;
      v[m] = cmul(v[m], cmul(pxc, p)) * scale;
    }
    block_fft_regs<R, LOG2N>(v, buf, t, stw, true);
    if (valid) {
#pragma unroll
      for (int m = 0; m < 16; ++m) u[size_t(t + G * m) * nx + col] = v[m];
    }
  }
}

// ---------------------------------------------------------------------------
// The same two passes for complex128 fields, in 64-bit block fixed point
// (fx.cuh): each row and each pair of columns is scaled to its own largest
// component on loading and written back in FP64, so the passes keep no state
// between them (the field is the caller's, and several fields may be under way).
// An infinity or a NaN makes its whole row, then every column, NaN.

// u[row][t + G m] of group threads t: the values' bits, and their largest
// exponent (fx_top).
template <int P, int E>
__device__ __forceinline__ unsigned fx_load(fxc (&v)[E], const double2* u, size_t stride, bool valid,
                                            unsigned* red) {
  unsigned mx = 0;
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const double2 a = valid ? u[stride * m] : make_double2(0.0, 0.0);
    mx = fx_top(fx_top(mx, a.x), a.y);
    v[m] = fx_mk(__double_as_longlong(a.x), __double_as_longlong(a.y));
  }
  mx = fx_post<P, true>(mx, red);
  __syncthreads();
  mx = fx_read<P, true>(mx, red);
  const int efm = fx_efm(mx);
#pragma unroll
  for (int m = 0; m < E; ++m)
    v[m] = fx_shr<5>(fx_mk(fx_from_f64(__longlong_as_double(v[m].x), efm), fx_from_f64(__longlong_as_double(v[m].y), efm)));
  return mx;
}
__device__ __forceinline__ double2 fx_store(fxc v, int ex, unsigned mx) {
  const double nan = __longlong_as_double(0x7FF8000000000000ll);
  return mx >= kFxInf ? make_double2(nan, nan) : make_double2(fx_to_f64(v.x, ex), fx_to_f64(v.y, ex));
}

template <int LOG2N>
__global__ void __launch_bounds__(FxOne<LOG2N>::T, FxOne<LOG2N>::MINB)
k_fx_c2c_rows(const double2* src, double2* dst, int ny, const fxw* __restrict__ stw_g, int inv) {
  using GG = FxOne<LOG2N>;
  constexpr int N = GG::N, E = GG::E, G = GG::G, PER = GG::PER, W = GG::W;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fxw* stw = reinterpret_cast<fxw*>(smem_raw);
  fxc* sm = reinterpret_cast<fxc*>(stw + GG::STW);
  unsigned* red = reinterpret_cast<unsigned*>(sm + PER * GG::FB);
  fx_copy(stw, stw_g, FxRad<LOG2N>::stw());
  const int pr = threadIdx.x / G, t = threadIdx.x - pr * G;
  fxc* buf = sm + pr * GG::FB;
  __syncthreads();
  const int items = (ny + PER - 1) / PER;
  grid_dep_wait();
#pragma unroll 1
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    if (item + int(gridDim.x) >= items) grid_dep_trigger();  // last item of this CTA
    const int row = item * PER + pr;
    const bool valid = row < ny;
    const size_t at = size_t(valid ? row : 0) * N + t;
    fxc v[E];
    const unsigned mx = fx_load<G, E>(v, src + at, G, valid, red + 2 * W);
    if (inv) {
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = fx_swap(v[m]);
    }
    const int ex = fx_efm(mx) - kFxBias + 5 + fx_fft<LOG2N, G>(v, buf, t, stw, red);
    if (valid) {
#pragma unroll
      for (int m = 0; m < E; ++m) dst[at + G * m] = fx_store(inv ? fx_swap(v[m]) : v[m], ex, mx);
    }
  }
}

// Two adjacent columns per pair of groups, their threads interleaved (whole
// 32-byte sectors), with one scale; buffers 4 elements apart modulo 8, so that
// the two columns' lanes of a quarter warp fall in different banks.
template <int LOG2N>
struct FxCols : FxGeo<LOG2N> {
  using B = FxGeo<LOG2N>;
  static constexpr int FBS = B::FB + 4 + ((8 - (B::FB & 7)) & 7);
  static constexpr size_t smem = size_t(B::STW + B::PER * 2 * FBS) * 16 + ((B::RED * 4 + 15) & ~15);
  static_assert(smem <= 232448, "shared memory per CTA");
};

// px, py: the phases in fixed point (k_phase_tables_fx); the result carries
// 2^lscale = 1/(nx ny).
template <int LOG2N>
__global__ void __launch_bounds__(FxCols<LOG2N>::T, FxCols<LOG2N>::MINB)
k_fx_c2c_cols_phase(double2* __restrict__ u, int nx, const fxw* __restrict__ stw_g, const fxw* __restrict__ px,
                    const fxw* __restrict__ py, int lscale, int adj) {
  using GG = FxCols<LOG2N>;
  constexpr int E = GG::E, G = GG::G, P = GG::P, PER = GG::PER, W = GG::W;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fxw* stw = reinterpret_cast<fxw*>(smem_raw);
  fxc* sm = reinterpret_cast<fxc*>(stw + GG::STW);
  unsigned* red = reinterpret_cast<unsigned*>(sm + PER * 2 * GG::FBS);
  fx_copy(stw, stw_g, FxRad<LOG2N>::stw());
  const int pr = threadIdx.x / P, tp = threadIdx.x - pr * P;
  const int h = tp & 1, t = tp >> 1;
  fxc* buf = sm + (2 * pr + h) * GG::FBS;
  __syncthreads();
  const int items = (nx / 2 + PER - 1) / PER;
  grid_dep_wait();
#pragma unroll 1
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    if (item + int(gridDim.x) >= items) grid_dep_trigger();  // last item of this CTA
    const int col = 2 * (item * PER + pr) + h;
    const bool valid = col < nx;
    double2* uc = u + size_t(t) * nx + (valid ? col : h);
    fxc v[E];
    const unsigned mx = fx_load<P, E>(v, uc, size_t(G) * nx, valid, red + 2 * W);
    int ex = fx_efm(mx) - kFxBias + 5 + lscale;
#pragma unroll 1
    for (int inv = 0;; ++inv) {  // forward, then inverse (one copy of the transform's code)
      ex += fx_fft<LOG2N, P>(v, buf, t, stw, red);
      if (inv) break;
      const unsigned mag = fx_post<P>(fx_mag(v), red + 2 * W);
      __syncthreads();
      const int s = fx_norm_shift<62>(fx_read<P>(mag, red + 2 * W));
      ex += 4 - 3 + 4 - s;
      fxw wx = fx_ldw(px + (valid ? col : 0));
      if (adj) wx = fx_conj(wx);
#pragma unroll
      for (int m = 0; m < E; ++m) {
        fxw wy = fx_ldw(py + t + G * m);
        if (adj) wy = fx_conj(wy);
        // /16 by each phase (magnitudes < 2^62.5), 2^3 between them; components
        // exchanged for the inverse transform
        v[m] = fx_swap(fx_mul(fx_shl(fx_mul(fx_shl(v[m], s), wy), 3), wx));
      }
    }
    if (valid) {
#pragma unroll
      for (int m = 0; m < E; ++m) uc[size_t(G) * m * nx] = fx_store(fx_swap(v[m]), ex, mx);
    }
  }
}

// rho = |u|^2 (FP64 out).
template <typename R>
__global__ void k_abs2(const cpx<R>* __restrict__ u, double* __restrict__ rho, size_t n) {
  grid_dep_wait();
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
    const cpx<R> a = u[i];
    rho[i] = to_f64<R>(a.x * a.x + a.y * a.y);
  }
}

// Vector-Jacobian product of rho = |u|^2 for a real loss (gradients in the
// d/dRe + i d/dIm convention): grad_u = 2 g_rho u, g_rho FP64.
template <typename R>
__global__ void k_abs2_vjp(const cpx<R>* __restrict__ u, const double* __restrict__ g_rho,
                           cpx<R>* __restrict__ grad, size_t n) {
  grid_dep_wait();
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
    const cpx<R> a = u[i];
    const R g2 = R(2) * from_f64<R>(g_rho[i]);
    grad[i] = mk<R>(g2 * a.x, g2 * a.y);
  }
}

template <typename R>
__device__ __forceinline__ void sincos_r(R a, R* s, R* c) {
  if constexpr (sizeof(R) == 4) sincosf(a, s, c);
  else sincos(a, s, c);
}

// theta = tau (2 beta |u|^2 + 4 beta Phi) at a point.
template <typename R>
__device__ __forceinline__ R nl_angle(cpx<R> a, double phi, R tau, R beta) {
  return tau * (R(2) * beta * (a.x * a.x + a.y * a.y) + R(4) * beta * from_f64<R>(phi));
}

// out = u e^{i theta} (out may be u).
template <typename R>
__global__ void k_nonlinear(const cpx<R>* u, cpx<R>* out, const double* __restrict__ phi, size_t n, R tau,
                            R beta) {
  grid_dep_wait();
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
    const cpx<R> a = u[i];
    R s, c;
    sincos_r(nl_angle(a, phi[i], tau, beta), &s, &c);
    out[i] = cmul(a, mk<R>(c, s));
  }
}

// Backward of u' = u e^{i theta(|u|^2)} for a real loss, gradients in the
// (d/dRe + i d/dIm) convention:  given g' at u', returns
//   part = g' e^{-i theta}        (the direct term)
//   sfld = Im(g' conj(u'))        (so that dL = <tau (2 beta s + 4 beta A^T s), d rho> + ...)
template <typename R>
__global__ void k_nonlinear_vjp(const cpx<R>* __restrict__ u, const double* __restrict__ phi,
                                const cpx<R>* __restrict__ g, size_t n, R tau, R beta,
                                double* __restrict__ sfld, cpx<R>* __restrict__ part) {
  grid_dep_wait();
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
    const cpx<R> a = u[i];
    R s, c;
    sincos_r(nl_angle(a, phi[i], tau, beta), &s, &c);
    const cpx<R> e = mk<R>(c, s);
    const cpx<R> up = cmul(a, e);
    const cpx<R> gi = g[i];
    part[i] = cmulc(gi, e);                              // g' e^{-i theta}
    sfld[i] = to_f64<R>(gi.y * up.x - gi.x * up.y);      // Im(g' conj u')
  }
}

// grad_u = part + 2 tau (2 beta s + 4 beta (A^T s)) u   (in place on part)
template <typename R>
__global__ void k_nonlinear_vjp_finish(const cpx<R>* __restrict__ u, const double* __restrict__ sfld,
                                       const double* __restrict__ ats, size_t n, R tau, R beta,
                                       cpx<R>* __restrict__ part) {
  grid_dep_wait();
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
    const R grho = tau * (R(2) * beta * from_f64<R>(sfld[i]) + R(4) * beta * from_f64<R>(ats[i]));
    const cpx<R> a = u[i];
    const cpx<R> p = part[i];
    part[i] = mk<R>(p.x + R(2) * grho * a.x, p.y + R(2) * grho * a.y);
  }
}

// Linear-flow phase tables in FFT order: px[q] = e^{-i tau k_x^2} and
// py[q] = e^{+i tau alpha k_y^2}, k = qs dk with qs the signed index.  The
// angles and their sine/cosine are formed in FP64 and rounded to FP32 (or put
// in fixed point, below); launched on the caller's stream, so a change of step size needs
// no host round trip.
template <typename R>
__global__ void k_phase_tables(cpx<R>* __restrict__ px, cpx<R>* __restrict__ py, int nx, int ny, double dkx,
                               double dky, double tau, double alpha) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nx) {
    const double k = double(i < nx / 2 ? i : i - nx) * dkx;
    double s, c;
    sincos(-tau * k * k, &s, &c);
    px[i] = mk<R>(R(c), R(s));
  }
  if (i < ny) {
    const double k = double(i < ny / 2 ? i : i - ny) * dky;
    double s, c;
    sincos(tau * alpha * k * k, &s, &c);
    py[i] = mk<R>(R(c), R(s));
  }
}

// The same in fixed point (fxw, 2^kFxTwBits), for complex128 plans.
__device__ __forceinline__ fxw fx_unit(double c, double s) {
  auto half = [](double v, int& h, int& l) {
    const double x = v * double(1 << kFxTwBits), r = rint(x);
    h = int(r);
    l = int(fmax(fmin(rint((x - r) * 4294967296.0), 2147483647.0), -2147483647.0));
  };
  fxw w;
  half(c, w.rh, w.rl);
  half(s, w.ih, w.il);
  return w;
}
__global__ void k_phase_tables_fx(fxw* __restrict__ px, fxw* __restrict__ py, int nx, int ny, double dkx, double dky,
                                  double tau, double alpha) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double s, c;
  if (i < nx) {
    const double k = double(i < nx / 2 ? i : i - nx) * dkx;
    sincos(-tau * k * k, &s, &c);
    px[i] = fx_unit(c, s);
  }
  if (i < ny) {
    const double k = double(i < ny / 2 ? i : i - ny) * dky;
    sincos(tau * alpha * k * k, &s, &c);
    py[i] = fx_unit(c, s);
  }
}

}  // namespace dsnu

using namespace dsnu;

struct dsnu_ds_plan_s {
  dsnu_ds_params prm;
  int log2nx, log2ny;
  void* block;       // stage twiddles of both axes + phase tables
  void* stw_x;
  void* stw_y;
  void* px;          // nx complex
  void* py;          // ny complex
  double tau, alpha; // phases currently loaded
  bool has_phase;
  int grid_rows, grid_cols;
  bool pdl;          // launches with programmatic stream serialization
};

namespace {

dsnu_status ds_fail(dsnu_status s, const std::string& m) {
  dsnu::set_last_error(m);
  return s;
}

template <typename R, typename V>
void upload(void* dst, const V& v, cudaStream_t st, cudaError_t* e) {
  std::vector<R> tmp(v.begin(), v.end());
  if (*e == cudaSuccess) *e = cudaMemcpyAsync(dst, tmp.data(), tmp.size() * sizeof(R), cudaMemcpyHostToDevice, st);
  if (*e == cudaSuccess) *e = cudaStreamSynchronize(st);
}

template <typename K>
int grid_for(K kernel, int threads, size_t smem, int items) {
  int dev = 0, sms = 1, per = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
  if (per < 1) per = 1;
  const int cap = sms * per;
  return items < cap ? (items > 0 ? items : 1) : cap;
}

#define DSNU_C2C_CASES(CALL) \
  case 4: CALL(4); break;    \
  case 5: CALL(5); break;    \
  case 6: CALL(6); break;    \
  case 7: CALL(7); break;    \
  case 8: CALL(8); break;    \
  case 9: CALL(9); break;    \
  case 10: CALL(10); break;  \
  case 11: CALL(11); break;  \
  case 12: CALL(12); break;

cudaError_t prepare_f32(dsnu_ds_plan_s* P) {
  using R = float;
  cudaError_t e = cudaSuccess;
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
#define DSNU_PR(L2)                                                                                 \
  e = cudaFuncSetAttribute(k_c2c_rows<R, L2>, A, int(GeoC2C<R, L2>::smem));                        \
  if (e == cudaSuccess)                                                                             \
    P->grid_rows = grid_for(k_c2c_rows<R, L2>, GeoC2C<R, L2>::T, GeoC2C<R, L2>::smem,            \
                               (P->prm.ny + GeoC2C<R, L2>::PER - 1) / GeoC2C<R, L2>::PER)
#define DSNU_PC(L2)                                                                                 \
  e = cudaFuncSetAttribute(k_c2c_cols_phase<R, L2>, A, int(GeoC2C<R, L2>::smem_cols));             \
  if (e == cudaSuccess)                                                                             \
    P->grid_cols = grid_for(k_c2c_cols_phase<R, L2>, GeoC2C<R, L2>::TC, GeoC2C<R, L2>::smem_cols, \
                            (P->prm.nx / GeoC2C<R, L2>::C + GeoC2C<R, L2>::SETS - 1) / GeoC2C<R, L2>::SETS)
  switch (P->log2nx) {
    DSNU_C2C_CASES(DSNU_PR)
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  switch (P->log2ny) {
    DSNU_C2C_CASES(DSNU_PC)
    default: return cudaErrorInvalidValue;
  }
#undef DSNU_PR
#undef DSNU_PC
  return e;
}

cudaError_t prepare_f64(dsnu_ds_plan_s* P) {
  cudaError_t e = cudaSuccess;
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
#define DSNU_PR(L2)                                                                                 \
  e = cudaFuncSetAttribute(k_fx_c2c_rows<L2>, A, int(FxOne<L2>::smem));                             \
  if (e == cudaSuccess)                                                                             \
    P->grid_rows = grid_for(k_fx_c2c_rows<L2>, FxOne<L2>::T, FxOne<L2>::smem,                       \
                            (P->prm.ny + FxOne<L2>::PER - 1) / FxOne<L2>::PER)
#define DSNU_PC(L2)                                                                                 \
  e = cudaFuncSetAttribute(k_fx_c2c_cols_phase<L2>, A, int(FxCols<L2>::smem));                      \
  if (e == cudaSuccess)                                                                             \
    P->grid_cols = grid_for(k_fx_c2c_cols_phase<L2>, FxCols<L2>::T, FxCols<L2>::smem,               \
                            (P->prm.nx / 2 + FxCols<L2>::PER - 1) / FxCols<L2>::PER)
  switch (P->log2nx) {
    DSNU_C2C_CASES(DSNU_PR)
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  switch (P->log2ny) {
    DSNU_C2C_CASES(DSNU_PC)
    default: return cudaErrorInvalidValue;
  }
#undef DSNU_PR
#undef DSNU_PC
  return e;
}

dsnu_status linear_f32(dsnu_ds_plan_s* P, const void* uv, void* ov, int adjoint, cudaStream_t st) {
  using R = float;
  const cpx<R>* in = static_cast<const cpx<R>*>(uv);
  cpx<R>* u = static_cast<cpx<R>*>(ov);
  const R scale = R(1.0 / (double(P->prm.nx) * double(P->prm.ny)));
  const cpx<R>* sx = static_cast<const cpx<R>*>(P->stw_x);
  const cpx<R>* sy = static_cast<const cpx<R>*>(P->stw_y);
  const cpx<R>* px = static_cast<const cpx<R>*>(P->px);
  const cpx<R>* py = static_cast<const cpx<R>*>(P->py);
#define DSNU_ROWS(L2, SRC, INV)                                                                       \
  launch_k(P->pdl, k_c2c_rows<R, L2>, dim3(P->grid_rows), dim3(GeoC2C<R, L2>::T), GeoC2C<R, L2>::smem, st, SRC, u, \
           P->prm.ny, sx, INV)
#define DSNU_RF(L2) DSNU_ROWS(L2, in, 0)
#define DSNU_RI(L2) DSNU_ROWS(L2, static_cast<const cpx<R>*>(u), 1)
#define DSNU_CP(L2)                                                                                   \
  launch_k(P->pdl, k_c2c_cols_phase<R, L2>, dim3(P->grid_cols), dim3(GeoC2C<R, L2>::TC), GeoC2C<R, L2>::smem_cols, st, \
           u, P->prm.nx, sy, px, py, scale, adjoint)
  switch (P->log2nx) {
    DSNU_C2C_CASES(DSNU_RF)
    default: return DSNU_EUNSUPPORTED;
  }
  switch (P->log2ny) {
    DSNU_C2C_CASES(DSNU_CP)
    default: return DSNU_EUNSUPPORTED;
  }
  switch (P->log2nx) {
    DSNU_C2C_CASES(DSNU_RI)
    default: return DSNU_EUNSUPPORTED;
  }
#undef DSNU_ROWS
#undef DSNU_RF
#undef DSNU_RI
#undef DSNU_CP
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DSNU_OK : ds_fail(DSNU_ECUDA, std::string("launch: ") + cudaGetErrorString(e));
}

dsnu_status linear_f64(dsnu_ds_plan_s* P, const void* uv, void* ov, int adjoint, cudaStream_t st) {
  const double2* in = static_cast<const double2*>(uv);
  double2* u = static_cast<double2*>(ov);
  const int lscale = -(P->log2nx + P->log2ny);
  const fxw* sx = static_cast<const fxw*>(P->stw_x);
  const fxw* sy = static_cast<const fxw*>(P->stw_y);
  const fxw* px = static_cast<const fxw*>(P->px);
  const fxw* py = static_cast<const fxw*>(P->py);
#define DSNU_ROWS(L2, SRC, INV)                                                                        \
  launch_k(P->pdl, k_fx_c2c_rows<L2>, dim3(P->grid_rows), dim3(FxOne<L2>::T), FxOne<L2>::smem, st, SRC, u, P->prm.ny, \
           sx, INV)
#define DSNU_RF(L2) DSNU_ROWS(L2, in, 0)
#define DSNU_RI(L2) DSNU_ROWS(L2, static_cast<const double2*>(u), 1)
#define DSNU_CP(L2)                                                                                    \
  launch_k(P->pdl, k_fx_c2c_cols_phase<L2>, dim3(P->grid_cols), dim3(FxCols<L2>::T), FxCols<L2>::smem, st, u, P->prm.nx, \
           sy, px, py, lscale, adjoint)
  switch (P->log2nx) {
    DSNU_C2C_CASES(DSNU_RF)
    default: return DSNU_EUNSUPPORTED;
  }
  switch (P->log2ny) {
    DSNU_C2C_CASES(DSNU_CP)
    default: return DSNU_EUNSUPPORTED;
  }
  switch (P->log2nx) {
    DSNU_C2C_CASES(DSNU_RI)
    default: return DSNU_EUNSUPPORTED;
  }
#undef DSNU_ROWS
#undef DSNU_RF
#undef DSNU_RI
#undef DSNU_CP
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DSNU_OK : ds_fail(DSNU_ECUDA, std::string("launch: ") + cudaGetErrorString(e));
}

int grid_1d(size_t n) {
  const size_t b = (n + 255) / 256;
  return int(b < 4096 ? b : 4096);
}

dsnu_status check_launch() {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DSNU_OK : ds_fail(DSNU_ECUDA, std::string("launch: ") + cudaGetErrorString(e));
}

// Bytes of a field, and whether two ranges share any.
size_t field_bytes(const dsnu_ds_plan_s* P) {
  return size_t(P->prm.nx) * P->prm.ny * (P->prm.precision == DSNU_MIXED ? sizeof(float2) : sizeof(double2));
}
bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const char *p = static_cast<const char*>(a), *q = static_cast<const char*>(b);
  return p < q + nb && q < p + na;
}

dsnu_status linear(dsnu_ds_plan_s* P, const void* u, void* out, int adjoint, cudaStream_t st) {
  if (!P->has_phase) return ds_fail(DSNU_EINVAL, "no linear step set (dsnu_ds_set_linear_step)");
  return P->prm.precision == DSNU_MIXED ? linear_f32(P, u, out, adjoint, st) : linear_f64(P, u, out, adjoint, st);
}

dsnu_status nonlinear(dsnu_ds_plan_s* P, const void* u, const double* phi, void* out, double tau, double beta,
                      cudaStream_t st) {
  const size_t n = size_t(P->prm.nx) * P->prm.ny;
  if (P->prm.precision == DSNU_MIXED)
    launch_k(P->pdl, k_nonlinear<float>, dim3(grid_1d(n)), dim3(256), 0, st, static_cast<const cpx<float>*>(u),
             static_cast<cpx<float>*>(out), phi, n, float(tau), float(beta));
  else
    launch_k(P->pdl, k_nonlinear<double>, dim3(grid_1d(n)), dim3(256), 0, st, static_cast<const cpx<double>*>(u),
             static_cast<cpx<double>*>(out), phi, n, tau, beta);
  return check_launch();
}

int ilog2i(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l;
}

}  // namespace

extern "C" {

dsnu_status dsnu_ds_plan_create(const dsnu_ds_params* params, void* stream, dsnu_ds_plan* out) {
  if (!params || !out) return ds_fail(DSNU_EINVAL, "NULL params or out");
  const dsnu_ds_params p = *params;
  auto pow2 = [](int v) { return v >= 16 && v <= 4096 && (v & (v - 1)) == 0; };
  if (!pow2(p.nx) || !pow2(p.ny)) return ds_fail(DSNU_EINVAL, "nx, ny must be powers of two in [16, 4096]");
  if (!(p.lx > 0.0) || !(p.ly > 0.0) || !std::isfinite(p.lx) || !std::isfinite(p.ly))
    return ds_fail(DSNU_EINVAL, "lx, ly must be positive and finite");
  if (p.precision != DSNU_FP64 && p.precision != DSNU_MIXED) return ds_fail(DSNU_EINVAL, "unknown precision");
  dsnu_ds_plan_s* P = new (std::nothrow) dsnu_ds_plan_s();
  if (!P) return ds_fail(DSNU_ENOMEM, "host allocation failed");
  P->prm = p;
  P->log2nx = ilog2i(p.nx);
  P->log2ny = ilog2i(p.ny);
  const size_t rsz = p.precision == DSNU_MIXED ? 4 : 8;
  std::vector<double> sx, sy;
  const bool fx = p.precision == DSNU_FP64;
  fft_stage_twiddles(P->log2nx, sx, fx ? fx_log2_radix(P->log2nx) : 4);
  fft_stage_twiddles(P->log2ny, sy, fx ? fx_log2_radix(P->log2ny) : 4);
  auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
  const size_t o_sx = 0, o_sy = al(sx.size() * rsz), o_px = o_sy + al(sy.size() * rsz);
  const size_t o_py = o_px + al(2 * size_t(p.nx) * rsz), total = o_py + al(2 * size_t(p.ny) * rsz);
  cudaError_t e = cudaMalloc(&P->block, total);
  if (e != cudaSuccess) {
    delete P;
    return ds_fail(DSNU_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  char* d = static_cast<char*>(P->block);
  P->stw_x = d + o_sx;
  P->stw_y = d + o_sy;
  P->px = d + o_px;
  P->py = d + o_py;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (p.precision == DSNU_MIXED) {
    upload<float>(P->stw_x, sx, st, &e);
    upload<float>(P->stw_y, sy, st, &e);
    if (e == cudaSuccess) e = prepare_f32(P);
  } else {
    upload<int>(P->stw_x, fx_table(sx, kFxTwBits), st, &e);
    upload<int>(P->stw_y, fx_table(sy, kFxTwBits), st, &e);
    if (e == cudaSuccess) e = prepare_f64(P);
  }
  if (e != cudaSuccess) {
    cudaFree(P->block);
    delete P;
    return ds_fail(DSNU_ECUDA, std::string("DS plan set-up: ") + cudaGetErrorString(e));
  }
  P->has_phase = false;
  const char* env = std::getenv("DSNU_PDL");  // DSNU_PDL=0: plain stream-ordered launches
  P->pdl = !(env && env[0] == '0');
  *out = P;
  return DSNU_OK;
}

dsnu_status dsnu_ds_set_linear_step(dsnu_ds_plan plan, double tau, double alpha, void* stream) {
  if (!plan) return ds_fail(DSNU_EINVAL, "NULL plan");
  if (!std::isfinite(tau) || !std::isfinite(alpha)) return ds_fail(DSNU_EINVAL, "tau, alpha must be finite");
  if (plan->has_phase && plan->tau == tau && plan->alpha == alpha) return DSNU_OK;
  const dsnu_ds_params& p = plan->prm;
  const double dkx = M_PI / p.lx, dky = M_PI / p.ly;  // 2 pi / (n h), h = 2 l / n
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int n = p.nx > p.ny ? p.nx : p.ny;
  if (p.precision == DSNU_MIXED)
    k_phase_tables<float><<<(n + 255) / 256, 256, 0, st>>>(static_cast<cpx<float>*>(plan->px),
                                                           static_cast<cpx<float>*>(plan->py), p.nx, p.ny,
                                                           dkx, dky, tau, alpha);
  else
    k_phase_tables_fx<<<(n + 255) / 256, 256, 0, st>>>(static_cast<fxw*>(plan->px), static_cast<fxw*>(plan->py), p.nx,
                                                       p.ny, dkx, dky, tau, alpha);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return ds_fail(DSNU_ECUDA, std::string("phase tables: ") + cudaGetErrorString(e));
  plan->tau = tau;
  plan->alpha = alpha;
  plan->has_phase = true;
  return DSNU_OK;
}

dsnu_status dsnu_ds_linear_to(dsnu_ds_plan plan, const void* u_dev, void* out_dev, int32_t adjoint, void* stream) {
  if (!plan || !u_dev || !out_dev) return ds_fail(DSNU_EINVAL, "NULL plan or field");
  const size_t nb = field_bytes(plan);
  if (out_dev != u_dev && overlap(u_dev, nb, out_dev, nb))
    return ds_fail(DSNU_EINVAL, "input and output overlap in part");
  return linear(plan, u_dev, out_dev, adjoint, static_cast<cudaStream_t>(stream));
}

dsnu_status dsnu_ds_linear(dsnu_ds_plan plan, void* u_dev, int32_t adjoint, void* stream) {
  if (!plan || !u_dev) return ds_fail(DSNU_EINVAL, "NULL plan or field");
  return linear(plan, u_dev, u_dev, adjoint, static_cast<cudaStream_t>(stream));
}

dsnu_status dsnu_ds_abs2(dsnu_ds_plan plan, const void* u_dev, double* rho_dev, void* stream) {
  if (!plan || !u_dev || !rho_dev) return ds_fail(DSNU_EINVAL, "NULL argument");
  const size_t n = size_t(plan->prm.nx) * plan->prm.ny;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan->prm.precision == DSNU_MIXED)
    launch_k(plan->pdl, k_abs2<float>, dim3(grid_1d(n)), dim3(256), 0, st, static_cast<const cpx<float>*>(u_dev), rho_dev, n);
  else
    launch_k(plan->pdl, k_abs2<double>, dim3(grid_1d(n)), dim3(256), 0, st, static_cast<const cpx<double>*>(u_dev), rho_dev, n);
  return check_launch();
}

dsnu_status dsnu_ds_abs2_vjp(dsnu_ds_plan plan, const void* u_dev, const double* g_rho_dev, void* grad_dev,
                             void* stream) {
  if (!plan || !u_dev || !g_rho_dev || !grad_dev) return ds_fail(DSNU_EINVAL, "NULL argument");
  const size_t n = size_t(plan->prm.nx) * plan->prm.ny;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan->prm.precision == DSNU_MIXED)
    launch_k(plan->pdl, k_abs2_vjp<float>, dim3(grid_1d(n)), dim3(256), 0, st, static_cast<const cpx<float>*>(u_dev), g_rho_dev,
                                                 static_cast<cpx<float>*>(grad_dev), n);
  else
    launch_k(plan->pdl, k_abs2_vjp<double>, dim3(grid_1d(n)), dim3(256), 0, st, static_cast<const cpx<double>*>(u_dev), g_rho_dev,
                                                  static_cast<cpx<double>*>(grad_dev), n);
  return check_launch();
}

dsnu_status dsnu_ds_nonlinear_to(dsnu_ds_plan plan, const void* u_dev, const double* phi_dev, void* out_dev, double tau,
                                 double beta, void* stream) {
  if (!plan || !u_dev || !phi_dev || !out_dev) return ds_fail(DSNU_EINVAL, "NULL argument");
  const size_t nb = field_bytes(plan);
  if ((out_dev != u_dev && overlap(u_dev, nb, out_dev, nb)) ||
      overlap(phi_dev, size_t(plan->prm.nx) * plan->prm.ny * sizeof(double), out_dev, nb))
    return ds_fail(DSNU_EINVAL, "the output overlaps phi, or the input in part");
  return nonlinear(plan, u_dev, phi_dev, out_dev, tau, beta, static_cast<cudaStream_t>(stream));
}

dsnu_status dsnu_ds_nonlinear(dsnu_ds_plan plan, void* u_dev, const double* phi_dev, double tau, double beta,
                              void* stream) {
  if (!plan || !u_dev || !phi_dev) return ds_fail(DSNU_EINVAL, "NULL argument");
  return nonlinear(plan, u_dev, phi_dev, u_dev, tau, beta, static_cast<cudaStream_t>(stream));
}

dsnu_status dsnu_ds_nonlinear_vjp(dsnu_ds_plan plan, const void* u_dev, const double* phi_dev, const void* g_dev,
                                  double tau, double beta, double* s_dev, void* part_dev, void* stream) {
  if (!plan || !u_dev || !phi_dev || !g_dev || !s_dev || !part_dev) return ds_fail(DSNU_EINVAL, "NULL argument");
  const size_t n = size_t(plan->prm.nx) * plan->prm.ny;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan->prm.precision == DSNU_MIXED)
    launch_k(plan->pdl, k_nonlinear_vjp<float>, dim3(grid_1d(n)), dim3(256), 0, st, 
        static_cast<const cpx<float>*>(u_dev), phi_dev, static_cast<const cpx<float>*>(g_dev), n, float(tau),
        float(beta), s_dev, static_cast<cpx<float>*>(part_dev));
  else
    launch_k(plan->pdl, k_nonlinear_vjp<double>, dim3(grid_1d(n)), dim3(256), 0, st, 
        static_cast<const cpx<double>*>(u_dev), phi_dev, static_cast<const cpx<double>*>(g_dev), n, tau, beta,
        s_dev, static_cast<cpx<double>*>(part_dev));
  return check_launch();
}

dsnu_status dsnu_ds_nonlinear_vjp_finish(dsnu_ds_plan plan, const void* u_dev, const double* s_dev,
                                         const double* ats_dev, double tau, double beta, void* grad_dev,
                                         void* stream) {
  if (!plan || !u_dev || !s_dev || !ats_dev || !grad_dev) return ds_fail(DSNU_EINVAL, "NULL argument");
  const size_t n = size_t(plan->prm.nx) * plan->prm.ny;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan->prm.precision == DSNU_MIXED)
    launch_k(plan->pdl, k_nonlinear_vjp_finish<float>, dim3(grid_1d(n)), dim3(256), 0, st, 
        static_cast<const cpx<float>*>(u_dev), s_dev, ats_dev, n, float(tau), float(beta),
        static_cast<cpx<float>*>(grad_dev));
  else
    launch_k(plan->pdl, k_nonlinear_vjp_finish<double>, dim3(grid_1d(n)), dim3(256), 0, st, 
        static_cast<const cpx<double>*>(u_dev), s_dev, ats_dev, n, tau, beta, static_cast<cpx<double>*>(grad_dev));
  return check_launch();
}

dsnu_status dsnu_ds_plan_destroy(dsnu_ds_plan plan) {
  if (!plan) return DSNU_OK;
  const cudaError_t e = cudaFree(plan->block);
  delete plan;
  return e == cudaSuccess ? DSNU_OK : ds_fail(DSNU_ECUDA, std::string("cudaFree: ") + cudaGetErrorString(e));
}

}  // extern "C"
