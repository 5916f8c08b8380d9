// FP64 (DSNU_FP64) plans: the FFT passes in 64-bit block fixed point
// (kernels_fx.cuh, standard_fx.cuh), interpolation and spreading sums too
// (spread_fx.cuh), the polar weighting in FP64.
#include <algorithm>

#include "kernels_fx.cuh"
#include "pipeline.cuh"
#include "spread_fx.cuh"
#include "standard_fx.cuh"

namespace dsnu {

namespace {

template <int L2>
cudaError_t prepare_fx_rows(PlanGeom& g) {
  using GG = FxGeo<L2>;
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e;
  g.smem_rowi = GG::smem_row_inv(g.Q);
  if ((e = cudaFuncSetAttribute(k_fx_row_fwd<L2>, A, int(GG::smem)))) return e;
  if ((e = cudaFuncSetAttribute(k_fx_row_inv<L2>, A, int(GG::smem_row_inv(GG::N))))) return e;
  if ((e = resident_ctas(k_fx_row_fwd<L2>, GG::T, GG::smem, &g.cap_rowf))) return e;
  return resident_ctas(k_fx_row_inv<L2>, GG::T, g.smem_rowi, &g.cap_rowi);
}

template <int L2>
cudaError_t prepare_fx_cols(PlanGeom& g) {
  using GG = FxGeo<L2>;
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_fx_col_main<L2, false>, A, int(GG::smem)))) return e;
  if ((e = cudaFuncSetAttribute(k_fx_col_main<L2, true>, A, int(GG::smem)))) return e;
  if ((e = cudaFuncSetAttribute(k_fx_band_fwd<L2>, A, int(GG::smem)))) return e;
  if ((e = cudaFuncSetAttribute(k_fx_band_inv<L2>, A, int(GG::smem)))) return e;
  if ((e = g.m1_full ? resident_ctas(k_fx_col_main<L2, true>, GG::T, GG::smem, &g.cap_col)
                     : resident_ctas(k_fx_col_main<L2, false>, GG::T, GG::smem, &g.cap_col)))
    return e;
  if ((e = resident_ctas(k_fx_band_fwd<L2>, GG::T, GG::smem, &g.cap_bandf))) return e;
  return resident_ctas(k_fx_band_inv<L2>, GG::T, GG::smem, &g.cap_bandi);
}

template <int L2>
cudaError_t prepare_fx_std_rows(PlanGeom& g) {
  using GG = FxOne<L2>;
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_fx_std_row_fwd<L2>, A, int(GG::smem)))) return e;
  if ((e = cudaFuncSetAttribute(k_fx_std_row_inv<L2>, A, int(GG::smem)))) return e;
  if ((e = resident_ctas(k_fx_std_row_fwd<L2>, GG::T, GG::smem, &g.cap_rowf))) return e;
  return resident_ctas(k_fx_std_row_inv<L2>, GG::T, GG::smem, &g.cap_rowi);
}

template <int L2>
cudaError_t prepare_fx_std_cols(PlanGeom& g) {
  using GG = FxOne<L2>;
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_fx_std_col<L2, false>, A, int(GG::smem)))) return e;
  if ((e = cudaFuncSetAttribute(k_fx_std_col<L2, true>, A, int(GG::smem)))) return e;
  return g.m1_full ? resident_ctas(k_fx_std_col<L2, true>, GG::T, GG::smem, &g.cap_col)
                   : resident_ctas(k_fx_std_col<L2, false>, GG::T, GG::smem, &g.cap_col);
}

// The standard solver's three passes (run_standard in fixed point).
dsnu_status run_standard_fx(const PlanGeom& g, const PlanTables& t, const WsLayout& L, const Members& mem,
                            cudaStream_t st, cudaEvent_t* ev) {
  const fxw* sx = static_cast<const fxw*>(t.fx_stw_x);
  const fxw* sy = static_cast<const fxw*>(t.fx_stw_y);
  const FxMult mt{static_cast<const fxr*>(t.m1tab), t.fx_mexp, g.m1_ld};
  const bool pdl = g.pdl != 0;
  const int ldq = L.ldqA;
  auto grid = [&](long n, int per, int cap) { return dim3(persistent_grid(mem.count * ((n + per - 1) / per), cap)); };
#define DSNU_SROWF(L2)                                                                                         \
  launch_k(pdl, k_fx_std_row_fwd<L2>, grid(g.ny / 2, FxOne<L2>::PER, g.cap_rowf), dim3(FxOne<L2>::T),          \
           FxOne<L2>::smem, st, mem, L.off_A, L.off_rexp, ldq, g.ny, sx)
#define DSNU_SCOL(L2)                                                                                          \
  if (g.m1_full)                                                                                               \
    launch_k(pdl, k_fx_std_col<L2, true>, grid(ldq, FxOne<L2>::PER, g.cap_col), dim3(FxOne<L2>::T),            \
             FxOne<L2>::smem, st, mem, L.off_A, L.off_rexp, L.off_cexp, ldq, ldq, sy, mt);                     \
  else                                                                                                         \
    launch_k(pdl, k_fx_std_col<L2, false>, grid(ldq, FxOne<L2>::PER, g.cap_col), dim3(FxOne<L2>::T),           \
             FxOne<L2>::smem, st, mem, L.off_A, L.off_rexp, L.off_cexp, ldq, ldq, sy, mt)
#define DSNU_SROWI(L2)                                                                                         \
  launch_k(pdl, k_fx_std_row_inv<L2>, grid(g.ny / 2, FxOne<L2>::PER, g.cap_rowi), dim3(FxOne<L2>::T),          \
           FxOne<L2>::smem, st, mem, L.off_A, L.off_cexp, ldq, g.ny, sx, -(ilogb(double(g.nx)) + ilogb(double(g.ny))))
  if (ev) cudaEventRecord(ev[0], st);
  switch (g.log2nx) {
    DSNU_LOG2_CASES(DSNU_SROWF)
    default: return DSNU_EUNSUPPORTED;
  }
  if (ev)
    for (int i = 1; i <= 6; ++i) cudaEventRecord(ev[i], st);
  switch (g.log2ny) {
    DSNU_LOG2_CASES(DSNU_SCOL)
    default: return DSNU_EUNSUPPORTED;
  }
  if (ev) cudaEventRecord(ev[7], st);
  switch (g.log2nx) {
    DSNU_LOG2_CASES(DSNU_SROWI)
    default: return DSNU_EUNSUPPORTED;
  }
  if (ev) cudaEventRecord(ev[8], st);
#undef DSNU_SROWF
#undef DSNU_SCOL
#undef DSNU_SROWI
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string("kernel launch failed: ") + cudaGetErrorString(e));
    return DSNU_ECUDA;
  }
  return DSNU_OK;
}

}  // namespace

cudaError_t prepare_kernels_f64(PlanGeom& g) {
  cudaError_t e = cudaFuncSetAttribute(k_fx_interp_tile, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(interp_fx_smem(16)));
  if (e != cudaSuccess) return e;
#define DSNU_PREP_R(L2) e = g.standard ? prepare_fx_std_rows<L2>(g) : prepare_fx_rows<L2>(g)
#define DSNU_PREP_C(L2) e = g.standard ? prepare_fx_std_cols<L2>(g) : prepare_fx_cols<L2>(g)
  switch (g.log2nx) {
    DSNU_LOG2_CASES(DSNU_PREP_R)
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  switch (g.log2ny) {
    DSNU_LOG2_CASES(DSNU_PREP_C)
    default: return cudaErrorInvalidValue;
  }
#undef DSNU_PREP_R
#undef DSNU_PREP_C
  return e;
}

dsnu_status run_pipeline_f64(const PlanGeom& g, const PlanTables& t, const WsLayout& L, const Members& mem,
                             cudaStream_t st, int cj, cudaEvent_t* ev, const Overlap* ov) {
  // the conjugated pipeline of a real input is the conjugate of this one: the
  // same result (kernels_fx.cuh), so `cj` selects nothing
  (void)cj;
  if (g.standard) return run_standard_fx(g, t, L, mem, st, ev);
  const WsOff off{L.off_A, L.off_B, L.off_Bband, L.off_Sband, L.off_c, L.off_partial, L.off_sched};
  const FxOff fo{L.off_A, L.off_B, L.off_Bband, L.off_Sband, L.off_rexp, L.off_rexpb, L.off_cexp, L.off_bexp};
  const FxAxis ax{static_cast<const fxw*>(t.fx_stw_x), static_cast<const fxw*>(t.fx_wm_x),
                  static_cast<const fxr*>(t.fx_dec_x)};
  const FxAxis ay{static_cast<const fxw*>(t.fx_stw_y), static_cast<const fxw*>(t.fx_wm_y),
                  static_cast<const fxr*>(t.fx_dec_y)};
  const FxMult mt{static_cast<const fxr*>(t.m1tab), t.fx_mexp, g.m1_ld};
  const bool pdl = g.pdl != 0;
  const long nm = mem.count;
  auto grid = [&](long n, int per, int cap) { return dim3(persistent_grid(nm * ((n + per - 1) / per), cap)); };
#define DSNU_ROWF(L2)                                                                                       \
  launch_k(pdl, k_fx_row_fwd<L2>, grid(g.ny, FxGeo<L2>::PER, g.cap_rowf), dim3(FxGeo<L2>::T), FxGeo<L2>::smem, st, \
           mem, fo, L.ldqA, L.ldqB, g.Q, g.ny, ax, g.kdx)
#define DSNU_BANDF(L2)                                                                                      \
  launch_k(pdl, k_fx_band_fwd<L2>, grid(g.Q + 1, FxGeo<L2>::PER, g.cap_bandf), dim3(FxGeo<L2>::T), FxGeo<L2>::smem, \
           bst, mem, fo, L.ldqB, g.Q + 1, L.ldq, g.Q, ay, g.kdy)
#define DSNU_BANDI(L2)                                                                                      \
  launch_k(pdl, k_fx_band_inv<L2>, grid(g.Q + 1, FxGeo<L2>::PER, g.cap_bandi), dim3(FxGeo<L2>::T), FxGeo<L2>::smem, \
           bst, mem, fo, L.ldq, g.Q, g.Q + 1, L.ldqB, ay, g.kdy)
#define DSNU_COLM(L2)                                                                                       \
  if (g.m1_full)                                                                                            \
    launch_k(pdl, k_fx_col_main<L2, true>, grid(g.nx + 1, FxGeo<L2>::PER, capc), dim3(FxGeo<L2>::T),   \
             FxGeo<L2>::smem, cst, mem, fo, L.ldqA, g.nx + 1, ay, mt);                                       \
  else                                                                                                      \
    launch_k(pdl, k_fx_col_main<L2, false>, grid(g.nx + 1, FxGeo<L2>::PER, capc), dim3(FxGeo<L2>::T),  \
             FxGeo<L2>::smem, cst, mem, fo, L.ldqA, g.nx + 1, ay, mt)
#define DSNU_ROWI(L2)                                                                                       \
  launch_k(pdl, k_fx_row_inv<L2>, grid(g.ny, FxGeo<L2>::PER, g.cap_rowi), dim3(FxGeo<L2>::T), g.smem_rowi, st, \
           mem, fo, L.ldqA, L.ldqB, g.Q, g.ny, ax, g.kdx, -(ilogb(double(g.mx)) + ilogb(double(g.my))))
#define DSNU_STEP(SIZE, CALL)              \
  switch (SIZE) {                          \
    DSNU_LOG2_CASES(CALL)                  \
    default: return DSNU_EUNSUPPORTED;     \
  }
#define DSNU_MARK(I) \
  if (ev) cudaEventRecord(ev[I], st)
  // the band chain (stream bst) next to the column pass (cst), one of them on
  // the plan's side stream and the column pass leaving `reserve` SMs free, or
  // both in line (no `ov`, profiling)
  cudaStream_t bst = st, cst = st;
  int capc = g.cap_col;
  auto band_chain = [&]() -> dsnu_status {
    DSNU_STEP(g.log2ny, DSNU_BANDF)
    DSNU_MARK(2);
    launch_k(pdl, k_fx_interp_tile, dim3(g.n_itiles, mem.count), dim3(256), interp_fx_smem(g.w), bst, mem, off, L.ldq,
             g.Q, t.node_q0, static_cast<const int2*>(t.node_w), t.node_D, t.itile_ptr, t.itile_org, t.itile_nodes, g.w,
             g.n_half);
    DSNU_MARK(3);
    launch_spread_fx(g.spread_cfg, mem, off, t, g, L.ldq, bst, 0, pdl);
    DSNU_MARK(4);
    launch_spread_fx(g.spread_cfg, mem, off, t, g, L.ldq, bst, 1, pdl);
    DSNU_MARK(5);
    DSNU_STEP(g.log2ny, DSNU_BANDI)
    DSNU_MARK(6);
    return DSNU_OK;
  };
  DSNU_MARK(0);
  DSNU_STEP(g.log2nx, DSNU_ROWF)
  DSNU_MARK(1);
  if (ov && !ev) {
    cudaEventRecord(ov->fork, st);
    cudaStreamWaitEvent(ov->side, ov->fork, 0);
    capc = std::max(1, g.cap_col - ov->reserve * (g.cap_col / g.sms));
    (ov->col_side ? cst : bst) = ov->side;
    DSNU_STEP(g.log2ny, DSNU_COLM)
    const dsnu_status sb = band_chain();
    if (sb != DSNU_OK) return sb;
    cudaEventRecord(ov->join, ov->side);
    cudaStreamWaitEvent(st, ov->join, 0);
  } else {
    const dsnu_status sb = band_chain();
    if (sb != DSNU_OK) return sb;
    DSNU_STEP(g.log2ny, DSNU_COLM)
  }
  DSNU_MARK(7);
  DSNU_STEP(g.log2nx, DSNU_ROWI)
  DSNU_MARK(8);
#undef DSNU_ROWF
#undef DSNU_COLM
#undef DSNU_BANDF
#undef DSNU_BANDI
#undef DSNU_ROWI
#undef DSNU_STEP
#undef DSNU_MARK
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string("kernel launch failed: ") + cudaGetErrorString(e));
    return DSNU_ECUDA;
  }
  return DSNU_OK;
}

cudaError_t time_spread_f64(const PlanGeom& g, const PlanTables& t, const WsLayout& L, void* ws, int reps,
                            float* ms) {
  return time_spread(L, ws, reps, ms, [&](const Members& mem, const WsOff& off) {
    launch_spread_fx(g.spread_cfg, mem, off, t, g, L.ldq, 0, 2, false);
  });
}

}  // namespace dsnu
