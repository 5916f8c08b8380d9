// spread_fx.cuh -- type-2 interpolation and type-1 spreading of the FP64 plans
// in fixed point (see k_interp_tile and k_spread in kernels.cuh for the tiles,
// items and node lists, which are the same).
//
// Both are sums of products with the ES weights: in FP64 three instructions of
// 16-20 SM cycles per stencil point, here six 32 x 32 + 64 bit multiply-adds of
// about one.  A work item scales its values (band values of the tile's region,
// coefficients of the item's nodes) to 54 bits relative to the largest of them,
//     v = vh 2^28 + vl,   weight w = wh 2^-28 + wl 2^-56   (|vl|, |wl| <= 2^27),
// and adds up  P += vh wh,  Q += vh wl + vl wh;  the sum of v w is P + Q 2^-28
// (the dropped vl wl terms are below 1/4 of the quantum).
// 16384 nodes of width 15 on Q = 170 (1024^2): interpolation 37 -> 16.6 us,
// spreading 31 -> 17.7 us (event times).
#pragma once

#include "fx.cuh"
#include "kernels.cuh"

namespace dsnu {

// |v| <= 2^54 in halves
__device__ __forceinline__ void fx_split28(i64 v, int& h, int& l) {
  l = int(unsigned(v) << 4) >> 4;
  h = int((v - l) >> 28);
}
__device__ __forceinline__ int4 fx_split28(fxc v) {
  int4 r;
  fx_split28(v.x, r.x, r.y);
  fx_split28(v.y, r.z, r.w);
  return r;
}
// FP64 pair -> 54 bits, relative to exponent field efm: value 2^(kFxBias54 - efm)
constexpr int kFxBias54 = kFxBias - 8;
__device__ __forceinline__ fxc fx_from2(double2 a, int efm) {
  return fx_shr<8>(fx_mk(fx_from_f64(a.x, efm), fx_from_f64(a.y, efm)));
}
__device__ __forceinline__ i64 fx_sum28(i64 p, i64 q) { return p + ((q + (1 << 27)) >> 28); }

// CTA-wide maximum (contains barriers).
__device__ __forceinline__ unsigned fx_cta_top(unsigned m, unsigned* red) {
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  unsigned r = red[0];
  for (int w = 1; w < int(blockDim.x >> 5); ++w) r = max(r, red[w]);
  return r;
}

inline size_t interp_fx_smem(int w) {
  return size_t(kItile + w - 1) * size_t(kItile + w - 1) * 16 + size_t(kItileNodes) * 2 * w * 8;
}

// wts: per node 2 w weights (x then y) as {wh, wl}.  The nodes come in pairs
// k, -k (n_half = n_theta/2 apart) with conjugate transforms of the real density:
// one of each pair is interpolated.
__global__ void __launch_bounds__(256)
k_fx_interp_tile(Members mem, WsOff off, int ldq, int Q, const int2* __restrict__ q0, const int2* __restrict__ wts,
                 const double* __restrict__ D, const int* __restrict__ tile_ptr, const int2* __restrict__ tile_org,
                 const int* __restrict__ tile_nodes, int w, int n_half) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[8];
  const int S = kItile + w - 1, w2 = 2 * w;
  int4* reg = reinterpret_cast<int4*>(smem_raw);            // [dx][dy], S x S
  int2* sw = reinterpret_cast<int2*>(reg + S * S);          // [node of the item][2 w]
  const int2 org = tile_org[blockIdx.x];
  const int n0 = tile_ptr[blockIdx.x], cnt = tile_ptr[blockIdx.x + 1] - n0;
  // eight threads per node, thread h of a node taking the stencil rows b = h and h + 8
  const int s = threadIdx.x >> 3, h = threadIdx.x & 7;
  const bool have = s < cnt;
  const int j = have ? tile_nodes[n0 + s] : 0;
  const int2 b0 = have ? q0[j] : org;
  const double d = have ? D[j] : 0.0;
  for (int i = threadIdx.x; i < cnt * w2; i += 256) {
    const int e = i / w2;
    sw[i] = wts[size_t(tile_nodes[n0 + e]) * w2 + (i - e * w2)];
  }
  grid_dep_wait();
  const Member mb = member_at(mem, blockIdx.y);
  const double2* __restrict__ Bband = ws_ptr<double2>(mb, off.Bband);
  double2* __restrict__ c = ws_ptr<double2>(mb, off.c);
  constexpr int PER = ((kItile + 15) * (kItile + 15) + 255) / 256;
  double2 v[PER];
  unsigned mx = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = threadIdx.x + 256 * k;
    const int dx = i / S, dy = i - dx * S;
    const int qx = org.x + dx, qy = org.y + dy;
    v[k] = make_double2(0.0, 0.0);
    if (i < S * S && qx <= Q && qx >= -Q && qy <= Q && qy >= -Q) {
      v[k] = (qx >= 0) ? Bband[size_t(qx) * ldq + qy + Q] : Bband[size_t(-qx) * ldq + (Q - qy)];
      if (qx < 0) v[k].y = -v[k].y;
      const cpx<double> u = mul_ipow(mk<double>(v[k].x, v[k].y), qx + qy);  // centring phase i^{q_x + q_y}
      v[k] = make_double2(u.x, u.y);
    }
    mx = fx_top(fx_top(mx, v[k].x), v[k].y);
  }
  mx = fx_cta_top(mx, red);
  const int efm = fx_efm(mx);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = threadIdx.x + 256 * k;
    if (i < S * S) reg[i] = fx_split28(fx_from2(v[k], efm));
  }
  __syncthreads();
  i64 px = 0, qx = 0, py = 0, qy = 0;  // the node's sum over this thread's rows
  if (have) {
    const int2* wx = sw + s * w2;
    const int4* rb = reg + (b0.x - org.x) * S + (b0.y - org.y);
    for (int b = h; b < w; b += 8) {
      i64 p = 0, q = 0, r = 0, u = 0;
#pragma unroll 4
      for (int a = 0; a < w; ++a) {
        const int4 x = rb[a * S + b];
        const int2 f = wx[a];
        p = fx_mad(x.x, f.x, p);
        q = fx_mad(x.y, f.x, fx_mad(x.x, f.y, q));
        r = fx_mad(x.z, f.x, r);
        u = fx_mad(x.w, f.x, fx_mad(x.z, f.y, u));
      }
      // the row's sum, back to 54 bits (at most 16 terms)
      const int4 t = fx_split28(fx_shr<4>(fx_mk(fx_sum28(p, q), fx_sum28(r, u))));
      const int2 f = wx[w + b];
      px = fx_mad(t.x, f.x, px);
      qx = fx_mad(t.y, f.x, fx_mad(t.x, f.y, qx));
      py = fx_mad(t.z, f.x, py);
      qy = fx_mad(t.w, f.x, fx_mad(t.z, f.y, qy));
    }
  }
  i64 sx = fx_sum28(px, qx), sy = fx_sum28(py, qy);
#pragma unroll
  for (int i = 1; i < 8; i <<= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, i);
    sy += __shfl_xor_sync(0xffffffffu, sy, i);
  }
  if (have && h == 0) {
    const int ex = efm - kFxBias54 + 4;
    double2 r = make_double2(d * fx_to_f64(sx, ex), d * fx_to_f64(sy, ex));
    if (mx >= kFxInf) r.x = r.y = __longlong_as_double(0x7FF8000000000000ll);
    c[j] = r;
    c[j + n_half] = make_double2(r.x, -r.y);
  }
}

// One work item of a tile: a thread adds up eight cells (one q_x, eight q_y) over
// every 8 SPLIT-th entry of the item, so that c w_x is formed once for eight
// cells; the parts are added through shared memory in a fixed order.
template <int TILE, int SPLIT, int CHUNK>
__global__ void __launch_bounds__(TILE * TILE * SPLIT)
k_fx_spread(Members mem, WsOff off, const int2* __restrict__ item_range, const int* __restrict__ ent_node,
            const int2* __restrict__ ent_q0, const int2* __restrict__ ent_w, const int* __restrict__ item_tile, int w,
            int tiles_x, int Q) {
  constexpr int CELLS = TILE * TILE, THREADS = CELLS * SPLIT, PARTS = 8 * SPLIT;
  static_assert(THREADS >= CHUNK && PARTS >= 8, "one entry per thread");
  union Sm {
    int2 w[CHUNK * 32];
    longlong2 part[PARTS / 2][CELLS];
  };
  __shared__ Sm sm;
  __shared__ int2 s_q0[CHUNK];
  __shared__ int4 s_c[CHUNK];
  __shared__ unsigned red[THREADS / 32];
  const int item = blockIdx.x, tid = threadIdx.x;
  const int2 rg = item_range[item];
  const int s0 = rg.x, cnt = rg.y - rg.x;  // cnt <= CHUNK
  const int w2 = 2 * w;
  const int tile = item_tile[item];
  const int node = (tid < cnt) ? ent_node[s0 + tid] : 0;
  if (tid < cnt) s_q0[tid] = ent_q0[s0 + tid];
  const int2* src = ent_w + size_t(s0) * w2;
  for (int i = tid; i < cnt * w2; i += THREADS) {
    const int e = i / w2;
    sm.w[e * 32 + (i - e * w2)] = src[i];
  }
  grid_dep_wait();
  const Member mb = member_at(mem, blockIdx.y);
  const double2* __restrict__ c = ws_ptr<double2>(mb, off.c);
  double2* __restrict__ partial = ws_ptr<double2>(mb, off.partial);
  const double2 cv = (tid < cnt) ? c[node] : make_double2(0.0, 0.0);
  const unsigned mx = fx_cta_top(fx_top(fx_top(0u, cv.x), cv.y), red);
  const int efm = fx_efm(mx);
  if (tid < cnt) s_c[tid] = fx_split28(fx_from2(cv, efm));
  __syncthreads();
  const int cx = tid & (TILE - 1), r = tid / TILE;
  const int part = r & (PARTS - 1), hb = r / PARTS;  // cells (cx, 8 hb + i)
  const int qx = (tile % tiles_x) * TILE + cx;
  const int qy = (tile / tiles_x) * TILE + 8 * hb - Q;
  i64 px[8], ux[8], py[8], uy[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) px[i] = ux[i] = py[i] = uy[i] = 0;
  for (int k = part; k < cnt; k += PARTS) {
    const int a = qx - s_q0[k].x, b0 = qy - s_q0[k].y;
    if ((unsigned)a < (unsigned)w && b0 > -8 && b0 < w) {
      const int4 cc = s_c[k];
      const int2 f = sm.w[k * 32 + a];
      // c w_x, 54 bits
      const int4 u = fx_split28(fx_mk(fx_sum28(fx_mulw(cc.x, f.x), fx_mad(cc.y, f.x, fx_mulw(cc.x, f.y))),
                                      fx_sum28(fx_mulw(cc.z, f.x), fx_mad(cc.w, f.x, fx_mulw(cc.z, f.y)))));
      const int2* wy = &sm.w[k * 32 + w];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int b = b0 + i;
        if ((unsigned)b < (unsigned)w) {
          const int2 g = wy[b];
          px[i] = fx_mad(u.x, g.x, px[i]);
          ux[i] = fx_mad(u.y, g.x, fx_mad(u.x, g.y, ux[i]));
          py[i] = fx_mad(u.z, g.x, py[i]);
          uy[i] = fx_mad(u.w, g.x, fx_mad(u.z, g.y, uy[i]));
        }
      }
    }
  }
  __syncthreads();  // the weights are read: their memory takes the parts' sums
  // the upper half of the parts first to the lower one's threads (all in one
  // warp: lanes 16 apart hold parts an even distance apart)
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    px[i] = fx_sum28(px[i], ux[i]);
    py[i] = fx_sum28(py[i], uy[i]);
    px[i] += __shfl_xor_sync(0xffffffffu, px[i], 16);
    py[i] += __shfl_xor_sync(0xffffffffu, py[i], 16);
  }
  if ((tid & 16) == 0) {
    constexpr int PW = 32 / TILE;                       // parts per warp (of one hb)
    const int row = (part / PW) * (PW / 2) + (part % PW) % (PW / 2 > 0 ? PW / 2 : 1);
#pragma unroll
    for (int i = 0; i < 8; ++i) sm.part[row][(8 * hb + i) * TILE + cx] = make_longlong2(px[i], py[i]);
  }
  __syncthreads();
  if (tid < CELLS) {
    i64 sx = 0, sy = 0;
#pragma unroll
    for (int p = 0; p < PARTS / 2; ++p) {
      const longlong2 v = sm.part[p][tid];
      sx += v.x;
      sy += v.y;
    }
    const int ex = efm - kFxBias54;
    double2 o = make_double2(fx_to_f64(sx, ex), fx_to_f64(sy, ex));
    if (mx >= kFxInf) o.x = o.y = __longlong_as_double(0x7FF8000000000000ll);
    partial[size_t(item) * CELLS + tid] = o;
  }
}

// Launch the spreading pair with configuration `cfg`, as launch_spread.
inline void launch_spread_fx(int cfg, const Members& mem, const WsOff& off, const PlanTables& t, const PlanGeom& g,
                             int ldq, cudaStream_t st, int part, bool pdl) {
  const int2* ew = static_cast<const int2*>(t.ent_w);
#define DSNU_SPREAD(TL, SP, CH)                                                                                       \
  if (part != 1 && g.n_items > 0)                                                                                     \
    launch_k(pdl, k_fx_spread<TL, SP, CH>, dim3(g.n_items, mem.count), dim3(TL * TL * SP), 0, st, mem, off,           \
             t.item_range, t.ent_node, t.ent_q0, ew, t.item_tile, g.w, g.tiles_x, g.Q);                               \
  if (part != 0)                                                                                                      \
    launch_k(pdl, k_spread_reduce<double, TL>, dim3(g.n_tiles, mem.count), dim3(TL * TL), 0, st, mem, off,            \
             t.tile_items, g.tiles_x, g.n_tiles, g.Q, ldq, 0)
  switch (cfg) {
    case 1: DSNU_SPREAD(8, 2, 128); break;
    case 2: DSNU_SPREAD(16, 1, 128); break;
    case 3: DSNU_SPREAD(16, 2, 64); break;
    default: DSNU_SPREAD(8, 4, 128); break;
  }
#undef DSNU_SPREAD
}

}  // namespace dsnu
