// lbm_column.cuh -- the double-precision step of thin columns (is_column) for
// sm_103a: the arithmetic of step_tile on 32 x 1 tiles with four warps each.
//
// A column has fewer tiles than the chip has SMs, so a step takes as long as
// one tile does: a chain of FP64 latencies.  One warp a tile (step_tile on
// 32 x 1 tiles) runs the chain of its own nodes, then three rounds of its 70
// ring nodes, then the three collisions one after another: 42 us a step of
// 512 x 8, its SM's FP64 pipe a fifth busy.  Here the four warps of a tile
// take what does not depend on each other: warp 0 the own nodes while the
// others take the ring; warp 0 the macroscopic quantities; then warp 0
// collides the flow, warp 1 the phase field, warp 2 the enthalpy, and warp 3
// stores the lags: 19 us (1024 x 24, where the FP64 pipe fills: 78 -> 48).
//
// The bits: the compiler contracts a sum of two products one way or the
// other, depending on the code around it, so every such sum whose order came
// out differently here on a one-dimensional column is written in step_tile's
// order (PIN, sum2): the Neumann and Stefan columns have step_tile's bits.  A
// state that varies across the column may differ from it in the last ones.  A
// step that reduces the sums is compiled to another order in places and stays
// with step_tile, its ring on warps of its own (30 us).
#pragma once

#include "lbm_step.cuh"

namespace lbmk {

constexpr int COL_WARPS = 4;
constexpr int COL_NT = COL_WARPS * TX;
inline dim3 column_dims() { return dim3(TX, COL_WARPS, 1); }

// The step of the 32 x 1 tile (bx, by), tile b of nb; a CTA of TX x COL_WARPS
// threads.
template <int LATC>
__device__ __forceinline__ void column_step(const Args<double>& a, int bx, int by) {
  using R = double;
  constexpr int HN = Shape<1>::HN, RING = Shape<1>::RING;
  static_assert(RING <= (COL_WARPS - 1) * TX, "one ring node a thread of warps 1 to 3");
  const Geom& g = a.g;
  const Coef<R>& c = a.c;
  const int lat = LATC ? LATC : g.lattices;
  const int P = (int)g.plane;
  __shared__ R s_phi[HN], s_fs[HN], s_rho[HN], s_p[HN], s_phi0[HN];
  // what warp 0 hands to the others: the node's state and macroscopic values
  enum { X_T, X_FL, X_MDOT, X_RHOH, X_W, X_UX, X_UY, X_UU, X_PR, X_MUPHI, X_N };
  __shared__ R s_x[X_N][TX];

  const int tx = threadIdx.x, warp = threadIdx.y;
  const int tid = warp * TX + tx;
  const int x0 = bx * TX, y0 = by;
  const int gx = x0 + tx, gy = y0;
  const bool valid = gx < g.nx;
  const int mx = wrap_or_clamp(gx, g.nx, g.bc[0], g.bc[1]);
  const int my = wrap_or_clamp(gy, g.ny, g.bc[2], g.bc[3]);
  const int n = my * g.pitch + mx;
  const int hc = HX + tx + 1;  // the node's cell in the tile with its ring
  const double* pn = a.pin + n;

  // the populations this warp collides: flow (0), phase (1), enthalpy (2);
  // loaded with everything else, before the first barrier
  const R phi0 = a.phi0[n];
  const R wp = a.lin[LAG_W * P + n];
  const bool masked = (lat & LAT_HEAT) && g.has_mask && a.mask[n];
  R q[9];
  R phuxp = R(0), phuyp = R(0);
#pragma unroll
  for (int i = 0; i < 9; i++) q[i] = R(0);
  if (warp == 0) {
    if (lat & LAT_FLOW) {
#pragma unroll
      for (int i = 0; i < 9; i++) q[i] = pn[i * P];
    }
  } else if (warp == 1) {
    if (lat & LAT_PHASE) {
#pragma unroll
      for (int i = 0; i < 9; i++) q[i] = pn[(9 + i) * P];
      phuxp = a.lin[LAG_PHUX * P + n];
      phuyp = a.lin[LAG_PHUY * P + n];
    }
  } else if (warp == 2 && (lat & LAT_HEAT) && !masked) {
#pragma unroll
    for (int i = 0; i < 9; i++) q[i] = pn[(18 + i) * P];
  }

  // ---- phase A: own nodes (warp 0) and ring (warps 1 to 3) -------------------
  Local<R> L;
  R pp = R(0);
  if (warp == 0) {
    const R flp = a.lin[LAG_FL * P + n];
    const R Qp = a.lin[LAG_Q * P + n];
    pp = a.lin[LAG_P * P + n];
    R sg = R(0), sh = R(0);
    if (lat & LAT_PHASE) {
      R v[9];
#pragma unroll
      for (int i = 0; i < 9; i++) v[i] = pn[(9 + i) * P];
      sg = sum_g(v);
    }
    if (lat & LAT_HEAT) {
      R v[9];
      if (masked) {
        cold_mask_h(c, wp, phi0, v);
      } else {
#pragma unroll
        for (int i = 0; i < 9; i++) v[i] = pn[(18 + i) * P];
      }
      sh = sum_h(v);
    }
    L = local_state(c, lat, sg, sh, flp, wp, Qp, phi0);
    s_phi[hc] = L.phi;
    s_fs[hc] = L.fs;
    s_rho[hc] = L.rho;
    s_p[hc] = pp;
    s_phi0[hc] = phi0;
  } else if (tid - TX < RING) {
    int hx, hy;
    ring_pos<1>(tid - TX, hx, hy);
    const int rx = wrap_or_clamp(x0 + hx - 1, g.nx, g.bc[0], g.bc[1]);
    const int ry = wrap_or_clamp(y0 + hy - 1, g.ny, g.bc[2], g.bc[3]);
    const int m = ry * g.pitch + rx;
    const bool rmask = g.has_mask && a.mask[m];
    const double* pm = a.pin + m;
    const R q0 = a.phi0[m];
    const R wq = a.lin[LAG_W * P + m], flq = a.lin[LAG_FL * P + m], Qq = a.lin[LAG_Q * P + m];
    const R pq = a.lin[LAG_P * P + m];
    // the sums in step_tile's order (thirds of a ring node's populations)
    R sgq = R(0), shq = R(0);
    if (lat & LAT_PHASE) {
      R v[9];
#pragma unroll
      for (int i = 0; i < 9; i++) v[i] = pm[(9 + i) * P];
      sgq = (v[0] + v[1] + v[2] + v[3] + v[4] + v[5]) + (v[6] + v[7] + v[8]);
    }
    if (lat & LAT_HEAT) {
      R v[9];
      if (rmask) {
        cold_mask_h(c, wq, q0, v);
        shq = sum_h(v);
      } else {
#pragma unroll
        for (int i = 0; i < 9; i++) v[i] = pm[(18 + i) * P];
        shq = (v[0] + v[1] + v[2]) + (v[3] + v[4] + v[5] + v[6] + v[7] + v[8]);
      }
    }
    const Local<R> Lq = local_state(c, lat, sgq, shq, flq, wq, Qq, q0);
    const int hi = hy * HX + hx;
    s_phi[hi] = Lq.phi;
    s_fs[hi] = Lq.fs;
    s_rho[hi] = Lq.rho;
    s_p[hi] = pq;
    s_phi0[hi] = q0;
  }
  __syncthreads();

  // ---- phase B1: stencils and macroscopic quantities (warp 0) ----------------
  const int yb = y0 / 8 * 8;  // the 32 x 8 tile that step_tile chooses its copy by
  const bool in_tile = x0 >= 1 && x0 + TX < g.nx && yb >= 1 && yb + 8 < g.ny;
  const bool inner = gx > 0 && gx < g.nx - 1 && gy > 0 && gy < g.ny - 1;
  Macro<R> M;
  if (warp == 0) {
    if (valid)
      node_macros<R, false, true>(g, c, lat, gx, gy, inner, L, phi0, pp, q, s_phi + hc, s_fs + hc,
                            s_rho + hc, HX, s_p + hc, s_phi0 + hc, HX, M);
    s_x[X_T][tx] = L.T;
    s_x[X_FL][tx] = L.fl;
    s_x[X_MDOT][tx] = L.mdot;
    s_x[X_RHOH][tx] = L.rhoH;
    s_x[X_W][tx] = L.w;
    s_x[X_UX][tx] = M.ux;
    s_x[X_UY][tx] = M.uy;
    s_x[X_UU][tx] = M.uu;
    s_x[X_PR][tx] = M.pr;
    s_x[X_MUPHI][tx] = M.muphi;
  }
  __syncthreads();
  allow_next();

  // ---- phase B2: the collisions, sums and lags, a warp each ------------------
  if (warp != 0) {
    L.T = s_x[X_T][tx];
    L.fl = s_x[X_FL][tx];
    L.mdot = s_x[X_MDOT][tx];
    L.rhoH = L.rhoHr = s_x[X_RHOH][tx];
    L.w = s_x[X_W][tx];
    L.phi = L.phir = s_phi[hc];
    L.fs = s_fs[hc];
    L.rho = s_rho[hc];
    M.ux = s_x[X_UX][tx];
    M.uy = s_x[X_UY][tx];
    M.uu = s_x[X_UU][tx];
    M.pr = s_x[X_PR][tx];
    M.muphi = s_x[X_MUPHI][tx];
    // products, formed again so that they contract with the sums they enter
    // as in step_tile
    M.phux = L.phi * M.ux;
    M.phuy = L.phi * M.uy;
    M.cap = L.rho * interp(L.fs, L.w, c.cp_s, c.cp_l, c.cp_g);
  }
  double* out = a.pout;
  if (warp == 0) {
    if (valid && (lat & LAT_FLOW)) {
      if (inner) collide_flow<R, true, true>(g, c, out, P, gx, gy, n, q, L.rho, M, in_tile);
      else collide_flow<R, false, true>(g, c, out, P, gx, gy, n, q, L.rho, M);
    }
  } else if (warp == 1) {
    if (valid && (lat & LAT_PHASE)) {
      if (inner)
        collide_phase<R, true>(g, c, out + 9 * P, P, gx, gy, n, q, L.phi, L.phir, L.mdot, phuxp,
                               phuyp, M, R(0));
      else
        collide_phase<R, false>(g, c, out + 9 * P, P, gx, gy, n, q, L.phi, L.phir, L.mdot, phuxp,
                                phuyp, M, R(0));
    }
  } else if (warp == 2) {
    if (valid && (lat & LAT_HEAT)) {
      if (masked) cold_mask_h(c, wp, phi0, q);
      if (inner)
        collide_heat<R, true>(g, c, out + 18 * P, P, gx, gy, n, q, L.fs, L.w, L.T, L.rhoHr,
                              L.mdot, M, R(0));
      else
        collide_heat<R, false>(g, c, out + 18 * P, P, gx, gy, n, q, L.fs, L.w, L.T, L.rhoHr,
                               L.mdot, M, R(0));
    }
  } else {
    if (valid) {
      a.lout[LAG_FL * P + n] = L.fl;
      a.lout[LAG_W * P + n] = L.w;
      a.lout[LAG_P * P + n] = (lat & LAT_FLOW) ? M.pr : R(0);
      a.lout[LAG_PHUX * P + n] = (lat & LAT_PHASE) ? M.phux : R(0);
      a.lout[LAG_PHUY * P + n] = (lat & LAT_PHASE) ? M.phuy : R(0);
      a.lout[LAG_Q * P + n] = (lat & LAT_HEAT) ? M.cap * L.T * L.mdot : R(0);
    }
  }
}

template <int LATC>
__global__ void __launch_bounds__(COL_NT) lbm_column_kernel(const Args<double> a) {
  after_previous();
  column_step<LATC>(a, blockIdx.x, blockIdx.y);
}

// Columns of a double batch in one launch: CTA t takes tile t of the
// concatenated tile list, as lbm_batch_kernel.
template <int LATC>
__global__ void __launch_bounds__(COL_NT)
    lbm_column_batch_kernel(const __grid_constant__ BatchTable<double> B) {
  after_previous();
  const int t = blockIdx.x;
  int lo = 0, hi = B.ngrids;  // tile_base[lo] <= t < tile_base[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (B.tile_base[mid] <= t) lo = mid;
    else hi = mid;
  }
  const Args<double>& a = B.args[lo];
  const int local = t - B.tile_base[lo];
  const int tiles_x = (a.g.nx + TX - 1) / TX;
  column_step<LATC>(a, local % tiles_x, local / tiles_x);
}

}  // namespace lbmk
