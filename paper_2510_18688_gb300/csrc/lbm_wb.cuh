// lbm_wb.cuh -- phase B of the float step: the macroscopic fields of a node
// and its three collisions on well-balanced populations (kShift), written for
// the fewest instructions, for sm_103a.  Every float grid but the columns
// (is_column, lbm_kernels.cuh) takes it, in the TMA-staged and in the other
// tile kernels alike.
//
// The tile kernels are bound by instruction issue (at 71-77 % of the issue
// slots the 2048 x 1024 porous grid took 108 us against 85 us of HBM time), so
// what counts is instructions per node.  The equations are those of
// node_macros, collide_flow_wb, collide_phase and collide_heat_wb
// (lbm_step.cuh); the forms differ:
//   * quadratic and odd equilibrium and source terms are dot products with
//     vectors scaled once per node, diagonal weights a quarter of the axis ones;
//   * by the magic relation 1/tau_s + 1/tau_a = 2 the enthalpy collision is
//     h_i* = q_i + (1/tau_a - 1) (h_o - q_o), o the opposite of i,
//     q = h_eq + w C T mdot / 2;
//   * one Laplacian for the wetting terms: s_wet holds cos(theta) phi0 +
//     cos(psi) fs;
//   * nodes of a tile inside the grid store at offsets the compiler knows, all
//     others at precomputed neighbour offsets with one wall test a link (one
//     copy of the collisions for each, instead of three).
#pragma once

#include "lbm_kernels.cuh"

namespace lbmk {

// Where the links of a node lead: offsets to its neighbours along each axis
// (wrapped on a periodic axis) and the walls beside it (bit 0 x low, 1 x high,
// 2 y low, 3 y high).  IN: a tile inside the grid, nothing to look up.
template <bool IN>
struct Links {
  int xl, xh, yl, yh;
  unsigned wall;
  __device__ __forceinline__ Links(const Geom& g, int x, int y)
      : xl(-1), xh(1), yl(-g.pitch), yh(g.pitch), wall(0) {
    if (!IN) {
      if (x == 0) {
        if (g.bc[0] == BC_PERIODIC) xl = g.nx - 1; else wall |= 1u;
      }
      if (x == g.nx - 1) {
        if (g.bc[1] == BC_PERIODIC) xh = 1 - g.nx; else wall |= 2u;
      }
      if (y == 0) {
        if (g.bc[2] == BC_PERIODIC) yl = (g.ny - 1) * g.pitch; else wall |= 4u;
      }
      if (y == g.ny - 1) {
        if (g.bc[3] == BC_PERIODIC) yh = (1 - g.ny) * g.pitch; else wall |= 8u;
      }
    }
  }
  __device__ __forceinline__ int to(int i) const {
    return (qx(i) > 0 ? xh : (qx(i) < 0 ? xl : 0)) + (qy(i) > 0 ? yh : (qy(i) < 0 ? yl : 0));
  }
  // walls that direction i crosses
  __device__ __forceinline__ unsigned hit(int i) const {
    return IN ? 0u
              : wall & ((qx(i) > 0 ? 2u : (qx(i) < 0 ? 1u : 0u)) |
                        (qy(i) > 0 ? 8u : (qy(i) < 0 ? 4u : 0u)));
  }
};

// Store of one post-collision population (flow, phase) of direction i.
template <bool IN, typename S>
__device__ __forceinline__ void put(S* __restrict__ plane0, int P, int n, const Links<IN>& k, int i,
                                    float v) {
  if (k.hit(i)) stp(plane0 + qopp(i) * P + n, v);
  else stp(plane0 + i * P + n + k.to(i), v);
}
// Store of an enthalpy remainder, as push_h (lbm_step.cuh).
template <bool IN, typename S>
__device__ __forceinline__ void put_h(const Geom& g, const Coef<float>& c, S* __restrict__ plane0,
                                      int P, int n, const Links<IN>& k, int i, float X,
                                      float ref_old, float wrr, float T_self, float T_dest) {
  const unsigned hit = k.hit(i);
  if (hit == 0u) {
    stp(plane0 + i * P + n + k.to(i), X - ref_delta(ref_hi(wrr, T_dest), ref_old));
  } else {
    const int wall = __ffs((int)hit) - 1;  // the x wall decides at corners
    const float rn = ref_hi(wrr, T_self);
    float v = X - ref_delta(rn, ref_old);
    if (g.bc[wall] == BC_DIRICHLET) {
      const float wTw = ref_hi(wrr, c.T_wall[wall]);
      v = -X + (ref_delta(wTw, ref_old) + ref_delta(wTw, rn));
    }
    stp(plane0 + qopp(i) * P + n, v);
  }
}

// 6 sum_i w_i (v(x + c_i) - v(x)) over an array of row stride s
__device__ __forceinline__ float lap_wb(const float* v, int s) {
  const float c = v[0];
  const float a = ((v[1] - c) + (v[-1] - c)) + ((v[s] - c) + (v[-s] - c));
  const float d = ((v[s + 1] - c) + (v[-s - 1] - c)) + ((v[s - 1] - c) + (v[1 - s] - c));
  return 6.f * fmaf(1.f / 36.f, d, (1.f / 9.f) * a);
}
// 3 sum_i w_i c_i v(x + c_i).  Here and in the odd terms below the factor 3 is
// kept apart from the weights: 3 x float(1/9) is nearer to 1/3 than float(1/3)
// is (7e-9 against 3e-8 relative), and a relative error of the momentum the
// equilibrium carries is the same at every step, so it grows (256 steps of
// the 160 x 160 droplet: velocity 2.5e-6 instead of 8.5e-7 off).
__device__ __forceinline__ void grad_wb(const float* v, int s, float& gx, float& gy) {
  const float d13 = v[1] - v[-1], d24 = v[s] - v[-s];
  const float d57 = v[s + 1] - v[-s - 1], d86 = v[-s + 1] - v[s - 1];
  gx = 3.f * fmaf(1.f / 36.f, d57 + d86, (1.f / 9.f) * d13);
  gy = 3.f * fmaf(1.f / 36.f, d57 - d86, (1.f / 9.f) * d24);
}

struct MacroWb {
  float ux, uy, uu, pr, prl, Ftx, Fty, Gx, Gy, S, fsym0, tauf, mu, phux, phuy;
};

// Velocity, pressure, forces.  cphi, cwet, crho at the node in arrays of row
// stride HX, cp in one of row stride sb.  f: the node's flow populations,
// referred on return to its new pressure (collide_flow_wb's form).
template <bool IN>
__device__ __forceinline__ MacroWb macros_wb(const Coef<float>& c, int lat, const Links<IN>& k,
                                             const Local<float>& L, float phi0, float* f,
                                             const float* cphi, const float* cwet,
                                             const float* crho, const float* cp, int sb) {
  MacroWb M;
  const float phi = L.phi, fs = L.fs, rho = L.rho, pp = cp[0];
  float Fx = rho * c.gx, Fy = rho * c.gy;
  M.mu = 0.f;
  if (lat & LAT_PHASE) {
    float gx, gy;
    grad_wb(cphi, HX, gx, gy);
    const float lap = lap_wb(cphi, HX) + lap_wb(cwet, HX);
    const float v = (phi - 1.f) * (phi + 1.f), v3 = fmaf(3.f, v, 2.f);
    const float q2 = phi0 * phi0, f2 = fs * fs;
    float m = phi * fmaf(c.s9, q2 + f2, c.s3 * v);
    m = fmaf(c.s3 * c.cos_th * phi0, v3 + q2, m);
    m = fmaf(c.s3 * c.cos_ps * fs, v3 + f2, m);
    M.mu = fmaf(-c.klap, lap, m);
    Fx = fmaf(M.mu, gx, Fx);
    Fy = fmaf(M.mu, gy, Fy);
  }
  M.ux = M.uy = M.uu = M.pr = M.prl = 0.f;
  if (lat & LAT_FLOW) {
    float grx, gry, gpx, gpy;
    grad_wb(crho, HX, grx, gry);
    grad_wb(cp, sb, gpx, gpy);
    // moments of the remainders, and of the references 3 w_i p_src(i) as
    // differences from the node's own lagged pressure pp
    float jx = (f[1] - f[3]) + ((f[5] - f[6]) + (f[8] - f[7]));
    float jy = (f[2] - f[4]) + ((f[5] + f[6]) - (f[7] + f[8]));
    float snz = ((f[1] + f[3]) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]));
    float d[9];
#pragma unroll
    for (int i = 1; i < 9; i++) {
      d[i] = cp[-(qy(i) * sb + qx(i))] - pp;
      if (!IN && k.hit(qopp(i))) d[i] = 0.f;  // came back from the node itself
    }
    {
      const float a = d[5] - d[7], b = d[8] - d[6];
      jx = fmaf(3.f, fmaf(1.f / 9.f, d[1] - d[3], (1.f / 36.f) * (a + b)), jx);
      jy = fmaf(3.f, fmaf(1.f / 9.f, d[2] - d[4], (1.f / 36.f) * (a - b)), jy);
      snz = fmaf(3.f, fmaf(1.f / 9.f, (d[1] + d[3]) + (d[2] + d[4]),
                           (1.f / 36.f) * ((d[5] + d[7]) + (d[6] + d[8]))), snz);
    }
    // Eq. (17a,b) rounded once, as node_macros: j + F/2 kept as s + e, the
    // quotient corrected by its exact residual plus e
    const float irho = qdiv(1.f, rho);
    float sx, esx, sy, esy;
    two_sum(jx, 0.5f * Fx, sx, esx);
    two_sum(jy, 0.5f * Fy, sy, esy);
    const float qx_ = sx * irho, qy_ = sy * irho;
    const float qxl = (fmaf(-qx_, rho, sx) + esx) * irho;
    const float qyl = (fmaf(-qy_, rho, sy) + esy) * irho;
    const float h = fmaf(-0.5f, fs, 1.f);
    M.ux = fmaf(qx_, h, qxl * h);
    M.uy = fmaf(qy_, h, qyl * h);
    const float rf = rho * fs;
    M.Gx = fmaf(-rf, qx_ + qxl, Fx);
    M.Gy = fmaf(-rf, qy_ + qyl, Fy);
    M.uu = fmaf(M.uy, M.uy, M.ux * M.ux);
    M.S = fmaf(M.uy, gry, fmaf(M.ux, grx, rho * L.mdot));
    // modified force (reading R-FT), lagged pressure (reading R-FP)
    M.Ftx = fmaf(1.f / 3.f, grx, Fx - gpx);
    M.Fty = fmaf(1.f / 3.f, gry, Fy - gpy);
    M.fsym0 = fmaf(-3.f, fmaf(M.uy, M.Fty, M.ux * M.Ftx), M.S);
    // tau_f = 3 mu / rho + 1/2 rounded once, as node_macros
    const float mu = interp(fs, L.w, c.mu_s, c.mu_l, c.mu_g);
    const float q0 = mu * irho;
    const float qe = fmaf(-q0, rho, mu) * irho;
    const float t1 = 3.f * q0, t1e = fmaf(3.f, q0, -t1);
    float sm, se;
    two_sum(t1, 0.5f, sm, se);
    M.tauf = sm + (se + fmaf(3.f, qe, t1e));
    // Eq. (17c) as an increment of pp, its rounding residual kept
    float F0 = M.fsym0;
    if (c.readings & 1u) F0 -= M.S;
    float t = fmaf(0.5f, M.S, snz);
    t = fmaf((4.f / 9.f) * (M.tauf - 0.5f), F0, t);
    t = fmaf((4.f / 9.f) * -1.5f * rho, M.uu, t);
    // 1 / (3 (1 - w_0)) of the float weights, 0.59999996: the references
    // 3 w_i p hold the same weights, and the pressure is the sum of these
    // increments over the whole run.  With float(3/5), 1e-7 above it, p is
    // 17 % and u 14-16 % further off on porous grids (36 states of 8 to 160
    // steps against the 64-bit solution).
    const float dp = ((1.f / 3.f) / (1.f - 4.f / 9.f)) * t;
    M.pr = pp + dp;
    const float bb = M.pr - pp;
    M.prl = (pp - (M.pr - bb)) + (dp - bb);
    // the populations referred to the new pressure
    f[0] = fmaf(5.f / 3.f, bb, f[0]);
#pragma unroll
    for (int i = 1; i < 9; i++) f[i] = fmaf(i <= 4 ? 3.f / 9.f : 3.f / 36.f, d[i] - bb, f[i]);
  }
  M.phux = phi * M.ux;
  M.phuy = phi * M.uy;
  return M;
}

// Eqs. (11), (14)-(16): out_i = (1 - 1/tau) f_i + even +- odd
template <bool IN, typename S>
__device__ __forceinline__ void flow_wb(const Coef<float>& c, S* __restrict__ out, int P, int n,
                                        const Links<IN>& k, const float* f, float rho,
                                        const MacroWb& M) {
  constexpr float w1 = 1.f / 9.f, kd = 0.25f;
  const float it = qdiv(1.f, M.tauf), om = 1.f - it, fc = fmaf(-0.5f, it, 1.f);
  const float ir = it * rho, p3 = 3.f * it * M.prl;
  const float Kn = fmaf(-1.5f * ir, M.uu, fmaf(fc, M.fsym0, p3));
  float Ka = w1 * Kn, Kd = kd * Ka, K0 = fmaf(4.f / 9.f, Kn, -p3);
  if (c.readings & 1u) {  // variant of the modified force: 3/2 S (c.c - 2/3)
    const float fS = fc * M.S;
    Ka = fmaf(0.5f * w1, fS, Ka);
    Kd = fmaf(2.f * w1 * kd, fS, Kd);
    K0 = fmaf(-4.f / 9.f, fS, K0);
  }
  const float k1 = 3.f * ir, k2 = 3.f * fc, a1 = (1.5f * w1) * k1, b1 = (3.f * w1) * k2;
  const float X = fmaf(a1, M.ux, b1 * M.Ftx), Y = fmaf(a1, M.uy, b1 * M.Fty);
  const float Vx = fmaf(k1, M.ux, k2 * M.Gx), Vy = fmaf(k1, M.uy, k2 * M.Gy);
  put<IN>(out, P, n, k, 0, fmaf(om, f[0], K0));
  auto pair = [&](int i, float even, float w, float odd) {
    put<IN>(out, P, n, k, i, fmaf(w, odd, fmaf(om, f[i], even)));
    put<IN>(out, P, n, k, qopp(i), fmaf(-w, odd, fmaf(om, f[qopp(i)], even)));
  };
  pair(1, fmaf(M.ux, X, Ka), w1, Vx);
  pair(2, fmaf(M.uy, Y, Ka), w1, Vy);
  pair(5, fmaf(kd * (M.ux + M.uy), X + Y, Kd), w1 * kd, Vx + Vy);
  pair(6, fmaf(kd * (M.uy - M.ux), Y - X, Kd), w1 * kd, Vy - Vx);
}

// Eqs. (18)-(20); gq[0] and phir relative to the reader's reference, dref taken
// off the stored rest population
template <bool IN, typename S>
__device__ __forceinline__ void phase_wb(const Coef<float>& c, S* __restrict__ out, int P, int n,
                                         const Links<IN>& k, const float* gq, float phi, float phir,
                                         float mdot, float phuxp, float phuyp, const MacroWb& M,
                                         float dref) {
  constexpr float w1 = 1.f / 9.f, kd = 0.25f;
  const float it = c.inv_tau_g, om = 1.f - it, gc = fmaf(-0.5f, it, 1.f);
  const float em = it * c.eta * M.mu, Zs = fmaf(gc * phi, mdot, em);
  const float Za = w1 * Zs, Zd = kd * Za;
  const float v1 = 3.f * it, v2 = 3.f * gc;
  const float Vx = fmaf(v2, M.phux - phuxp, v1 * M.phux);
  const float Vy = fmaf(v2, M.phuy - phuyp, v1 * M.phuy);
  put<IN>(out, P, n, k, 0,
          fmaf(om, gq[0], fmaf(it, phir, fmaf(4.f / 9.f, Zs, -em))) - dref);
  auto pair = [&](int i, float even, float w, float odd) {
    put<IN>(out, P, n, k, i, fmaf(w, odd, fmaf(om, gq[i], even)));
    put<IN>(out, P, n, k, qopp(i), fmaf(-w, odd, fmaf(om, gq[qopp(i)], even)));
  };
  pair(1, Za, w1, Vx);
  pair(2, Za, w1, Vy);
  pair(5, Zd, w1 * kd, Vx + Vy);
  pair(6, Zd, w1 * kd, Vy - Vx);
}

// Eqs. (23)-(27); CT = rho Cp T, other arguments as collide_heat_wb
template <bool IN, typename S>
__device__ __forceinline__ void heat_wb(const Geom& g, const Coef<float>& c, S* __restrict__ out,
                                        int P, int n, const Links<IN>& k, const float* hr,
                                        const Local<float>& L, float CT, float dT, float e,
                                        const MacroWb& M, float aold, float dold, float dref0,
                                        const float* cT) {
  constexpr float w1 = 1.f / 9.f, kd = 0.25f;
  const float lam = interp(L.fs, L.w, c.lam_s, c.lam_l, c.lam_g);
  const float am = qdiv(1.f, fmaf(lam, c.inv_rr3, 0.5f)) - 1.f;
  const float Kn = fmaf(0.5f * CT, L.mdot, fmaf(-1.5f * CT, M.uu, c.rr * dT));
  const float Ka = w1 * Kn, Kd = kd * Ka;
  const float ya = (4.5f * w1) * CT, za = 3.f * CT;
  {
    // the reference of h0 holds (1 - w_0) rho_ref Cp_ref T' of the others
    const float q0 = fmaf(4.f / 9.f, Kn, fmaf(-c.rr, dT, e));
    stp(out + n, fmaf(am, hr[0] - q0, q0) - dref0);
  }
  auto pair = [&](int i, float even, float w, float odd, float ro, float wrr) {
    const int o = qopp(i);
    const float qi = fmaf(w, odd, even), qo = fmaf(-w, odd, even);
    put_h<IN>(g, c, out, P, n, k, i, fmaf(am, hr[o] - qo, qi), ro, wrr, L.T,
              cT[qy(i) * HX + qx(i)]);
    put_h<IN>(g, c, out, P, n, k, o, fmaf(am, hr[i] - qi, qo), ro, wrr, L.T,
              cT[qy(o) * HX + qx(o)]);
  };
  pair(1, fmaf(ya * M.ux, M.ux, Ka), w1, za * M.ux, aold, c.wrr1);
  pair(2, fmaf(ya * M.uy, M.uy, Ka), w1, za * M.uy, aold, c.wrr1);
  const float up = M.ux + M.uy, um = M.uy - M.ux, yd = kd * ya;
  pair(5, fmaf(yd * up, up, Kd), w1 * kd, za * up, dold, c.wrr5);
  pair(6, fmaf(yd * um, um, Kd), w1 * kd, za * um, dold, c.wrr5);
}

}  // namespace lbmk
