// lbm_adjoint_full.cuh -- reverse mode of the whole coupled step (flow,
// phase field and enthalpy lattices; FP64; readings == 0), one thread per
// node on the node step's own planes and stencils (lbm_node.cuh).
//
// On top of the freezing coupling of the phase-field and enthalpy adjoint
// (lbm_adjoint.cuh), the flow lattice moves: the velocity of Eq. (17a,b)
// from the flow populations, the surface-tension and body forces and the
// penalty force; the source S = rho mdot + u . grad rho and the modified
// force F~ = F - grad(p_prev - rho / 3) of Eq. (16); the pressure of
// Eq. (17c); the flow collision Eqs. (11), (14)-(16); phi u in the phase
// equilibrium and source (Eqs. (19)-(20), with its lagged value); u in the
// enthalpy equilibrium (Eq. (25)).  Four stencils are transposed: the
// Laplacian of chi = phi + cos(theta) phi0 + cos(psi) fs (through mu_phi,
// Eq. (6)) and the gradients of phi (F_s), rho (S) and pi = p_prev - rho / 3
// (F~).
//
// Per reverse step: node_local on the recomputed state (its planes phi, chi,
// rho, T, rho H, mdot, fl, w); rev_collide, the reverse of node_collide
// at each node, which stores the adjoints of its stencils (mu_phi and three
// gradients), of its local state, and the direct adjoints of its
// populations; rev_local, which gathers the neighbours' stencil adjoints in
// a fixed order and runs the local chain back to this state's populations
// and lags (fl, w, p, phi u, Q).  Like the step, this is bound by the number
// of FP64 instructions: the quadratic and odd parts of all three collisions
// reverse through one symmetric matrix and one vector per lattice, and the
// local reverse is evaluated once (its seven adjoints and the direct
// population adjoints, 43 planes written and 25 read back from L2, replace a
// second evaluation that took most of the former sweep).
// A cold-mask node reads its enthalpy populations as the equilibrium at
// T_cold (R-BC) built from its lagged w, so their adjoint goes to the lagged
// w, to T_cold and to L instead of to the stored populations.
// Accumulator planes: d/dT_wall[0..3], d/dL, d/dtheta_deg, d/dsigma, d/dgx,
// d/dgy, d/dT_cold.
#pragma once

#include "lbm_adjoint.cuh"
#include "lbm_node.cuh"

namespace lbmn {

constexpr int FULL_NACC = 10;
// Two-warp blocks: the FP64 work of a 256 x 256 grid divides over 152 SMs to
// within a twelfth (four-warp blocks: a fifth).
constexpr int REV_NT = 64;
// adjoints of the stencils, and of the local state
enum { SB_MU = 0, SB_GPHI, SB_GRHO = 3, SB_GP = 5, NSB = 7 };
enum { OWN_PHI = 0, OWN_FS, OWN_W, OWN_RHO, OWN_MDOT, OWN_T, OWN_RHOH, NOWN };

struct RevArgs {
  NodeArgs<double, 2> f;        // the state (pin, lin), its sc planes; lout holds its fl and w
  const double* __restrict__ lam_in;   // 27 planes: adjoints of the next f, g, h
  const double* __restrict__ llag_in;  // lag planes: adjoints of the next state's lags
  double* lam_out;              // 27 planes
  double* __restrict__ llag_out;
  double* sb;                   // NSB planes
  double* own;                  // NOWN planes
  const double* __restrict__ phib_seed;  // crossing seed, or null
  double* __restrict__ acc;     // FULL_NACC planes (+=)
  double dcos_dtheta, inv_sigma;
  double inv_sum_w, ff;         // frozen-fraction seed
  int axis, index;              // crossing seed
  double* __restrict__ out;
};

#ifdef LBM_ADJOINT_KERNELS

// Moments of one lattice's pulled adjoints: with S = A + B and D = A - B of
// a pair (A of direction c, B of its opposite), sum = sum_axes S + kd
// sum_diagonals S, m = sum S c c^T and d = sum D c in the same weighting.
struct PairMoments {
  double sum, mxx, mxy, myy, dx, dy;
  __device__ __forceinline__ explicit PairMoments(const double* b) {
    constexpr double kd = Lat<2>::kd;
    const double s1 = b[1] + b[3], s2 = b[2] + b[4], s5 = b[5] + b[7], s6 = b[6] + b[8];
    const double d1 = b[1] - b[3], d2 = b[2] - b[4], d5 = b[5] - b[7], d6 = b[6] - b[8];
    const double sd = kd * (s5 + s6);
    mxx = s1 + sd;
    myy = s2 + sd;
    sum = mxx + s2;
    mxy = kd * (s5 - s6);
    dx = fma(kd, d5 - d6, d1);
    dy = fma(kd, d5 + d6, d2);
  }
};

// Reverse of node_collide at node id.
static __global__ void __launch_bounds__(REV_NT, 6) rev_collide_kernel(const RevArgs a) {
  constexpr double w0 = Lat<2>::w0, w1 = Lat<2>::w1;
  using G_ = Lag<2>;
  const NodeGeom<2>& g = a.f.g;
  const NodeCoef<double, 2>& c = a.f.c;
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= g.nodes) return;
  lbmk::after_previous();
  const int P = (int)g.plane;
  const Pos<2> pos = node_pos<2>(g, id);
  const int n = pos.n;
  const Nbr<2> nb = neighbours<2>(g, pos);

  // ---- forward values, as node_collide forms them ------------------------------
  const double* sc = a.f.sc + n;
  const double phi = sc[SC_PHI * P], rho = sc[SC_RHO * P], T = sc[SC_T * P];
  const double mdot = sc[SC_MDOT * P], rhoH = sc[SC_RHOH * P];
  const double fl = a.f.lout[G_::FL * P + n], w = a.f.lout[G_::W * P + n];
  const double phi0 = a.f.phi0[n];
  const double fs = min1(fma(w, 1.0 - fl, phi0));
  const Mix<double> mix(fs, w);
  double gph[2], gr[2], gp[2];
  gradient<double, 2>(sc + SC_PHI * P, nb, gph);
  gradient<double, 2>(sc + SC_RHO * P, nb, gr);
  gradient<double, 2>(a.f.lin + G_::P * P + n, nb, gp);
  const double lap = laplacian<double, 2>(sc + SC_CHI * P, sc[SC_CHI * P], nb);
  const double v3 = fma(3.0, (phi - 1.0) * (phi + 1.0), 2.0);
  const double q2 = phi0 * phi0, f2 = fs * fs;
  const double chem_cos = phi0 * (v3 + q2);  // times s3: d mu / d cos theta
  double mu = phi * fma(f2 + q2, c.s9, (phi - 1.0) * (phi + 1.0) * c.s3);
  mu = fma(c.s3ct, chem_cos, mu);
  mu = fma(fs * c.s3cp, v3 + f2, mu);
  mu = fma(lap, -c.klap, mu);
  double f[9];
#pragma unroll
  for (int i = 0; i < 9; i++) f[i] = a.f.pin[i * P + n];
  double j[2];
  {
    const double d1 = f[1] - f[3], d2 = f[2] - f[4], d5 = f[5] - f[7], d6 = f[6] - f[8];
    j[0] = d1 + (d5 - d6);
    j[1] = d2 + (d5 + d6);
  }
  const double irho = rcp(rho), half = fma(fs, -0.5, 1.0), rf = rho * fs;
  double F[2], us[2], u[2], Gf[2], Ft[2];
#pragma unroll
  for (int k = 0; k < 2; k++) {
    F[k] = fma(mu, gph[k], rho * c.g[k]);
    us[k] = fma(F[k], 0.5, j[k]) * irho;
    u[k] = us[k] * half;
    Gf[k] = fma(-rf, us[k], F[k]);
    Ft[k] = fma(gr[k], 1.0 / 3.0, F[k] - gp[k]);
  }
  const double uu = fma(u[1], u[1], u[0] * u[0]);
  const double uFt = fma(u[1], Ft[1], u[0] * Ft[0]);
  const double S = fma(u[1], gr[1], fma(u[0], gr[0], rho * mdot));
  const double fsym0 = fma(uFt, -3.0, S);
  const double tm = mix(c.mu) * irho * 3.0;
  const double itau = rcp(tm + 0.5);

  // ---- pulled adjoints ------------------------------------------------------------
  double fb[9], gb[9], hb[9];
  double dTw[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 9; i++) {
    const unsigned hit = i ? (nb.wall & crossing<2>(i)) : 0u;
    if (hit == 0u) {
      const int t = n + toward<2>(nb, i);
      fb[i] = a.lam_in[i * P + t];
      gb[i] = a.lam_in[(9 + i) * P + t];
      hb[i] = a.lam_in[(18 + i) * P + t];
    } else {
      const int o = Lat<2>::opp(i), side = __ffs((int)hit) - 1;
      fb[i] = a.lam_in[o * P + n];
      gb[i] = a.lam_in[(9 + o) * P + n];
      const double lb = a.lam_in[(18 + o) * P + n];
      hb[i] = lb;
      if (g.bc[side] == BC_DIRICHLET) {
        hb[i] = -lb;
        const double t = lb * (2.0 * (i <= 4 ? w1 : w1 * Lat<2>::kd)) * c.rr;
#pragma unroll
        for (int k = 0; k < 4; k++)
          if (k == side) dTw[k] += t;
      }
    }
  }

  double ub[2], uub, rhob, mdotb, phib, fsb, mub, prb = a.llag_in[G_::P * P + n];
  double Ftb[2], Gb[2], itaub, fsym0b;
  double phub[2] = {a.llag_in[G_::PHU * P + n], a.llag_in[(G_::PHU + 1) * P + n]};
  double* lam = a.lam_out + n;

  // ---- flow collision: out_i = omi f_i + P_s +- P_a --------------------------------
  const double omi = 1.0 - itau;
  {
    const double fco = fma(itau, -0.5, 1.0), ir = itau * rho;
    const double k1 = ir * (3.0 * w1), k2 = fco * (3.0 * w1), a1 = 1.5 * k1, b1 = 3.0 * k2;
    const PairMoments m(fb);
    const double X0 = fma(a1, u[0], b1 * Ft[0]), X1 = fma(a1, u[1], b1 * Ft[1]);
    const double Xb0 = fma(m.mxy, u[1], m.mxx * u[0]), Xb1 = fma(m.myy, u[1], m.mxy * u[0]);
    ub[0] = fma(m.mxy, X1, m.mxx * X0);
    ub[1] = fma(m.myy, X1, m.mxy * X0);
    // X = a1 u + b1 Ft, V = k1 u + k2 G
    ub[0] = fma(a1, Xb0, fma(k1, m.dx, ub[0]));
    ub[1] = fma(a1, Xb1, fma(k1, m.dy, ub[1]));
    Ftb[0] = b1 * Xb0;
    Ftb[1] = b1 * Xb1;
    Gb[0] = k2 * m.dx;
    Gb[1] = k2 * m.dy;
    const double k1b = fma(1.5, fma(Xb1, u[1], Xb0 * u[0]), fma(m.dy, u[1], m.dx * u[0]));
    const double k2b = fma(3.0, fma(Xb1, Ft[1], Xb0 * Ft[0]), fma(m.dy, Gf[1], m.dx * Gf[0]));
    // K = 3 p / tau - 3/2 rho uu / tau + fco (S - 3 u.Ft)
    const double Kb = fma(w1, m.sum, w0 * fb[0]), p3b = Kb - fb[0];
    const double irb = fma(uu * -1.5, Kb, (3.0 * w1) * k1b);
    const double fcob = fma(fsym0, Kb, (3.0 * w1) * k2b);
    uub = ir * -1.5 * Kb;
    fsym0b = fco * Kb;
    rhob = itau * irb;
    double omib = fb[0] * f[0];
#pragma unroll
    for (int i = 1; i < 9; i++) omib = fma(fb[i], f[i], omib);
    // Eq. (17c) of the forward step gives p
    double t = fma(S, 0.5, (((f[1] + f[3]) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8]))));
    t = fma(tm * w0, fsym0, t);
    t = fma(rho * (-1.5 * w0), uu, t);
    const double pr = t * (1.0 / (3.0 * (1.0 - w0)));
    itaub = fma(rho, irb, fma(pr * 3.0, p3b, -omib)) - 0.5 * fcob;
    prb = fma(itau * 3.0, p3b, prb);
  }
  // ---- phase collision ---------------------------------------------------------------
  {
    const PairMoments m(gb);
    const double Zb = fma(w1, m.sum, w0 * gb[0]);
    mub = c.itg_eta * (Zb - gb[0]);
    const double sb = c.gcoef * Zb;
    phib = fma(mdot, sb, c.itg * gb[0]);
    mdotb = phi * sb;
    phub[0] = fma(c.v_new, m.dx, phub[0]);
    phub[1] = fma(c.v_new, m.dy, phub[1]);
    a.llag_out[G_::PHU * P + n] = -c.v_old * m.dx;
    a.llag_out[(G_::PHU + 1) * P + n] = -c.v_old * m.dy;
#pragma unroll
    for (int i = 0; i < 9; i++) lam[(9 + i) * P] = c.omg * gb[i];
  }
  // ---- enthalpy collision: h_i* = (1/tau_a - 1) h_opp + E --------------------------
  double Tb, rhoHb, iab, Cb;
  const double cp = mix(c.cp);
  {
    double h[9];
    if (g.has_mask && a.f.mask[n]) {
      cold_node<2>(c, a.f.lin[G_::W * P + n], phi0, h);
    } else {
#pragma unroll
      for (int i = 0; i < 9; i++) h[i] = a.f.pin[(18 + i) * P + n];
    }
    const double ia = rcp(fma(mix(c.lam), c.inv_rr3, 0.5));
    const double is = 2.0 - ia, am = ia - 1.0;
    const double CT = rho * cp * T, rrT = T * c.rr;
    const PairMoments m(hb);
    double amb = hb[0] * h[0];
#pragma unroll
    for (int i = 1; i < 9; i++) amb = fma(hb[i], h[Lat<2>::opp(i)], amb);
    const double Kb = fma(w1, m.sum, w0 * hb[0]);
    const double Mu0 = fma(m.mxy, u[1], m.mxx * u[0]), Mu1 = fma(m.myy, u[1], m.mxy * u[0]);
    const double yb = (4.5 * w1) * fma(Mu1, u[1], Mu0 * u[0]);
    const double zb = (3.0 * w1) * fma(m.dy, u[1], m.dx * u[0]);
    const double ya2 = is * CT * (9.0 * w1), za = ia * CT * (3.0 * w1);
    ub[0] = fma(ya2, Mu0, fma(za, m.dx, ub[0]));
    ub[1] = fma(ya2, Mu1, fma(za, m.dy, ub[1]));
    const double q15 = fma(uu * -1.5, Kb, yb);
    const double isb = fma(CT, q15, fma(rrT, Kb, (rhoH - rrT) * hb[0]));
    double CTb = fma(is, q15, ia * zb);
    uub = fma(is * CT * -1.5, Kb, uub);
    iab = fma(CT, zb, amb) - isb;
    rhoHb = is * hb[0];
    const double rrTb = fma(is, Kb, -rhoHb);
    // source (1 - 1/(2 tau_a)) C T mdot, and the lag Q = C T mdot
    iab = fma(CT * mdot * -0.5, Kb, iab);
    const double CTmb = fma(fma(ia, -0.5, 1.0), Kb, a.llag_in[G_::Q * P + n]);
    CTb = fma(mdot, CTmb, CTb);
    mdotb = fma(CT, CTmb, mdotb);
    Tb = fma(c.rr, rrTb, rho * cp * CTb);
    Cb = T * CTb;
    iab = -iab * ia * ia * c.inv_rr3;  // adjoint of lambda
    lam[18 * P] = am * hb[0];
#pragma unroll
    for (int i = 1; i < 9; i++) lam[(18 + i) * P] = am * hb[Lat<2>::opp(i)];
  }
  lbmk::allow_next();
  // ---- pressure Eq. (17c), tau_f, forces, velocity ------------------------------------
  {
    const double pk = prb * (1.0 / (3.0 * (1.0 - w0)));  // adjoint of sum_{i>0} f_i
    double Sb = 0.5 * pk;
    double tmb = fma(w0 * fsym0, pk, -(itaub * itau) * itau);
    fsym0b = fma(w0 * tm, pk, fsym0b);
    rhob = fma(uu * (-1.5 * w0), pk, rhob);
    uub = fma(rho * (-1.5 * w0), pk, uub);
    Sb += fsym0b;
    const double uFtb = -3.0 * fsym0b;
    // tau_f - 1/2 = 3 mu / rho
    const double muvb = 3.0 * irho * tmb;
    rhob = fma(-irho * tm, tmb, rhob);
    rhob = fma(cp, Cb, rhob);
    // lambda, Cp and mu of Eq. (10), collected by phase
    const double cpb = rho * Cb;
    const double ps = fma(iab, c.lam[0], fma(cpb, c.cp[0], muvb * c.mu[0]));
    const double pl = fma(iab, c.lam[1], fma(cpb, c.cp[1], muvb * c.mu[1]));
    const double pg = fma(iab, c.lam[2], fma(cpb, c.cp[2], muvb * c.mu[2]));
    fsb = ps - pg - w * (pl - pg);
    double wb = (1.0 - fs) * (pl - pg);
    wb += a.llag_in[G_::W * P + n];
    rhob = fma(mdot, Sb, rhob);
    mdotb = fma(rho, Sb, mdotb);
    double jb[2], rfb = 0.0, hfb = 0.0, ucb = 0.0;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      phib = fma(phub[k], u[k], phib);
      double b = fma(phi, phub[k], ub[k]);
      b = fma(uFtb, Ft[k], b);
      b = fma(Sb, gr[k], b);
      b = fma(2.0 * uub, u[k], b);
      const double ftb = fma(uFtb, u[k], Ftb[k]);
      a.sb[(SB_GRHO + k) * P + n] = fma(ftb, 1.0 / 3.0, Sb * u[k]);
      a.sb[(SB_GP + k) * P + n] = -ftb;
      // u = half us, G = F - rf us, us = (j + F / 2) / rho
      hfb = fma(b, us[k], hfb);
      rfb = fma(Gb[k], us[k], rfb);
      const double usb = fma(half, b, -rf * Gb[k]);
      ucb = fma(usb, us[k], ucb);
      jb[k] = usb * irho;
      const double Fb = fma(0.5, jb[k], ftb + Gb[k]);
      mub = fma(Fb, gph[k], mub);
      a.sb[(SB_GPHI + k) * P + n] = mu * Fb;
      rhob = fma(Fb, c.g[k], rhob);
      a.acc[(7 + k) * P + n] += Fb * rho;
    }
    fsb = fma(-0.5, hfb, fsb);
    fsb = fma(-rho, rfb, fsb);
    rhob = fma(-fs, rfb, rhob);
    rhob = fma(-irho, ucb, rhob);
    const double jd = jb[0] + jb[1], je = jb[1] - jb[0];
    lam[0] = omi * fb[0];
    lam[1 * P] = fma(omi, fb[1], pk + jb[0]);
    lam[2 * P] = fma(omi, fb[2], pk + jb[1]);
    lam[3 * P] = fma(omi, fb[3], pk - jb[0]);
    lam[4 * P] = fma(omi, fb[4], pk - jb[1]);
    lam[5 * P] = fma(omi, fb[5], pk + jd);
    lam[6 * P] = fma(omi, fb[6], pk + je);
    lam[7 * P] = fma(omi, fb[7], pk - jd);
    lam[8 * P] = fma(omi, fb[8], pk - je);
    double* own = a.own + n;
    own[OWN_PHI * P] = phib;
    own[OWN_FS * P] = fsb;
    own[OWN_W * P] = wb;
    own[OWN_RHO * P] = rhob;
    own[OWN_MDOT * P] = mdotb;
    own[OWN_T * P] = Tb;
    own[OWN_RHOH * P] = rhoHb;
    a.sb[SB_MU * P + n] = mub;
  }
  const double lphi0 = laplacian<double, 2>(a.f.phi0 + n, phi0, nb);
  a.acc[5 * P + n] += mub * fma(-c.klap, lphi0, c.s3 * chem_cos) * a.dcos_dtheta;
  a.acc[6 * P + n] += mub * mu * a.inv_sigma;
  if (nb.wall) {
#pragma unroll
    for (int k = 0; k < 4; k++)
      if (dTw[k] != 0.0) a.acc[k * P + n] += dTw[k];
  }
}

// d(rho Cp) / dfs and / dw of Eq. (10)
__device__ __forceinline__ void cap_slopes(const NodeCoef<double, 2>& c, double fs, double w,
                                           double rho, double cp, double* dfs, double* dw) {
  const double rl = c.rho[1] - c.rho[2], cl = c.cp[1] - c.cp[2];
  *dfs = (c.rho[0] - fma(w, rl, c.rho[2])) * cp + rho * (c.cp[0] - fma(w, cl, c.cp[2]));
  *dw = (1.0 - fs) * fma(rl, cp, rho * cl);
}

// Reverse of the local state at node id: the gathered transposes of the
// neighbours' stencils, then fs -> w -> phi -> (sum g, mdot) -> inversion ->
// (sum h, lagged fl, w, Q).
static __global__ void __launch_bounds__(REV_NT, 8) rev_local_kernel(const RevArgs a) {
  constexpr double w0 = Lat<2>::w0, w1 = Lat<2>::w1, kd = Lat<2>::kd;
  using G_ = Lag<2>;
  const NodeGeom<2>& g = a.f.g;
  const NodeCoef<double, 2>& c = a.f.c;
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= g.nodes) return;
  lbmk::after_previous();
  const int P = (int)g.plane;
  const Pos<2> pos = node_pos<2>(g, id);
  const int n = pos.n;
  const Nbr<2> nb = neighbours<2>(g, pos);
  const double* sb = a.sb + n;
  const double mub = sb[SB_MU * P];
  // Transposed Laplacian (without its centre) and gradients.  Node n - c_i
  // takes this one with weight w_i, so the transpose of the gradient is minus
  // the divergence on the same stencil.  Beyond a wall the ghost mirrors the
  // wall node: its own direction -c_i leads back here, so it enters with the
  // normal component reversed.
  double lsum, gsum[3];
  {
    int to[9];
#pragma unroll
    for (int i = 1; i < 9; i++) to[i] = toward<2>(nb, i);
    const double* m = sb + SB_MU * P;
    lsum = (6.0 * w1) * fma(kd, (m[to[5]] + m[to[7]]) + (m[to[6]] + m[to[8]]),
                            (m[to[1]] + m[to[3]]) + (m[to[2]] + m[to[4]]));
    const unsigned flip[4] = {(nb.wall & 1u) << 31, (nb.wall & 2u) << 30, (nb.wall & 4u) << 29,
                              (nb.wall & 8u) << 28};  // sign bits: x low, x high, y low, y high
    auto at = [](double v, unsigned sign) {
      return __hiloint2double(__double2hiint(v) ^ (int)sign, __double2loint(v));
    };
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const double* px = sb + (SB_GPHI + 2 * q) * P;
      const double* py = px + P;
      const double da = (at(px[to[1]], flip[1]) - at(px[to[3]], flip[0])) +
                        (at(py[to[2]], flip[3]) - at(py[to[4]], flip[2]));
      // c . (G(n + c) - G(n - c)) for c = (1, 1) and c = (-1, 1)
      const double d5 = (at(px[to[5]], flip[1]) + at(py[to[5]], flip[3])) -
                        (at(px[to[7]], flip[0]) + at(py[to[7]], flip[2]));
      const double d6 = (at(py[to[6]], flip[3]) - at(px[to[6]], flip[0])) -
                        (at(py[to[8]], flip[2]) - at(px[to[8]], flip[1]));
      gsum[q] = (-3.0 * w1) * fma(kd, d5 + d6, da);
    }
  }

  const double* sc = a.f.sc + n;
  const double phi = sc[SC_PHI * P], mdot = sc[SC_MDOT * P], rhoH = sc[SC_RHOH * P];
  const double T = sc[SC_T * P];
  const double fl = a.f.lout[G_::FL * P + n], w = a.f.lout[G_::W * P + n];
  const double phi0 = a.f.phi0[n];
  const double wp = a.f.lin[G_::W * P + n], flp = a.f.lin[G_::FL * P + n];
  const double* own = a.own + n;
  double phib = own[OWN_PHI * P] + gsum[0], fsb = own[OWN_FS * P], wb = own[OWN_W * P];
  double rhob = own[OWN_RHO * P] + gsum[1], mdotb = own[OWN_MDOT * P];
  double rhoHb = own[OWN_RHOH * P], flb = a.llag_in[G_::FL * P + n];
  const double Tb = own[OWN_T * P];
  if (a.phib_seed) phib += a.phib_seed[n];
  a.llag_out[G_::P * P + n] = gsum[2];
  const double raw = fma(w, 1.0 - fl, phi0), fs = min1(raw);
  {
    // mu_phi: local part of Eq. (6), and chi through the Laplacian
    const double v3 = fma(3.0, (phi - 1.0) * (phi + 1.0), 2.0), f2 = fs * fs;
    const double dphi = fma(6.0 * phi, fma(c.s3ct, phi0, c.s3cp * fs),
                            fma(c.s3, v3, c.s9 * fma(phi0, phi0, f2)));
    const double dfs = fma(c.s3cp, fma(3.0, f2, v3), 2.0 * c.s9 * fs * phi);
    const double chib = c.klap * fma(6.0 * (1.0 - w0), mub, -lsum);
    phib += fma(mub, dphi, chib);
    fsb += fma(mub, dfs, c.cos_ps * chib);
  }
  // rho of Eq. (10)
  const double rlg = c.rho[1] - c.rho[2];
  fsb = fma(rhob, c.rho[0] - fma(w, rlg, c.rho[2]), fsb);
  wb = fma(rhob, (1.0 - fs) * rlg, wb);
  // fs = min(phi0 + w (1 - fl), 1)
  if (!(raw > 1.0)) {
    wb = fma(fsb, 1.0 - fl, wb);
    flb = fma(-w, fsb, flb);
  }
  // w = clamp((1 - phi0 + phi) / 2)
  const double wraw = (phi + (1.0 - phi0)) * 0.5;
  if (!(wraw < 0.0) && !(wraw > 1.0)) phib = fma(0.5, wb, phib);
  // phi = sum g / (1 - mdot / 2)
  const double sgb = is_zero(mdot) ? phib : quot(phib, fma(mdot, -0.5, 1.0));
  mdotb = fma(0.5 * phi, sgb, mdotb);
  // mdot = (1 - rho_s / rho_l) w_prev (fl_prev - fl)
  const double mr = mdotb * c.ratio;
  double wpb = mr * (flp - fl);
  const double flpb = mr * wp;
  flb -= flpb;
  lbmk::allow_next();
  // the inversion of Eq. (8)
  const double ell = wp * c.rl;
  const bool frozen = rhoH < 0.0, liquid = rhoH > ell && !frozen;
  double ellb = 0.0, dL, dTc = 0.0;
  if (frozen || liquid) {
    const double fr = frozen ? wp + phi0 : phi0, fx = min1(fr);
    const Mix<double> m(fx, wp);
    const double r = m(c.rho), cc = m(c.cp), t = quot(Tb, r * cc);
    rhoHb += t;
    if (liquid) ellb = -t;
    double cf, cw;
    cap_slopes(c, fx, wp, r, cc, &cf, &cw);
    if (frozen && !(fr > 1.0)) cw += cf;
    wpb = fma(-t * T, cw, wpb);
  } else if (ell > 0.0) {
    const double t = flb / ell;
    rhoHb += t;
    ellb = -t * (rhoH / ell);
  }
  wpb = fma(ellb, c.rl, wpb);
  dL = ellb * wp * c.rho[1];
  double* lam = a.lam_out + n;
  if (g.has_mask && a.f.mask[n]) {
    // the enthalpy populations read here are h_eq(T_cold, u = 0) at w_prev:
    // h_0 = rho H - rr T + w_0 rr T, h_i = w_i rr T with
    // rho H = cap(w_prev) T + w_prev rho_l L fl_c
    const double Tc = c.T_cold, flc = Tc < 0.0 ? 0.0 : 1.0;
    const double fr = Tc < 0.0 ? phi0 + wp : phi0, fx = min1(fr);
    const Mix<double> m(fx, wp);
    const double r = m(c.rho), cc = m(c.cp);
    double cf, cw;
    cap_slopes(c, fx, wp, r, cc, &cf, &cw);
    if (Tc < 0.0 && !(fr > 1.0)) cw += cf;
    double s = 0.0;  // sum over i > 0 of the adjoints times w_i
#pragma unroll
    for (int i = 1; i < 9; i++)
      s = fma(lam[(18 + i) * P] + rhoHb, i <= 4 ? w1 : w1 * kd, s);
    const double h0b = lam[18 * P] + rhoHb;
    wpb = fma(h0b, fma(cw, Tc, c.rl * flc), wpb);
    dTc = fma(h0b, fma(c.rr, w0 - 1.0, r * cc), s * c.rr);
    dL = fma(h0b, wp * c.rho[1] * flc, dL);
#pragma unroll
    for (int i = 0; i < 9; i++) lam[(18 + i) * P] = 0.0;
    a.acc[9 * P + n] += dTc;
  } else {
#pragma unroll
    for (int i = 0; i < 9; i++) lam[(18 + i) * P] += rhoHb;
  }
#pragma unroll
  for (int i = 0; i < 9; i++) lam[(9 + i) * P] += sgb;
  a.llag_out[G_::FL * P + n] = flpb;
  a.llag_out[G_::W * P + n] = wpb;
  a.llag_out[G_::Q * P + n] = 0.5 * rhoHb;
  if (dL != 0.0) a.acc[4 * P + n] += dL;
}

// Frozen-fraction seed: the adjoints of the lags fl and w the final state's
// reader writes (other lag and population adjoints zero).
static __global__ void __launch_bounds__(REV_NT) rev_seed_ff_kernel(const RevArgs a,
                                                                 double* __restrict__ llag) {
  const NodeGeom<2>& g = a.f.g;
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= g.nodes) return;
  const int P = (int)g.plane, n = node_pos<2>(g, id).n;
  const double fl = a.f.lout[Lag<2>::FL * P + n], w = a.f.lout[Lag<2>::W * P + n];
  llag[Lag<2>::FL * P + n] = -w * a.inv_sum_w;
  llag[Lag<2>::W * P + n] = ((1.0 - fl) - a.ff) * a.inv_sum_w;
}

// Crossing seed (one thread): the position of the last phi = 0 crossing along
// the line and its derivatives with respect to phi at the two nodes.
static __global__ void rev_seed_crossing_kernel(const RevArgs a, double* __restrict__ phib) {
  const NodeGeom<2>& g = a.f.g;
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double* phi = a.f.sc + SC_PHI * g.plane;
  const int len = a.axis == 0 ? g.n[0] : g.n[1];
  const int stride = a.axis == 0 ? 1 : g.pitch;
  const int base = a.axis == 0 ? a.index * g.pitch : a.index;
  double J = __longlong_as_double(0x7ff8000000000000ULL);
  for (int k = len - 2; k >= 0; k--) {
    const int n0 = base + k * stride, n1 = n0 + stride;
    const double va = phi[n0], vb = phi[n1];
    if ((va <= 0.0) != (vb <= 0.0)) {
      const double dd = va - vb;
      J = k + va / dd;
      phib[n0] = -vb / (dd * dd);
      phib[n1] = va / (dd * dd);
      break;
    }
  }
  a.out[0] = J;
}

// Gradient with respect to the initial temperature field (a run from
// set_geometry): the initial enthalpy populations are h_eq(rho H, T, u = 0)
// with rho H = cap T + w rho_l L fl (cap: the frozen capacity below T_m,
// the liquid one at and above, Eq. (8)), so dh_0/dT = cap - rr + w_0 rr and
// dh_i/dT = w_i rr; T is that of the initial state's local pass (its lagged
// w).  lam: the adjoints of the initial h (9 planes); out: dense [ny][nx].
static __global__ void __launch_bounds__(REV_NT) rev_dT0_kernel(const RevArgs a,
                                                             const double* __restrict__ lam,
                                                             double* __restrict__ out) {
  const NodeGeom<2>& g = a.f.g;
  const NodeCoef<double, 2>& c = a.f.c;
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= g.nodes) return;
  const int P = (int)g.plane, n = node_pos<2>(g, id).n;
  const double T = a.f.sc[SC_T * P + n], wp = a.f.lin[Lag<2>::W * P + n], phi0 = a.f.phi0[n];
  const Mix<double> m(T < 0.0 ? min1(wp + phi0) : phi0, wp);
  const double cap = m(c.rho) * m(c.cp);
  double d = lam[n] * (cap - c.rr + Lat<2>::w0 * c.rr);
#pragma unroll
  for (int i = 1; i < 9; i++)
    d += lam[i * P + n] * (i <= 4 ? Lat<2>::w1 : Lat<2>::w1 * Lat<2>::kd) * c.rr;
  out[id] = d;
}

#endif  // LBM_ADJOINT_KERNELS

// one reverse step from lam_in to lam_out (after launch_node_local of its state)
cudaError_t launch_rev_step(const RevArgs& a, cudaStream_t s);
cudaError_t launch_rev_seed_ff(const RevArgs& a, double* llag, cudaStream_t s);
cudaError_t launch_rev_seed_crossing(const RevArgs& a, double* phib, cudaStream_t s);
cudaError_t launch_rev_dT0(const RevArgs& a, const double* lam, double* out, cudaStream_t s);

}  // namespace lbmn
