// lbm_node.cuh -- the coupled step as two barrier-free kernels with one
// thread per node, on D2Q9 or D3Q19, for sm_103a: the double-precision and
// tangent steps of both lattices and the three-dimensional float step.
//
//   node_local    per node: the sums of the phase and enthalpy populations,
//                 the inversion of Eq. (8), mdot, phi, w, fs and rho (rows
//                 a1-a2); writes the three planes the neighbours' stencils
//                 read -- phi, chi = phi + cos(theta) phi0 + cos(psi) fs (the
//                 one Laplacian of Eq. (6) is that of chi) and rho --, T, rho H
//                 and mdot for the node itself, and fl and w straight into
//                 the next step's lag planes.
//   node_collide  per node: the stencils from those planes and the lagged
//                 pressure through L1/L2, mu_phi, forces, velocity and pressure, the three
//                 collisions, push streaming with the wall rules, lag store;
//                 or (MODE_READ) the field read-out; diagnostics by warp.
//
// What bounds it.  On this part the FP64 pipe takes a warp instruction every
// 16 cycles of an SM (1.25 TFLOP/s over 152 SMs), so the double step is
// bound by the number of FP64 instructions and nothing else: 70 loads per
// node cost a tenth of it.  Hence (a) every node's local state is evaluated
// once (a fused tile evaluates its ring again); (b) no lane idles -- node ids
// are linear over the grid, so a warp runs over row ends, and a grid of a
// few thousand nodes is spread over all SMs by one-warp blocks; (c) the
// collisions are written for the fewest operations: with the magic relation
// 1/tau_s + 1/tau_a = 2 of the TRT, h_i* = q_i + (1/tau_a - 1) (h_o - q_o),
// so a population of any lattice costs two or three operations; the odd
// and quadratic equilibrium terms are dot products with vectors scaled once
// per node (the diagonal weights are 1/4 or 1/2 of the axis ones, exact);
// reciprocals take a hardware seed and one third-order iteration; clamps
// compare integer words.  Edge nodes take the same arithmetic as inner ones
// and differ only in where they store.
//
// Measured (GB300): the double 512 x 512 droplet with sums every step, 374 us
// a step as one fused 32 x 8 tile kernel, 188 us as these two (35 + 153; 347
// FP64 instructions a node against about 640 and the ring's; FP64 pipe 85 %
// busy); the tangent step of 250 x 190 nodes 298 us and 88 us.
#pragma once

#include "lbm_kernels.cuh"

namespace lbmn {

using lbmk::BC_DIRICHLET;
using lbmk::BC_PERIODIC;
using lbmk::Dual;
using lbmk::LAT_FLOW;
using lbmk::LAT_HEAT;
using lbmk::LAT_PHASE;
using lbmk::MODE_READ;
using lbmk::MODE_STEP;
using lbmk::NDIAG;

// ---------------------------------------------------------------------------
// lattices: opposite pairs, the D axis pairs first
// ---------------------------------------------------------------------------

template <int D>
struct Lat;
template <>
struct Lat<2> {
  static constexpr int Q = 9, NP = 4;
  // first member of pair k; its opposite
  __host__ __device__ static constexpr int first(int k) { return k < 2 ? k + 1 : k + 3; }
  __host__ __device__ static constexpr int opp(int i) { return lbmk::qopp(i); }
  __host__ __device__ static constexpr int c(int i, int a) {
    return a == 0 ? lbmk::qx(i) : lbmk::qy(i);
  }
  static constexpr double w0 = 4.0 / 9.0, w1 = 1.0 / 9.0, kd = 0.25;  // diagonal weight = kd w1
  static constexpr double trace = 2.0 / 3.0;                          // D cs^2
};
template <>
struct Lat<3> {
  static constexpr int Q = 19, NP = 9;
  __host__ __device__ static constexpr int first(int k) { return 2 * k + 1; }
  __host__ __device__ static constexpr int opp(int i) {
    return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1);
  }
  // D3Q19 of Eq. (13): rest; the six axes; the twelve edge diagonals, in the
  // column order of the printed velocity matrix
  __host__ __device__ static constexpr int c(int i, int a) {
    return a == 0   ? ((i == 1 || i == 7 || i == 9 || i == 11 || i == 13)    ? 1
                       : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1
                                                                             : 0)
           : a == 1 ? ((i == 3 || i == 7 || i == 10 || i == 15 || i == 17)  ? 1
                       : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1
                                                                            : 0)
                    : ((i == 5 || i == 11 || i == 14 || i == 15 || i == 18)   ? 1
                       : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1
                                                                              : 0);
  }
  static constexpr double w0 = 1.0 / 3.0, w1 = 1.0 / 18.0, kd = 0.5;
  static constexpr double trace = 1.0;
};
template <int D>
__host__ __device__ constexpr bool is_axis(int k) { return k < D; }

// lag planes: fl, w, p, phi u (D), Q
template <int D>
struct Lag {
  static constexpr int FL = 0, W = 1, P = 2, PHU = 3, Q = 3 + D, N = 4 + D;
};
enum { SC_PHI = 0, SC_CHI, SC_RHO, SC_T, SC_RHOH, SC_MDOT, NSC };

// ---------------------------------------------------------------------------
// arithmetic: R is float, double or Dual, K<R> its plain type (constants
// that no parameter direction moves cost a tangent no derivative)
// ---------------------------------------------------------------------------

template <typename R>
struct Plain { using type = R; };
template <>
struct Plain<Dual> { using type = double; };
template <typename R>
using K = typename Plain<R>::type;

__device__ __forceinline__ Dual add(const Dual& a, double b) { return Dual(a.v + b, a.d); }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ Dual mul(const Dual& a, double b) { return Dual(a.v * b, a.d * b); }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ float mul(float a, float b) { return a * b; }
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ Dual mad(const Dual& a, const Dual& b, const Dual& c) {
  return Dual(fma(a.v, b.v, c.v), fma(a.d, b.v, fma(a.v, b.d, c.d)));
}
__device__ __forceinline__ Dual mad(const Dual& a, double b, const Dual& c) {
  return Dual(fma(a.v, b, c.v), fma(a.d, b, c.d));
}
__device__ __forceinline__ Dual mad(double b, const Dual& a, const Dual& c) { return mad(a, b, c); }
__device__ __forceinline__ Dual mad(const Dual& a, double b, double c) {
  return Dual(fma(a.v, b, c), a.d * b);
}
// a product that is rounded by itself, whatever it is added to
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ Dual mul_rn(const Dual& a, double b) {
  return Dual(__dmul_rn(a.v, b), __dmul_rn(a.d, b));
}
__device__ __forceinline__ double val(double x) { return x; }
__device__ __forceinline__ float val(float x) { return x; }
__device__ __forceinline__ double val(const Dual& x) { return x.v; }
template <typename R>
__device__ __forceinline__ K<R> plain(const R& x) { return val(x); }

// Reciprocal in double: the hardware's approximate reciprocal r0 (PTX
// rcp.approx.ftz.f64) and one step of the third-order iteration
// r = r0 + r0 (e + e^2), e = 1 - b r0 (Householder's method of order 2, three
// FMAs): the error e^3 of the step is far below half an ulp, so the result
// is off by less than one ulp (three FP64 instructions against about nine of
// the IEEE division).  Divisors here are positive normal numbers.
__device__ __forceinline__ double rcp(double b) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
  const double e = fma(-b, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ float rcp(float b) { return lbmk::qdiv(1.f, b); }
__device__ __forceinline__ Dual rcp(const Dual& b) {
  const double r = rcp(b.v);
  return Dual(r, -(b.d * r) * r);
}
// Quotient: a r corrected once by its exact residual (Markstein's correction
// step), within one ulp of a / b.
__device__ __forceinline__ double quot(double a, double b) {
  const double r = rcp(b), q = a * r;
  return fma(fma(-q, b, a), r, q);
}
__device__ __forceinline__ Dual quot(const Dual& a, const Dual& b) {
  const double r = rcp(b.v), q0 = a.v * r;
  const double q = fma(fma(-q0, b.v, a.v), r, q0);
  return Dual(q, fma(-q, b.d, a.d) * r);
}

// max(0, min(v, 1)) on the words of a double: the comparisons run on the
// integer pipe.  NaN stays NaN.
__device__ __forceinline__ int above_one(double v) {  // v >= 1 (not NaN)
  return (unsigned)(__double2hiint(v) - 0x3ff00000) <= 0x40000000u;
}
__device__ __forceinline__ int below_zero(double v) {  // v < 0 or v == -0 (not NaN)
  return (unsigned)__double2hiint(v) - 0x80000000u <= 0x7ff00000u;
}
__device__ __forceinline__ double clamp01(double v) {
  v = below_zero(v) ? 0.0 : v;
  return above_one(v) ? 1.0 : v;
}
__device__ __forceinline__ double min1(double v) { return above_one(v) ? 1.0 : v; }
// the derivative is that of the branch taken; at 0 and 1 exactly that of v
__device__ __forceinline__ Dual clamp01(const Dual& v) {
  return v.v < 0.0 ? Dual(0.0) : (v.v > 1.0 ? Dual(1.0) : v);
}
__device__ __forceinline__ Dual min1(const Dual& v) { return v.v > 1.0 ? Dual(1.0) : v; }
__device__ __forceinline__ float clamp01(float v) { return lbmk::clamp01(v); }
__device__ __forceinline__ float min1(float v) { return v > 1.f ? 1.f : v; }
__device__ __forceinline__ bool finite_word(double v) {
  return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ bool finite_word(const Dual& v) {
  return finite_word(v.v) && finite_word(v.d);
}
__device__ __forceinline__ bool is_zero(double v) {
  return ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) == 0;
}

// ---------------------------------------------------------------------------
// constants, geometry, arguments
// ---------------------------------------------------------------------------

template <typename R, int D>
struct NodeCoef {
  // Eq. (10) properties: solid, liquid, gas
  K<R> rho[3], mu[3], lam[3], cp[3];
  K<R> rr, inv_rr3;          // rho_ref Cp_ref; 1 / (rho_ref Cp_ref cs^2)
  K<R> s3, s9, klap, s3cp;   // Eq. (6): 3 sigma / eps, 9 sigma / eps, 3 eps sigma / 8, s3 cos psi
  K<R> cos_ps;
  K<R> omg, itg_eta, gcoef;  // 1 - 1/tau_g, eta / tau_g, 1 - 1/(2 tau_g)
  K<R> itg, eta;
  K<R> v_new, v_old;         // 3 w_1 (1/tau_g + gcoef), 3 w_1 gcoef
  K<R> ratio;                // 1 - rho_s / rho_l
  K<R> g[D];                 // body force
  R rl;                      // rho_l L
  R cos_th, s3ct;            // cos theta, s3 cos theta
  R T_cold;
  R T_wall[2 * D];
  unsigned readings;
};

// Division of a node id by a grid extent: q = (id m) >> (31 + s) with the
// round-up multiplier of Granlund and Montgomery, exact for 0 <= id < 2^31.
struct FastDiv {
  unsigned d, m, s;
};
inline FastDiv make_fastdiv(unsigned d) {
  FastDiv f;
  f.d = d;
  f.s = 0;
  while ((1u << f.s) < d && f.s < 31) f.s++;
  // ceil(2^(31 + s) / d) fits 32 bits; ids below 2^31 are divided exactly
  f.m = (unsigned)(((1ull << (31 + f.s)) + d - 1) / d);
  return f;
}
__host__ __device__ inline unsigned fast_div(unsigned id, const FastDiv& f) {
  return (unsigned)(((unsigned long long)id * f.m) >> (31 + f.s));
}

template <int D>
struct NodeGeom {
  int n[D];       // extents, x first
  int pitch;      // elements of a row
  int nodes;      // product of the extents
  FastDiv dx, dy; // by n[0], by n[1] (D = 3)
  long long plane;
  int bc[2 * D];
  int lattices, has_mask;
};

template <typename R, int D>
struct NodeArgs {
  NodeGeom<D> g;
  NodeCoef<R, D> c;
  const R* __restrict__ pin;
  R* __restrict__ pout;
  const R* __restrict__ lin;
  R* lout;                      // node_local writes fl and w, node_collide reads them back
  const R* __restrict__ phi0;
  const uint8_t* __restrict__ mask;
  R* sc;                        // NSC planes: node_local writes, node_collide reads
  double* diag;                 // [NDIAG][warps of the grid] partial sums
  int nwarps;
};

// Up to NODE_BATCH_GRIDS double grids in one launch: the table travels in the
// kernel's parameter space (448 B a grid).
constexpr int NODE_BATCH_GRIDS = 64, NODE_BATCH_THREADS = 128;
struct NodeBatch {
  int ngrids;
  int base[NODE_BATCH_GRIDS + 1];  // first block of each grid; [ngrids] = total
  NodeArgs<double, 2> args[NODE_BATCH_GRIDS];
};

constexpr int NFIELDS_MAX = 13;
struct ReadOut {
  double* out[NFIELDS_MAX];  // dense outputs in field order, or null
};

// position of a node
template <int D>
struct Pos {
  int x[D];
  int n;  // index within a plane
};
template <int D>
__device__ __forceinline__ Pos<D> node_pos(const NodeGeom<D>& g, int id) {
  Pos<D> p;
  const int row = (int)fast_div((unsigned)id, g.dx);
  p.x[0] = id - row * g.n[0];
  if constexpr (D == 2) {
    p.x[1] = row;
  } else {
    p.x[2] = (int)fast_div((unsigned)row, g.dy);
    p.x[1] = row - p.x[2] * g.n[1];
  }
  p.n = row * g.pitch + p.x[0];
  return p;
}
// the node at (x, y, z), and its id in the dense order of the outputs
__device__ __forceinline__ Pos<3> node_at(const NodeGeom<3>& g, int x, int y, int z) {
  Pos<3> p;
  p.x[0] = x;
  p.x[1] = y;
  p.x[2] = z;
  p.n = (z * g.n[1] + y) * g.pitch + x;
  return p;
}
template <int D>
__device__ __forceinline__ long long dense_id(const NodeGeom<D>& g, const Pos<D>& p) {
  if constexpr (D == 2) return (long long)p.x[1] * g.n[0] + p.x[0];
  else return ((long long)p.x[2] * g.n[1] + p.x[1]) * g.n[0] + p.x[0];
}

// Offsets to the neighbours along each axis (wrapped on a periodic axis, 0
// -- the node itself, mirrored -- beyond a wall) and the walls they lie
// behind (bit 2 a: low side of axis a, bit 2 a + 1: high side).
template <int D>
struct Nbr {
  int lo[D], hi[D];
  unsigned wall;
};
template <int D>
__device__ __forceinline__ Nbr<D> neighbours(const NodeGeom<D>& g, const Pos<D>& p) {
  Nbr<D> b;
  b.wall = 0;
  int stride = 1;
#pragma unroll
  for (int a = 0; a < D; a++) {
    b.lo[a] = -stride;
    b.hi[a] = stride;
    if (p.x[a] == 0) {
      const bool per = g.bc[2 * a] == BC_PERIODIC;
      b.lo[a] = per ? (g.n[a] - 1) * stride : 0;
      if (!per) b.wall |= 1u << (2 * a);
    }
    if (p.x[a] == g.n[a] - 1) {
      const bool per = g.bc[2 * a + 1] == BC_PERIODIC;
      b.hi[a] = per ? -(g.n[a] - 1) * stride : 0;
      if (!per) b.wall |= 2u << (2 * a);
    }
    stride = a == 0 ? g.pitch : stride * g.n[a];
  }
  return b;
}
// offset to x + c_i, and the walls that direction i crosses
template <int D>
__device__ __forceinline__ int toward(const Nbr<D>& b, int i) {
  int o = 0;
#pragma unroll
  for (int a = 0; a < D; a++) {
    const int c = Lat<D>::c(i, a);
    if (c) o += c > 0 ? b.hi[a] : b.lo[a];
  }
  return o;
}
template <int D>
__host__ __device__ constexpr unsigned crossing(int i) {
  unsigned m = 0;
  for (int a = 0; a < D; a++) {
    const int c = Lat<D>::c(i, a);
    if (c) m |= 1u << (2 * a + (c > 0 ? 1 : 0));
  }
  return m;
}

// Eq. (10) at (fs, w): weights and a property
template <typename R>
struct Mix {
  R s, l, g;
  __device__ __forceinline__ Mix(const R& fs, const R& w) {
    const R b = R(1) - fs;
    s = fs;
    l = b * w;
    g = b - l;
  }
  __device__ __forceinline__ R operator()(const K<R>* z) const {
    return mad(g, z[2], mad(l, z[1], mul(s, z[0])));
  }
};

// ---------------------------------------------------------------------------
// kernel 1
// ---------------------------------------------------------------------------

// Population sums in the fixed orders of the fused step (2-D) and in plane
// order (3-D): the initial state's sums decide by their last bits which side
// of a clamp phi = -(1 - phi0) falls on in the gas beside a solid.
template <int D, bool HEAT, typename R>
__device__ __forceinline__ R sum_pops(const R* v) {
  if constexpr (D == 2) {
    return HEAT ? lbmk::sum_h(v) : lbmk::sum_g(v);
  } else {
    R s = v[0];
#pragma unroll
    for (int i = 1; i < Lat<D>::Q; i++) s += v[i];
    return s;
  }
}

// h_eq(T_cold, u = 0) of Eq. (25) at a cold-mask node's lagged weight, which
// replaces its stored enthalpy populations when they are read: the rest
// population and rho_ref Cp_ref T_cold (the others are w_i times it)
template <int D, typename R>
__device__ __forceinline__ void cold_node(const NodeCoef<R, D>& c, const R& w, K<R> phi0, R* h) {
  const R T = c.T_cold;
  const bool cold = val(T) < 0;
  const Mix<R> m(cold ? min1(add(w, phi0)) : R(phi0), w);
  R rhoH = m(c.rho) * m(c.cp) * T;
  if (!cold) rhoH = mad(w, c.rl, rhoH);
  const R rrT = mul(T, c.rr);
  h[0] = mad(rrT, K<R>(Lat<D>::w0 - 1.0), rhoH);
#pragma unroll
  for (int i = 1; i < Lat<D>::Q; i++)
    h[i] = mul(rrT, K<R>(i <= 2 * D ? Lat<D>::w1 : Lat<D>::w1 * Lat<D>::kd));
}

template <typename R>
struct LocalState {
  R T, fl, mdot, rhoH, phi, w, fs, rho;
};

template <typename R, int D>
__device__ __forceinline__ LocalState<R> local_of(const NodeCoef<R, D>& c, int lat, const R& sg,
                                                  const R& sh, const R& flp, const R& wp,
                                                  const R& Qp, K<R> phi0) {
  LocalState<R> L;
  L.T = R(0);
  L.fl = flp;
  L.rhoH = R(0);
  L.mdot = R(0);
  if (lat & LAT_HEAT) {
    // Eq. (8) with reading R-T1: one heat capacity and one quotient whichever
    // side of the mushy range the node is on
    L.rhoH = mad(Qp, K<R>(0.5), sh);  // Eq. (28), lagged source
    const R ell = wp * c.rl;
    const bool frozen = val(L.rhoH) < K<R>(0), liquid = val(L.rhoH) > val(ell) && !frozen;
    if (frozen || liquid) {
      const Mix<R> m(frozen ? min1(add(wp, phi0)) : R(phi0), wp);
      const R cap = m(c.rho) * m(c.cp);
      if constexpr (std::is_same<R, float>::value)
        L.T = lbmk::qdiv(frozen ? L.rhoH : L.rhoH - ell, cap);
      else
        L.T = quot(frozen ? L.rhoH : L.rhoH - ell, cap);
      L.fl = frozen ? R(0) : R(1);
    } else {
      L.fl = val(ell) > K<R>(0) ? lbmk::qdiv(L.rhoH, ell) : R(1);
      L.fl = lbmk::clamp01(L.fl);
    }
    L.mdot = mul(wp, c.ratio) * (flp - L.fl);  // Eq. (1), phase-change part
  }
  if (lat & LAT_PHASE) {
    // Eq. (22) solved for phi; without phase change the divisor is exactly 1
    // (a tangent still divides: the derivative of mdot need not vanish)
    if constexpr (std::is_same<R, double>::value)
      L.phi = is_zero(L.mdot) ? sg : quot(sg, fma(-0.5, L.mdot, 1.0));
    else if constexpr (std::is_same<R, float>::value)
      L.phi = lbmk::qdiv(sg, 1.f - 0.5f * L.mdot);
    else
      L.phi = quot(sg, mad(L.mdot, K<R>(-0.5), K<R>(1)));
    L.w = clamp01(mul(add(L.phi, K<R>(1) - phi0), K<R>(0.5)));
  } else {
    L.w = wp;
    L.phi = add(add(mul(wp, K<R>(2)), K<R>(-1)), phi0);
  }
  L.fs = min1(mad(L.w, R(1) - L.fl, R(phi0)));
  L.rho = Mix<R>(L.fs, L.w)(c.rho);
  return L;
}

// I: the type of plane offsets (int while all population planes fit 31 bits)
template <typename R, int D, int LATC, typename I>
__device__ __forceinline__ void node_local(const NodeArgs<R, D>& a, int n) {
  const NodeGeom<D>& g = a.g;
  const NodeCoef<R, D>& c = a.c;
  constexpr int Q = Lat<D>::Q;
  using L_ = Lag<D>;
  const int lat = LATC ? LATC : g.lattices;
  const I P = (I)g.plane;
  const K<R> phi0 = plain(a.phi0[n]);
  const R flp = a.lin[L_::FL * P + n], wp = a.lin[L_::W * P + n], Qp = a.lin[L_::Q * P + n];
  R sg = R(0), sh = R(0);
  if (lat & LAT_PHASE) {
    R v[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) v[i] = a.pin[(Q + i) * P + n];
    sg = sum_pops<D, false>(v);
  }
  if (lat & LAT_HEAT) {
    R v[Q];
    if (g.has_mask && a.mask[n]) {
      cold_node<D>(c, wp, phi0, v);
    } else {
#pragma unroll
      for (int i = 0; i < Q; i++) v[i] = a.pin[(2 * Q + i) * P + n];
    }
    sh = sum_pops<D, true>(v);
  }
  const LocalState<R> L = local_of<R, D>(c, lat, sg, sh, flp, wp, Qp, phi0);
  lbmk::allow_next();
  R* sc = a.sc + n;
  sc[SC_PHI * P] = L.phi;
  sc[SC_CHI * P] = mad(L.fs, c.cos_ps, mad(c.cos_th, phi0, L.phi));
  sc[SC_RHO * P] = L.rho;
  sc[SC_T * P] = L.T;
  sc[SC_RHOH * P] = L.rhoH;
  sc[SC_MDOT * P] = L.mdot;
  a.lout[L_::FL * P + n] = L.fl;
  a.lout[L_::W * P + n] = L.w;
}

// ---------------------------------------------------------------------------
// kernel 2
// ---------------------------------------------------------------------------

// 3 sum_i w_i c_i v(x + c_i), opposite neighbours differenced first
template <typename R, int D>
__device__ __forceinline__ void gradient(const R* __restrict__ v, const Nbr<D>& b, R* out) {
  using L_ = Lat<D>;
  R d[L_::NP];
#pragma unroll
  for (int k = 0; k < L_::NP; k++) {
    const int i = L_::first(k);
    d[k] = v[toward<D>(b, i)] - v[toward<D>(b, L_::opp(i))];
  }
#pragma unroll
  for (int a = 0; a < D; a++) {
    R s = R(0);
    bool any = false;
#pragma unroll
    for (int k = D; k < L_::NP; k++) {
      const int c = L_::c(L_::first(k), a);
      if (c == 0) continue;
      s = any ? (c > 0 ? s + d[k] : s - d[k]) : (c > 0 ? d[k] : -d[k]);
      any = true;
    }
    out[a] = mad(s, K<R>(3.0 * L_::w1 * L_::kd), mul(d[a], K<R>(3.0 * L_::w1)));
  }
}

// 6 sum_i w_i (v(x + c_i) - v(x)).  Float subtracts the centre from every
// neighbour (exact for close ones); double from sums of 2, 4 and 8 neighbours,
// half the operations.  Both are exactly zero for a uniform v -- sums of a
// power of two of equal values do not round -- so a state at rest stays so
// and phi stays exactly 0 inside a solid, where its sign decides clamps.
template <typename R, int D>
__device__ __forceinline__ R laplacian(const R* __restrict__ v, const R& vc, const Nbr<D>& b) {
  using L_ = Lat<D>;
  R s[L_::NP];
#pragma unroll
  for (int k = 0; k < L_::NP; k++) {
    const int i = L_::first(k);
    if constexpr (std::is_same<R, float>::value)
      s[k] = (v[toward<D>(b, i)] - vc) + (v[toward<D>(b, L_::opp(i))] - vc);
    else
      s[k] = v[toward<D>(b, i)] + v[toward<D>(b, L_::opp(i))];
  }
  R sa, sd;
  if constexpr (std::is_same<R, float>::value) {
    sa = s[0];
    sd = s[D];
#pragma unroll
    for (int k = 1; k < D; k++) sa += s[k];
#pragma unroll
    for (int k = D + 1; k < L_::NP; k++) sd += s[k];
  } else {
    sa = mad(vc, K<R>(-4), s[0] + s[1]);
    if constexpr (D == 2) {
      sd = mad(vc, K<R>(-4), s[2] + s[3]);
    } else {
      sa += mad(vc, K<R>(-2), s[2]);
      sd = mad(vc, K<R>(-8), (s[3] + s[4]) + (s[5] + s[6])) + mad(vc, K<R>(-4), s[7] + s[8]);
    }
  }
  return mad(sd, K<R>(6.0 * L_::w1 * L_::kd), mul(sa, K<R>(6.0 * L_::w1)));
}

// Store of one post-collision population of direction i; behind a wall it
// comes back in the opposite one, at a Dirichlet wall of the enthalpy lattice
// (HEAT) by anti-bounce-back.  At a corner the first wall in the order of the
// axes decides.
template <bool HEAT, typename R, int D, typename I>
__device__ __forceinline__ void push(const NodeArgs<R, D>& a, R* __restrict__ plane0, I P, int n,
                                     const Nbr<D>& b, int i, R v) {
  const unsigned hit = i ? (b.wall & crossing<D>(i)) : 0u;
  if (hit == 0u) {
    plane0[i * P + n + toward<D>(b, i)] = v;
  } else {
    if (HEAT) {
      const int side = __ffs((int)hit) - 1;
      if (a.g.bc[side] == BC_DIRICHLET) {
        const K<R> w = K<R>(i <= 2 * D ? Lat<D>::w1 : Lat<D>::w1 * Lat<D>::kd);
        v = mad(a.c.T_wall[side], K<R>(2) * w * a.c.rr, -v);
      }
    }
    plane0[Lat<D>::opp(i) * P + n] = v;
  }
}

template <typename R>
__device__ __forceinline__ R warp_sum8(const R* v, int lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  R a[4], h[2];
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const R keep = b4 ? v[4 + j] : v[j], send = b4 ? v[j] : v[4 + j];
    a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int j = 0; j < 2; j++) {
    const R keep = b3 ? a[2 + j] : a[j], send = b3 ? a[j] : a[2 + j];
    h[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  R q;
  {
    const R keep = b2 ? h[1] : h[0], send = b2 ? h[0] : h[1];
    q = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  q += __shfl_xor_sync(0xffffffffu, q, 2);
  q += __shfl_xor_sync(0xffffffffu, q, 1);
  return q;
}

// One warp's sums of the nine diagnostics (the ninth counts nodes whose sums
// are not finite, by ballot) into its column of the partials.  Warps are the
// unit of the partial sums, so they do not depend on the block size.
__device__ __forceinline__ void warp_diag(double* diag, int nwarps, int wid, const double* v,
                                          bool bad) {
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(0xffffffffu, bad);
  const double s = warp_sum8(v, lane);
  if (wid >= nwarps) return;
  if ((lane & 3) == 0) diag[(long long)((lane >> 2) & 7) * nwarps + wid] = s;
  if (lane == 1) diag[8ll * nwarps + wid] = (double)__popc(m);
}
// tangent: the derivatives' sums follow as rows NDIAG ... 2 NDIAG - 1
__device__ __forceinline__ void warp_diag(double* diag, int nwarps, int wid, const Dual* v,
                                          bool bad) {
  double x[8], d[8];
#pragma unroll
  for (int k = 0; k < 8; k++) {
    x[k] = v[k].v;
    d[k] = v[k].d;
  }
  warp_diag(diag, nwarps, wid, x, bad);
  warp_diag(diag + (long long)NDIAG * nwarps, nwarps, wid, d, false);
}

// READ: the field read-out of the state instead of the step.  Every lane of
// a warp calls it (the diagnostics are warp sums, of warp wid).
template <typename R, int D, int LATC, bool READ, bool DIAG, typename I>
__device__ __forceinline__ void node_collide(const NodeArgs<R, D>& a, const ReadOut* ro, bool valid,
                                             const Pos<D>& pos, int wid) {
  const NodeGeom<D>& g = a.g;
  const NodeCoef<R, D>& c = a.c;
  using L_ = Lat<D>;
  using G_ = Lag<D>;
  constexpr int Q = L_::Q, NP = L_::NP;
  using k_t = K<R>;
  const int lat = LATC ? LATC : g.lattices;
  R dv[8];
  bool bad = false;
  if (DIAG) {
#pragma unroll
    for (int k = 0; k < 8; k++) dv[k] = R(0);
  }
  if (valid) {
    const I P = (I)g.plane;
    const int n = pos.n;
    const Nbr<D> nb = neighbours<D>(g, pos);
    const R* sc = a.sc + n;
    const R phi = sc[SC_PHI * P], rho = sc[SC_RHO * P];
    const R T = sc[SC_T * P], mdot = sc[SC_MDOT * P], rhoH = sc[SC_RHOH * P];
    const R fl = a.lout[G_::FL * P + n], w = a.lout[G_::W * P + n];
    const k_t phi0 = plain(a.phi0[n]);
    const R fs = min1(mad(w, R(1) - fl, R(phi0)));
    const Mix<R> mix(fs, w);

    // ---- chemical potential Eq. (6), forces -----------------------------------
    R mu = R(0), F[D];
#pragma unroll
    for (int k = 0; k < D; k++) F[k] = mul(rho, c.g[k]);
    if (lat & LAT_PHASE) {
      R gph[D];
      gradient<R, D>(sc + SC_PHI * P, nb, gph);
      const R lap = laplacian<R, D>(sc + SC_CHI * P, sc[SC_CHI * P], nb);
      const R v = add(phi, k_t(-1)) * add(phi, k_t(1));  // phi^2 - 1
      const R v3 = mad(v, k_t(3), k_t(2));               // 3 phi^2 - 1
      const k_t q2 = phi0 * phi0;
      const R f2 = fs * fs;
      R m = phi * mad(add(f2, q2), c.s9, mul(v, c.s3));
      m = mad(mul(c.s3ct, phi0), add(v3, q2), m);
      m = mad(mul(fs, c.s3cp), v3 + f2, m);
      mu = mad(lap, -c.klap, m);
#pragma unroll
      for (int k = 0; k < D; k++) F[k] = mad(mu, gph[k], F[k]);
    }

    // ---- velocity and pressure Eq. (17) ----------------------------------------
    R u[D], uu = R(0), pr = R(0), S = R(0), uFt = R(0), itau = R(0);
    R Ft[D], Gf[D], f[Q];
#pragma unroll
    for (int k = 0; k < D; k++) u[k] = R(0);
    R fsym0 = R(0), ftot = R(0);
    const bool iso = (c.readings & 1u) != 0;
    if (lat & LAT_FLOW) {
#pragma unroll
      for (int i = 0; i < Q; i++) f[i] = a.pin[i * P + n];
      R gr[D], gp[D];
      gradient<R, D>(sc + SC_RHO * P, nb, gr);
      gradient<R, D>(a.lin + G_::P * P + n, nb, gp);
      R j[D], snz = R(0);
      {
        R d[NP];
#pragma unroll
        for (int k = 0; k < NP; k++) {
          const int i = L_::first(k), o = L_::opp(i);
          d[k] = f[i] - f[o];
          const R s = f[i] + f[o];
          snz = k == 0 ? s : snz + s;
        }
#pragma unroll
        for (int k = 0; k < D; k++) {
          j[k] = d[k];
#pragma unroll
          for (int q = D; q < NP; q++) {
            const int cc = L_::c(L_::first(q), k);
            if (cc > 0) j[k] += d[q];
            else if (cc < 0) j[k] -= d[q];
          }
        }
      }
      if (DIAG) ftot = snz + f[0];
      // penalty force f = fs (u_s - u*), u_s = 0: u = (1 - fs / 2) u*
      const R irho = rcp(rho);
      const R half = mad(fs, k_t(-0.5), k_t(1)), rf = rho * fs;
#pragma unroll
      for (int k = 0; k < D; k++) {
        const R us = mad(F[k], k_t(0.5), j[k]) * irho;
        u[k] = us * half;
        Gf[k] = mad(-rf, us, F[k]);
        uu = k == 0 ? u[k] * u[k] : mad(u[k], u[k], uu);
        // modified force (reading R-FT), lagged pressure (reading R-FP)
        Ft[k] = mad(gr[k], k_t(1.0 / 3.0), F[k] - gp[k]);
        uFt = k == 0 ? u[k] * Ft[k] : mad(u[k], Ft[k], uFt);
      }
      S = rho * mdot;
#pragma unroll
      for (int k = 0; k < D; k++) S = mad(u[k], gr[k], S);
      fsym0 = mad(uFt, k_t(-3), S);
      const R tm = mul(mix(c.mu) * irho, k_t(3));  // tau_f - 1/2
      itau = rcp(add(tm, k_t(0.5)));
      // F_0 of Eq. (16) / w_0; the variant of the modified force adds
      // cs^2 S (c.c - D cs^2) 9/2 to it
      R F0 = fsym0;
      if (iso) F0 = mad(S, k_t(-1.5 * L_::trace), F0);
      R t = mad(S, k_t(0.5), snz);
      t = mad(mul(tm, k_t(L_::w0)), F0, t);
      t = mad(mul(rho, k_t(-1.5 * L_::w0)), uu, t);
      pr = mul(t, k_t(1.0 / (3.0 * (1.0 - L_::w0))));
    }

    if (DIAG) {
      const R wl = w * fl;
      dv[0] = rho;
      dv[3] = wl;
      dv[4] = w;
      dv[5] = w - wl;
      dv[1] = mad(dv[5], c.rho[0], mul(wl, c.rho[1]));
      dv[2] = rhoH;
      dv[6] = phi;
      dv[7] = mul(rho, k_t(0.5)) * uu;
    }

    if (READ) {
      const R vals2[12] = {phi, fs, fl, T, rhoH, pr, u[0], u[1], rho, mu, w, mdot};
      const long long N = g.nodes, id = dense_id<D>(g, pos);
      if constexpr (D == 2) {
#pragma unroll
        for (int k = 0; k < 12; k++)
          if (ro->out[k]) lbmk::put_out(ro->out[k], id, N, vals2[k]);
      } else {
        // derivatives follow all value planes of the read-out
        const R vals[13] = {phi, fs, fl, T, rhoH, pr, u[0], u[1], u[2], rho, mu, w, mdot};
#pragma unroll
        for (int k = 0; k < 13; k++)
          if (ro->out[k]) lbmk::put_out(ro->out[k], id, 13 * N, vals[k]);
      }
      if (DIAG) {
        // the populations' sums, for the non-finite count
        bad = !finite_word(ftot);
        if (lat & LAT_PHASE) {
          R v[Q];
#pragma unroll
          for (int i = 0; i < Q; i++) v[i] = a.pin[(Q + i) * P + n];
          bad = bad || !finite_word(sum_pops<D, false>(v));
        }
        bad = bad || !finite_word(rhoH);
      }
    } else {
      R phu[D];
#pragma unroll
      for (int k = 0; k < D; k++) phu[k] = phi * u[k];
      R* out = a.pout;
      // c_i . u of the diagonal pairs, shared by the flow and heat collisions
      R cud[NP - D];
#pragma unroll
      for (int k = D; k < NP; k++) {
        const int i = L_::first(k);
        R s = R(0);
        bool any = false;
#pragma unroll
        for (int q = 0; q < D; q++) {
          const int cc = L_::c(i, q);
          if (cc == 0) continue;
          s = any ? (cc > 0 ? s + u[q] : s - u[q]) : (cc > 0 ? u[q] : -u[q]);
          any = true;
        }
        cud[k - D] = s;
      }

      // ---- flow collision Eqs. (11), (14)-(16) -----------------------------------
      if (lat & LAT_FLOW) {
        const R omi = R(1) - itau, fco = mad(itau, k_t(-0.5), k_t(1));
        // even part without c: 3 p + rho s; source; the 9/2 cu^2 and 9 cu cFt
        // terms are cu (c . X), the odd ones c . V
        const R ir = itau * rho;
        const R p3 = mul(itau * pr, k_t(3));
        const R Kn = mad(mul(ir, k_t(-1.5)), uu, mad(fco, fsym0, p3));
        R Ka = mul(Kn, k_t(L_::w1)), Kd = mul(Kn, k_t(L_::w1 * L_::kd));
        R K0 = mad(Kn, k_t(L_::w0), -p3);
        if (iso) {
          const R fS = mul(fco * S, k_t(1.5));
          Ka = mad(fS, k_t(L_::w1 * (1.0 - L_::trace)), Ka);
          Kd = mad(fS, k_t(L_::w1 * L_::kd * (2.0 - L_::trace)), Kd);
          K0 = mad(fS, k_t(-L_::w0 * L_::trace), K0);
        }
        const R k1 = mul(ir, k_t(3.0 * L_::w1)), k2 = mul(fco, k_t(3.0 * L_::w1));
        const R a1 = mul(k1, k_t(1.5)), b1 = mul(k2, k_t(3));
        R X[D], V[D], Xd[D], Vd[D];
#pragma unroll
        for (int k = 0; k < D; k++) {
          X[k] = mad(a1, u[k], b1 * Ft[k]);
          V[k] = mad(k1, u[k], k2 * Gf[k]);
          Xd[k] = mul(X[k], k_t(L_::kd));
          Vd[k] = mul(V[k], k_t(L_::kd));
        }
        push<false>(a, out, P, n, nb, 0, mad(f[0], omi, K0));
#pragma unroll
        for (int k = 0; k < NP; k++) {
          const int i = L_::first(k), o = L_::opp(i);
          R Ps, Pa;
          if (is_axis<D>(k)) {
            Ps = mad(u[k < D ? k : 0], X[k < D ? k : 0], Ka);
            Pa = V[k < D ? k : 0];
          } else {
            R cX = R(0);
            Pa = R(0);
            bool any = false;
#pragma unroll
            for (int q = 0; q < D; q++) {
              const int cc = L_::c(i, q);
              if (cc == 0) continue;
              cX = any ? (cc > 0 ? cX + Xd[q] : cX - Xd[q]) : (cc > 0 ? Xd[q] : -Xd[q]);
              Pa = any ? (cc > 0 ? Pa + Vd[q] : Pa - Vd[q]) : (cc > 0 ? Vd[q] : -Vd[q]);
              any = true;
            }
            Ps = mad(cud[k < D ? 0 : k - D], cX, Kd);
          }
          push<false>(a, out, P, n, nb, i, mad(f[i], omi, Ps) + Pa);
          push<false>(a, out, P, n, nb, o, mad(f[o], omi, Ps) - Pa);
        }
      }

      // ---- phase-field collision Eqs. (18)-(20) --------------------------------
      if (lat & LAT_PHASE) {
        R gq[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) gq[i] = a.pin[(Q + i) * P + n];
        if (DIAG) bad = bad || !finite_word(sum_pops<D, false>(gq));
        const R src = mul(phi * mdot, c.gcoef);
        const R em = mul(mu, c.itg_eta);
        const R Zs = em + src;
        const R Za = mul(Zs, k_t(L_::w1)), Zd = mul(Zs, k_t(L_::w1 * L_::kd));
        R V[D], Vd[D];
#pragma unroll
        for (int k = 0; k < D; k++) {
          const R old = a.lin[(G_::PHU + k) * P + n];
          V[k] = mad(old, -c.v_old, mul(phu[k], c.v_new));
          Vd[k] = mul(V[k], k_t(L_::kd));
        }
        // itg (phi + (w_0 - 1) eta mu) + w_0 gcoef phi mdot
        if constexpr (std::is_same<R, float>::value) {
          // the small terms first: one rounding at the size of phi
          const R r0 = mad(gq[0], c.omg, mad(Zs, k_t(L_::w0), -em));
          push<false>(a, out + Q * P, P, n, nb, 0, mad(phi, c.itg, r0));
        } else {
          // itg times the equilibrium is rounded by itself, as in the fused
          // tile.  In the gas beside a solid phi = -(1 - phi0) to the last bit, and
          // an ulp decides whether the clamp of w passes a derivative: with one
          // rounding fewer (phi 8 % nearer to an 80-bit solution, two
          // instructions of 291 less) d/dg_y of sweeps under 30 steps is 1e-11 to
          // 2e-9 away from that form's.
          const R eq0 = mad(mul(mu, c.eta), k_t(L_::w0 - 1.0), phi);
          const R r0 = mad(gq[0], c.omg, mul_rn(eq0, c.itg));
          push<false>(a, out + Q * P, P, n, nb, 0, mad(src, k_t(L_::w0), r0));
        }
#pragma unroll
        for (int k = 0; k < NP; k++) {
          const int i = L_::first(k), o = L_::opp(i);
          R Pa = R(0);
          if (is_axis<D>(k)) {
            Pa = V[k < D ? k : 0];
          } else {
            bool any = false;
#pragma unroll
            for (int q = 0; q < D; q++) {
              const int cc = L_::c(i, q);
              if (cc == 0) continue;
              Pa = any ? (cc > 0 ? Pa + Vd[q] : Pa - Vd[q]) : (cc > 0 ? Vd[q] : -Vd[q]);
              any = true;
            }
          }
          const R Z = is_axis<D>(k) ? Za : Zd;
          push<false>(a, out + Q * P, P, n, nb, i, mad(gq[i], c.omg, Z) + Pa);
          push<false>(a, out + Q * P, P, n, nb, o, mad(gq[o], c.omg, Z) - Pa);
        }
      }

      lbmk::allow_next();
      // ---- enthalpy TRT collision Eqs. (23)-(27) --------------------------------
      R CTm = R(0);
      if (lat & LAT_HEAT) {
        R hq[Q];
        if (g.has_mask && a.mask[n]) {
          cold_node<D>(c, a.lin[G_::W * P + n], phi0, hq);
        } else {
#pragma unroll
          for (int i = 0; i < Q; i++) hq[i] = a.pin[(2 * Q + i) * P + n];
        }
        if (DIAG) bad = bad || !finite_word(rhoH);
        // By the magic relation 1/tau_s = 2 - 1/tau_a the collision is
        // h_i* = q_i + (1/tau_a - 1) (h_o - q_o), o the opposite of i, with
        // q = h_eq + w C T mdot / 2 (the source's factor 1 - 1/(2 tau_a) is
        // half of 1/tau_s): a population at q stays there exactly
        const R am = add(rcp(mad(mix(c.lam), c.inv_rr3, k_t(0.5))), k_t(-1));
        const R CT = rho * mix(c.cp) * T;
        CTm = CT * mdot;
        const R rrT = mul(T, c.rr);
        const R Kn = mad(CTm, k_t(0.5), mad(mul(CT, k_t(-1.5)), uu, rrT));
        const R Ka = mul(Kn, k_t(L_::w1)), Kd = mul(Kn, k_t(L_::w1 * L_::kd));
        const R ya = mul(CT, k_t(4.5 * L_::w1)), yd = mul(ya, k_t(L_::kd));
        const R za = mul(CT, k_t(3.0 * L_::w1)), zd = mul(za, k_t(L_::kd));
        {
          const R q0 = mad(Kn, k_t(L_::w0), rhoH - rrT);
          push<true>(a, out + 2 * Q * P, P, n, nb, 0, mad(hq[0] - q0, am, q0));
        }
#pragma unroll
        for (int k = 0; k < NP; k++) {
          const int i = L_::first(k), o = L_::opp(i);
          R Ps, Pa;
          if (is_axis<D>(k)) {
            const R cu = u[k < D ? k : 0];
            Ps = mad(cu * cu, ya, Ka);
            Pa = za * cu;
          } else {
            const R cu = cud[k < D ? 0 : k - D];
            Ps = mad(cu * cu, yd, Kd);
            Pa = zd * cu;
          }
          const R qi = Ps + Pa, qo = Ps - Pa;
          push<true>(a, out + 2 * Q * P, P, n, nb, i, mad(hq[o] - qo, am, qi));
          push<true>(a, out + 2 * Q * P, P, n, nb, o, mad(hq[i] - qi, am, qo));
        }
      }
      if (DIAG && (lat & LAT_FLOW)) bad = bad || !finite_word(ftot);
      a.lout[G_::P * P + n] = pr;
#pragma unroll
      for (int k = 0; k < D; k++)
        a.lout[(G_::PHU + k) * P + n] = (lat & LAT_PHASE) ? phu[k] : R(0);
      a.lout[G_::Q * P + n] = CTm;
    }
  }
  if constexpr (DIAG) warp_diag(a.diag, a.nwarps, wid, dv, bad);
}

// node ids linear over the grid
template <typename R, int D, int LATC, typename I>
__device__ __forceinline__ void node_local_linear(const NodeArgs<R, D>& a, int id) {
  if (id < a.g.nodes) node_local<R, D, LATC, I>(a, node_pos<D>(a.g, id).n);
}
template <typename R, int D, int LATC, bool READ, bool DIAG, typename I>
__device__ __forceinline__ void node_collide_linear(const NodeArgs<R, D>& a, const ReadOut* ro,
                                                    int id) {
  const bool valid = id < a.g.nodes;
  node_collide<R, D, LATC, READ, DIAG, I>(a, ro, valid, node_pos<D>(a.g, valid ? id : 0), id >> 5);
}

}  // namespace lbmn
