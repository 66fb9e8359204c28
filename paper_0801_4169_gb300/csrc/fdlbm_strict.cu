// fdlbm_strict.cu -- FDLBM_FP64_STRICT: the FP64 method in one canonical order of operations.
//
// Every value is formed from its defining equation one IEEE-754 FP64 operation at a time, in the
// order written below, each with an explicitly rounded intrinsic (__dadd_rn, __dsub_rn, __dmul_rn,
// __ddiv_rn, __dsqrt_rn): nothing is fused into a multiply-add, reassociated or replaced by a
// reciprocal. Any IEEE FP64 program that takes the same operations in the same order therefore
// produces the same bits, on any machine and under any compiler that keeps IEEE semantics.
//
//   velocities (Eq. 1)    v_q = v_k (cos, sin)(i pi/4) with the components 0, +-1, +-sqrt(1/2);
//                          q = 0 rest, q = 1 + 8k + d for ring k (speed v_{k+1}), angle (d + 1) pi/4.
//   moments (Eqs. 3-5)    n, jx, jy summed over q = 0..32 in turn (each product rounded before
//                          its sum); u = j / n; P = sum over q of ((1/2)(wx^2 + wy^2)) f_q with
//                          w = v_q - u; T = P / n (m = 1, so theta = T).
//   weights (Eqs. 11-13)  with a, b, c the squared speeds of the cyclic indices k+1, k+2, k+3:
//                          F_k = (((48 th^4 - (6 ((a + b) + c)) th^3) + (((ab + bc) + ca)) th^2)
//                                 - ((ab)c / 4) th) / (((v_k^2 (v_k^2 - a))(v_k^2 - b))(v_k^2 - c)),
//                          th^2 = th th, th^3 = th^2 th, th^4 = th^3 th; F_0 = 1 - 8 (((F_1 + F_2) + F_3) + F_4).
//   equilibrium (Eq. 10)  (n F_k) ((((t0 + t1) + t2) + t3) + t4) with h = 1 - u^2 / (2 th),
//                          t0 = h + u^4 / ((8 th) th), t1 = (v.u / th) h, t2 = ((v.u)^2 / ((2 th) th)) h,
//                          t3 = (v.u)^3 / (((6 th) th) th), t4 = (v.u)^4 / ((((24 th) th) th) th),
//                          powers by repeated products from the left, u^2 = ux ux + uy uy.
//   update (Eq. 17)       acc = f - r (f - f_eq), r = dt / tau; then for alpha = x, y in turn, with
//                          c = (v_alpha dt) / dr_alpha, kappa = (u_alpha dt) / dr_alpha:
//                          acc - (c / 2)(f+1 - f-1)                                       line I
//                          acc + ((c c) / 2)((f+1 - 2 f) + f-1)                           line II
//                          acc + ((c (1 - c c)) / 12)(((f+2 - 2 f+1) + 2 f-1) - f-2)      line III
//                          acc + (((theta_a |kappa|)(1 - |kappa|)) / 2)((f+1 - 2 f) + f-1) line IV
//                          theta_a = lambda |((P+ - 2 P0) + P-) / ((P+ + 2 P0) + P-)| (Eq. 16),
//                          P = n T at I+1, I, I-1 along alpha.
//
// Two launches per step: the moments of every node that the update reads (the interior and the ghost layer
// next to each edge) into the moment buffer, then the update of every interior node with the ghost copies it
// owns (periodic, zero-gradient, mirror). Dirichlet ghosts, the initial condition and boundary segments take
// the same f_eq.
//
// The step is bound by the FP64 pipe, and with every operation above taken as written for every node and
// velocity, most of it were divisions (300 x 75: 434 us per step; 192 now). The same bits come from fewer operations:
//   - c and what Eq. 17 forms from it alone depend on the velocity and the axis, not on the node: the host
//     forms them once per launch, with the same operations; a negative component only changes signs;
//   - opposite velocities have v.u of opposite sign and the same magnitude, so one set of quotients serves both;
//   - a quotient by theta, 2 theta^2, 6 theta^3 or 24 theta^4 is a q1 = q0 + (a - b q0) y step from the correctly
//     rounded y = 1/b, taken twice; by Markstein's theorem (IBM J. Res. Dev. 34, 1990) the second is the
//     correctly rounded quotient. Operands outside 2^+-600 and b outside 2^+-210 take the division.
// The update has one thread for each node and velocity ring, since a small grid has too few nodes to fill the
// schedulers evenly.
#include <cmath>

#include "fdlbm_kernels.cuh"

namespace fdlbm {

namespace {
namespace strict {

__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dvd(double a, double b) { return __ddiv_rn(a, b); }

// v_q of Eq. 1 (see the header comment for the ordering)
__device__ __forceinline__ void vel(int q, double& vx, double& vy) {
  if (q == 0) {
    vx = 0.0;
    vy = 0.0;
    return;
  }
  const int k = (q - 1) / 8, d = (q - 1) % 8;
  const double s = __dsqrt_rn(0.5);
  double cx, cy;
  switch (d) {
    case 0: cx = s; cy = s; break;        // 45 deg
    case 1: cx = 0.0; cy = 1.0; break;    // 90 deg
    case 2: cx = -s; cy = s; break;       // 135 deg
    case 3: cx = -1.0; cy = 0.0; break;   // 180 deg
    case 4: cx = -s; cy = -s; break;      // 225 deg
    case 5: cx = 0.0; cy = -1.0; break;   // 270 deg
    case 6: cx = s; cy = -s; break;       // 315 deg
    default: cx = 1.0; cy = 0.0; break;   // 0 deg
  }
  vx = mul(speed(k), cx);
  vy = mul(speed(k), cy);
}

// F_0..F_4 of Eqs. 11-13 at theta
__device__ __forceinline__ void weights(double th, double (&F)[5]) {
  double sumF = 0.0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double vk = speed(k), va = speed((k + 1) % 4), vb = speed((k + 2) % 4), vc = speed((k + 3) % 4);
    const double vk2 = mul(vk, vk), a = mul(va, va), b = mul(vb, vb), c = mul(vc, vc);
    const double den = mul(mul(mul(vk2, sub(vk2, a)), sub(vk2, b)), sub(vk2, c));
    const double t2 = mul(th, th), t3 = mul(t2, th), t4 = mul(t3, th);
    const double num = sub(add(sub(mul(48.0, t4), mul(mul(6.0, add(add(a, b), c)), t3)),
                               mul(add(add(mul(a, b), mul(b, c)), mul(c, a)), t2)),
                           mul(dvd(mul(mul(a, b), c), 4.0), th));
    F[k + 1] = dvd(num, den);
    sumF = add(sumF, F[k + 1]);
  }
  F[0] = sub(1.0, mul(8.0, sumF));
}

// f_eq of velocity q (Eq. 10)
__device__ __forceinline__ double feq(int q, double n, double ux, double uy, double th, const double (&F)[5]) {
  double vx, vy;
  vel(q, vx, vy);
  const double Fk = F[q == 0 ? 0 : 1 + (q - 1) / 8];
  const double u2 = add(mul(ux, ux), mul(uy, uy));
  const double vu = add(mul(vx, ux), mul(vy, uy));
  const double h = sub(1.0, dvd(u2, mul(2.0, th)));
  const double t0 = add(h, dvd(mul(u2, u2), mul(mul(8.0, th), th)));
  const double t1 = mul(dvd(vu, th), h);
  const double t2 = mul(dvd(mul(vu, vu), mul(mul(2.0, th), th)), h);
  const double t3 = dvd(mul(mul(vu, vu), vu), mul(mul(mul(6.0, th), th), th));
  const double t4 = dvd(mul(mul(mul(vu, vu), vu), vu), mul(mul(mul(mul(24.0, th), th), th), th));
  return mul(mul(n, Fk), add(add(add(add(t0, t1), t2), t3), t4));
}

struct Mac {
  double n, ux, uy, T;
};

// Eqs. 3-5 at the node at offset off
__device__ __forceinline__ Mac moments(const double* __restrict__ f, long long plane, long long off) {
  double x[Q];
  double n = 0.0, jx = 0.0, jy = 0.0;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    x[q] = f[(long long)q * plane + off];
    double vx, vy;
    vel(q, vx, vy);
    n = add(n, x[q]);
    jx = add(jx, mul(vx, x[q]));
    jy = add(jy, mul(vy, x[q]));
  }
  Mac m;
  m.n = n;
  m.ux = dvd(jx, n);
  m.uy = dvd(jy, n);
  double P = 0.0;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    double vx, vy;
    vel(q, vx, vy);
    const double wx = sub(vx, m.ux), wy = sub(vy, m.uy);
    P = add(P, mul(mul(0.5, add(mul(wx, wx), mul(wy, wy))), x[q]));
  }
  m.T = dvd(P, n);
  return m;
}

__device__ __forceinline__ bool mac_ok(const Mac& m) {
  return isfinite(m.n) && isfinite(m.ux) && isfinite(m.uy) && isfinite(m.T) && m.n > 0.0 && m.T > 0.0;
}

// Scheme parameters and what the host forms from them, in the order above: F_k's numerator coefficients and
// denominator, and c/2, (c c)/2, (c (1 - c c))/12 for axis a, ring k, l = 0 along the axis, 1 diagonal.
struct Params {
  double dt, dr[2], lam, r;
  double w3[4], w2[4], w1[4], den[4];
  double c1[2][4][2], c2[2][4][2], c3[2][4][2];
  int flags;
};

__device__ __noinline__ double dvd_rare(double a, double b) { return dvd(a, b); }
// a / b for b in 2^+-210, y = 1/b rounded to nearest
__device__ __forceinline__ double dvd_by(double a, double b, double y) {
  const unsigned ah = (unsigned)__double2hiint(a) & 0x7fffffffu;
  if (__builtin_expect(ah - ((1023u - 600u) << 20) >= 1200u << 20, 0))
    return (ah | (unsigned)__double2loint(a)) ? dvd_rare(a, b) : a;  // b > 0: a zero keeps its sign
  const double q0 = mul(a, y);
  const double q1 = __fma_rn(__fma_rn(-b, q0, a), y, q0);
  return __fma_rn(__fma_rn(-b, q1, a), y, q1);
}

// What Eq. 10 shares between a node's velocities
struct EqNode {
  double t0, h, b[4], y[4];
  bool near;  // theta in 2^+-50: dvd_by
};
__device__ __forceinline__ EqNode eq_node(double ux, double uy, double th) {
  EqNode e;
  const double u2 = add(mul(ux, ux), mul(uy, uy));
  e.h = sub(1.0, dvd(u2, mul(2.0, th)));
  e.t0 = add(e.h, dvd(mul(u2, u2), mul(mul(8.0, th), th)));
  e.b[0] = th;
  e.b[1] = mul(mul(2.0, th), th);
  e.b[2] = mul(mul(mul(6.0, th), th), th);
  e.b[3] = mul(mul(mul(mul(24.0, th), th), th), th);
  const unsigned hi = (unsigned)__double2hiint(th);
  e.near = hi - ((1023u - 50u) << 20) < 100u << 20;
#pragma unroll
  for (int i = 0; i < 4; ++i) e.y[i] = e.near ? __drcp_rn(e.b[i]) : 0.0;
  return e;
}
// The bracket of Eq. 10 for v.u = vu and for -vu
__device__ __forceinline__ void brackets(const EqNode& e, double vu, double& plus, double& minus) {
  const double p2 = mul(vu, vu), p3 = mul(p2, vu), p4 = mul(p3, vu);
  double q1, q2, q3, q4;
  if (__builtin_expect(e.near, 1)) {
    q1 = dvd_by(vu, e.b[0], e.y[0]);
    q2 = dvd_by(p2, e.b[1], e.y[1]);
    q3 = dvd_by(p3, e.b[2], e.y[2]);
    q4 = dvd_by(p4, e.b[3], e.y[3]);
  } else {
    q1 = dvd_rare(vu, e.b[0]);
    q2 = dvd_rare(p2, e.b[1]);
    q3 = dvd_rare(p3, e.b[2]);
    q4 = dvd_rare(p4, e.b[3]);
  }
  const double t1 = mul(q1, e.h), t2 = mul(q2, e.h);
  plus = add(add(add(add(e.t0, t1), t2), q3), q4);
  minus = add(sub(add(sub(e.t0, t1), t2), q3), q4);
}
__device__ __forceinline__ double weight(const Params& p, int k, double th, double t2, double t3, double t4) {
  return dvd(sub(add(sub(mul(48.0, t4), mul(p.w3[k], t3)), mul(p.w2[k], t2)), mul(p.w1[k], th)), p.den[k]);
}

// Eq. 17 for one velocity with component signs XS, YS (fq: its plane at the node), fe its f_eq, nuh line IV's factor.
template <int XS, int YS>
__device__ __forceinline__ double update_one(const double* __restrict__ fq, int pitch, const Params& p, int k,
                                             double fe, const double (&nuh)[2]) {
  constexpr int l = XS != 0 && YS != 0;
  const double f0 = fq[0];
  double acc = sub(f0, mul(p.r, sub(f0, fe)));
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int sg = a == 0 ? XS : YS, st = a == 0 ? 1 : pitch;
    const double c1 = sg == 0 ? 0.0 : p.c1[a][k][l], c2 = sg == 0 ? 0.0 : p.c2[a][k][l], c3 = sg == 0 ? 0.0 : p.c3[a][k][l];
    const double fp1 = fq[st], fm1 = fq[-st], fp2 = fq[2 * st], fm2 = fq[-2 * st];
    const double cu = add(sub(fp1, mul(2.0, f0)), fm1);
    acc = sub(acc, mul(sg < 0 ? -c1 : c1, sub(fp1, fm1)));
    if (!(p.flags & F_NO_LW)) acc = add(acc, mul(c2, cu));
    if (!(p.flags & F_NO_DISP))
      acc = add(acc, mul(sg < 0 ? -c3 : c3, sub(add(sub(fp2, mul(2.0, fp1)), mul(2.0, fm1)), fm2)));
    if (!(p.flags & F_NO_VISC)) acc = add(acc, mul(nuh[a], cu));
  }
  return acc;
}

template <int QQ>
__device__ __forceinline__ void feq_one(double* __restrict__ f, const Grid& g, int gx, int gy, const GhostOwn& go,
                                        double n, double ux, double uy, double T, const double (&F)[5]) {
  store_node<double, QQ>(f, g, gx, gy, go, feq(QQ, n, ux, uy, T, F));
}
template <int... QS>
__device__ __forceinline__ void feq_all(double* __restrict__ f, const Grid& g, int gx, int gy, const GhostOwn& go,
                                        double n, double ux, double uy, double T) {
  double F[5];
  weights(T, F);
  (feq_one<QS>(f, g, gx, gy, go, n, ux, uy, T, F), ...);
}
__device__ __forceinline__ void write_feq(double* __restrict__ f, const Grid& g, int gx, int gy, const GhostOwn& go,
                                          double n, double ux, double uy, double T) {
  feq_all<0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 21, 22, 23, 24, 25, 26, 27, 28,
          29, 30, 31, 32>(f, g, gx, gy, go, n, ux, uy, T);
}

// Moment-buffer planes (the grid's split-step buffer): n, ux, uy, T.
__device__ __forceinline__ double* mplane(const Grid& g, int a) { return static_cast<double*>(g.mom) + a * g.plane; }

// Pass 1: moments of the interior and of the ghost layer next to each edge (no corners).
__global__ void k_moments(const double* __restrict__ f, Grid g, unsigned* __restrict__ health) {
  const int gx = blockIdx.x * blockDim.x + threadIdx.x - 1, gy = blockIdx.y * blockDim.y + threadIdx.y - 1;
  if (gx > g.nx || gy > g.ny || !ring_node_needed(g, gx, gy)) return;
  const long long off = (long long)(gy + NG) * g.pitch + (gx + NG);
  const Mac m = moments(f, g.plane, off);
  if (!mac_ok(m)) atomicOr(health, H_NUMERIC);
  mplane(g, 0)[off] = m.n;
  mplane(g, 1)[off] = m.ux;
  mplane(g, 2)[off] = m.uy;
  mplane(g, 3)[off] = m.T;
}

// Pass 2: Eq. 17 at every interior node, a warp for 32 nodes of a row and one ring (threadIdx.y).
__global__ void __launch_bounds__(128) k_update(const double* __restrict__ f, double* __restrict__ fn, Grid g,
                                                Params p, unsigned* __restrict__ health) {
  const int gx = blockIdx.x * 32 + threadIdx.x, gy = blockIdx.y + blockIdx.z * gridDim.y, K = threadIdx.y;
  if (gx >= g.nx || gy >= g.ny) return;
  const long long off = (long long)(gy + NG) * g.pitch + (gx + NG);
  const double* Mn = mplane(g, 0);
  const double* MT = mplane(g, 3);
  Mac m;
  m.n = Mn[off];
  m.ux = mplane(g, 1)[off];
  m.uy = mplane(g, 2)[off];
  m.T = MT[off];
  double nuh[2];
  unsigned bits = 0;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const long long st = a == 0 ? 1 : g.pitch;
    const double Pp = mul(Mn[off + st], MT[off + st]);
    const double P0 = mul(m.n, m.T);
    const double Pm = mul(Mn[off - st], MT[off - st]);
    const double sw = (p.flags & F_SWITCH_CONST)
                          ? p.lam
                          : mul(p.lam, fabs(dvd(add(sub(Pp, mul(2.0, P0)), Pm), add(add(Pp, mul(2.0, P0)), Pm))));
    const double ak = fabs(dvd(mul(a == 0 ? m.ux : m.uy, p.dt), p.dr[a]));
    if (ak > 1.0) bits |= H_KAPPA;
    nuh[a] = mul(mul(mul(sw, ak), sub(1.0, ak)), 0.5);
  }
  const GhostOwn go = ghost_own(g, gx, gy);
  const EqNode e = eq_node(m.ux, m.uy, m.T);
  const double t2 = mul(m.T, m.T), t3 = mul(t2, m.T), t4 = mul(t3, m.T);
  double Fk;
  if (K == 0) {  // and the rest velocity, whose weight needs all four
    double sumF = 0.0;
    Fk = weight(p, 0, m.T, t2, t3, t4);
    sumF = add(sumF, Fk);
#pragma unroll 1
    for (int k = 1; k < 4; ++k) sumF = add(sumF, weight(p, k, m.T, t2, t3, t4));
    double b0, unused;
    brackets(e, add(mul(0.0, m.ux), mul(0.0, m.uy)), b0, unused);
    const double fe = mul(mul(m.n, sub(1.0, mul(8.0, sumF))), b0);
    store_node<double, 0>(fn, g, gx, gy, go, update_one<0, 0>(f + off, g.pitch, p, 0, fe, nuh));
  } else {
    Fk = weight(p, K, m.T, t2, t3, t4);
  }
  const double nF = mul(m.n, Fk), v = speed(K), vd = mul(v, __dsqrt_rn(0.5));
  const double* fr = f + (long long)(1 + 8 * K) * g.plane + off;
  double out[8];
  auto pair = [&](auto xs, auto ys, int dp, int dm, double vu) {
    constexpr int X = decltype(xs)::value, Y = decltype(ys)::value;
    double bp, bm;
    brackets(e, vu, bp, bm);
    out[dp] = update_one<X, Y>(fr + dp * g.plane, g.pitch, p, K, mul(nF, bp), nuh);
    out[dm] = update_one<-X, -Y>(fr + dm * g.plane, g.pitch, p, K, mul(nF, bm), nuh);
  };
  using P = std::integral_constant<int, 1>;
  using Z = std::integral_constant<int, 0>;
  using M = std::integral_constant<int, -1>;
  pair(P{}, Z{}, 7, 3, add(mul(v, m.ux), mul(0.0, m.uy)));
  pair(P{}, P{}, 0, 4, add(mul(vd, m.ux), mul(vd, m.uy)));
  pair(Z{}, P{}, 1, 5, add(mul(0.0, m.ux), mul(v, m.uy)));
  pair(M{}, P{}, 2, 6, add(mul(-vd, m.ux), mul(vd, m.uy)));
  store_ring<double>(fn, g, gx, gy, go, K, out);
  if (bits) atomicOr(health, bits);
}

__global__ void k_init(double* __restrict__ f, Grid g, const double* __restrict__ rho, const double* __restrict__ u,
                       const double* __restrict__ v, const double* __restrict__ T) {
  const int gx = blockIdx.x * blockDim.x + threadIdx.x, gy = blockIdx.y * blockDim.y + threadIdx.y;
  if (gx >= g.nx || gy >= g.ny) return;
  const long long i = (long long)gy * g.nx + gx;
  write_feq(f, g, gx, gy, ghost_own(g, gx, gy), rho[i], u[i], v[i], T[i]);
}

// the ghost node t of a side's two layers (t < 2 len): coordinates and index along the side
__device__ __forceinline__ void side_ghost(const Grid& g, int side, int t, int& gx, int& gy, int& along) {
  const int len = side < 2 ? g.ny : g.nx;
  along = t % len;
  const int layer = t / len;
  if (side == 0) { gx = -1 - layer; gy = along; }
  else if (side == 1) { gx = g.nx + layer; gy = along; }
  else if (side == 2) { gx = along; gy = -1 - layer; }
  else { gx = along; gy = g.ny + layer; }
}

__global__ void k_dirichlet(double* __restrict__ f, Grid g, BState bs) {
  const int side = blockIdx.y;
  if (g.bc[side] != BC_DIRICHLET) return;
  const int len = side < 2 ? g.ny : g.nx;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * len) return;
  int gx, gy, along;
  side_ghost(g, side, t, gx, gy, along);
  GhostOwn none;
  none.mx = 0;
  none.my = 0;
  write_feq(f, g, gx, gy, none, bs.s[side][0], bs.s[side][1], bs.s[side][2], bs.s[side][3]);
}

__global__ void k_segment(double* __restrict__ f, Grid g, Segment sg, double d) {
  const int len = sg.side < 2 ? g.ny : g.nx;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * len) return;
  int gx, gy, along;
  side_ghost(g, sg.side, t, gx, gy, along);
  const double pos = mul(add((double)along, 0.5), d);
  const bool in = sg.lower ? (pos < sg.split) : !(pos < sg.split);
  if (!in && !sg.base_dirichlet) return;
  const double* st = in ? sg.seg : sg.base;
  GhostOwn none;
  none.mx = 0;
  none.my = 0;
  write_feq(f, g, gx, gy, none, st[0], st[1], st[2], st[3]);
}

__global__ void k_macro(const double* __restrict__ f, Grid g, double* __restrict__ rho, double* __restrict__ u,
                        double* __restrict__ v, double* __restrict__ T) {
  const int gx = blockIdx.x * blockDim.x + threadIdx.x, gy = blockIdx.y * blockDim.y + threadIdx.y;
  if (gx >= g.nx || gy >= g.ny) return;
  const Mac m = moments(f, g.plane, (long long)(gy + NG) * g.pitch + (gx + NG));
  const long long o = (long long)gy * g.nx + gx;
  rho[o] = m.n;
  u[o] = m.ux;
  v[o] = m.uy;
  T[o] = m.T;
}

}  // namespace strict
}  // namespace

// Params with the header's operations, each rounded by itself on every host (no contraction).
static strict::Params strict_params(const Grid& g, const Coeffs& c) {
  auto mul = [](double a, double b) { volatile double r = a * b; return (double)r; };
  auto add = [](double a, double b) { volatile double r = a + b; return (double)r; };
  auto sub = [](double a, double b) { volatile double r = a - b; return (double)r; };
  strict::Params p;
  p.dt = c.sdt;
  p.dr[0] = c.sdr[0];
  p.dr[1] = c.sdr[1];
  p.lam = c.lam;
  p.r = c.sdt / c.stau;
  p.flags = g.flags;
  const double s = std::sqrt(0.5);
  for (int k = 0; k < 4; ++k) {
    const double v = speed(k), va = speed((k + 1) % 4), vb = speed((k + 2) % 4), vc = speed((k + 3) % 4);
    const double v2 = mul(v, v), a = mul(va, va), b = mul(vb, vb), d = mul(vc, vc);
    p.den[k] = mul(mul(mul(v2, sub(v2, a)), sub(v2, b)), sub(v2, d));
    p.w3[k] = mul(6.0, add(add(a, b), d));
    p.w2[k] = add(add(mul(a, b), mul(b, d)), mul(d, a));
    p.w1[k] = mul(mul(a, b), d) / 4.0;
    for (int ax = 0; ax < 2; ++ax)
      for (int l = 0; l < 2; ++l) {
        const double cc = mul(l == 0 ? v : mul(v, s), c.sdt) / p.dr[ax];
        p.c1[ax][k][l] = cc / 2.0;
        p.c2[ax][k][l] = mul(cc, cc) / 2.0;
        p.c3[ax][k][l] = mul(cc, sub(1.0, mul(cc, cc))) / 12.0;
      }
  }
  return p;
}

cudaError_t launch_step_strict(const void* f, void* fn, const Grid& g, const Coeffs& c, unsigned* health,
                               cudaStream_t s) {
  if (!g.mom) return cudaErrorInvalidValue;
  const strict::Params p = strict_params(g, c);
  dim3 mb(32, 4), mg((g.nx + 2 + 31) / 32, (g.ny + 2 + 3) / 4);
  strict::k_moments<<<mg, mb, 0, s>>>(static_cast<const double*>(f), g, health);
  const unsigned rows = (unsigned)g.ny < 65535u ? (unsigned)g.ny : 65535u;
  const dim3 ug((unsigned)((g.nx + 31) / 32), rows, ((unsigned)g.ny + rows - 1u) / rows);
  strict::k_update<<<ug, dim3(32, 4), 0, s>>>(static_cast<const double*>(f), static_cast<double*>(fn), g, p, health);
  return cudaGetLastError();
}

cudaError_t launch_init_strict(void* f, const Grid& g, const double* rho, const double* u, const double* v,
                               const double* T, cudaStream_t s) {
  dim3 b(32, 4);
  strict::k_init<<<grid2d(g, b), b, 0, s>>>(static_cast<double*>(f), g, rho, u, v, T);
  return cudaGetLastError();
}

cudaError_t launch_dirichlet_strict(void* f, const Grid& g, const double bstate[4][4], cudaStream_t s) {
  BState bs;
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) bs.s[i][j] = bstate[i][j];
  const int len = 2 * (g.nx > g.ny ? g.nx : g.ny);
  dim3 b(128), grid((len + 127) / 128, 4);
  strict::k_dirichlet<<<grid, b, 0, s>>>(static_cast<double*>(f), g, bs);
  return cudaGetLastError();
}

cudaError_t launch_segment_strict(void* f, const Grid& g, const Segment& sg, double dx, double dy, cudaStream_t s) {
  const int len = sg.side < 2 ? g.ny : g.nx;
  dim3 b(128), grid((2 * len + 127) / 128);
  strict::k_segment<<<grid, b, 0, s>>>(static_cast<double*>(f), g, sg, sg.side < 2 ? dy : dx);
  return cudaGetLastError();
}

cudaError_t launch_macro_strict(const void* f, const Grid& g, double* rho, double* u, double* v, double* T,
                                cudaStream_t s) {
  dim3 b(32, 4);
  strict::k_macro<<<grid2d(g, b), b, 0, s>>>(static_cast<const double*>(f), g, rho, u, v, T);
  return cudaGetLastError();
}

}  // namespace fdlbm
