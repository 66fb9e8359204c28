#pragma once
// fdlbm_fx64.cuh -- the FP64-storage step with its moments, equilibrium and stencils in fixed point.
//
// What bounds this step. An FP64 instruction issues at 2 lanes/clk/SM here. The step in FP64 arithmetic
// (570 operations per site) kept that pipe 88% busy at 0.94-0.97 GLUPS, with HBM at 9%. The integer pipes run
// 32 times faster and a 60-bit fixed-point sum carries more bits than FP64's significand, so everything
// that is a sum of products of known range moves there:
//   moments   the 33 values aligned to the node's largest exponent (60 bits), exact integer sums;
//   f_eq      fdlbm_fx.cuh (brackets of 55-59 bits, one scale per ring);
//   Eq. 17    values and weights as 58-bit integers in two limbs of radix 2^28, three 32 x 32 + 64-bit
//             multiply-adds for each product, f_eq added at the same scale, one rounding to FP64.
// In FP64 remain the macros, the site constants, the weights F_k, the switch and nu: about 100 operations.
//
// Exponent classes. Values of a stencil enter with a common unit. A value's class is c = (E + 3) >> 2
// (E its biased exponent), its integer V = +-m 2^(E - 4c + 5) with m the 53-bit significand: exact,
// below 2^58, in units of 2^(4c - 1080). A plane's values are converted once per tile, into shared
// memory, and the nine values of a stencil combine directly where the tile's classes agree. Where a
// tile holds several classes of a plane (f crosses a power of 16, or zero) its cells stay FP64 numbers,
// and a stencil converts its nine values to their largest class itself (align_cells), rounding what drops
// out; where that one agrees throughout, the integers are the same. So a result depends on the node's nine
// values, its weights and its f_eq alone, not on the tile: every tile shape gives the same bits.
// The integers carry a few units of error whatever the weights are. Where a stencil's values differ by classes, a value
// that hardly counts can set the unit, so there a result has to have 2^45 units, or the node's density 2^49 of them; the
// FP64 form (stencils_f64) takes the others' place, as it does for values or weights outside the integers' range:
// infinities, NaN, exponents beyond 2^+-800, nu above the bound that the weights' scale leaves, weights that do not fit.
#include "fdlbm_kernels.cuh"

namespace fdlbm {
namespace {

using fx::s64;
using fx::u64;

// The values of f. With programmatic dependent launches a step's blocks are resident while the step before
// still writes them, which the read-only path of __ldg does not allow: an ordinary load, after the wait.
template <bool COH>
__device__ __forceinline__ double ldf(const double* p) {
  if constexpr (COH) return __ldcg(p);
  else return __ldca(p);
}

// ---------------------------------------------------------------------------------------------
// Moments: see node_moments for FP32 storage, whose scheme this is. The largest term's leading bit is
// bit 59; a term more than 2^7 below the largest loses the bits under the unit, less than 2^-59 of the
// largest value. Sums that can pass 2^63 are held as (H, L): H 2^32 + L, L unsigned.
struct Wide {
  s64 H, L;
};
__device__ __forceinline__ void wide_add(Wide& w, s64 v, int factor) {
  w.H = fx::mad((int)(v >> 32), factor, w.H);
  w.L = fx::mad_u((unsigned)v, (unsigned)factor, w.L);
}
// H 2^32 + L, times 2^ex, rounded to nearest even FP64 (ties decided on 64 bits). |H| < 2^62.
__device__ __forceinline__ double wide_to_f64(const Wide& w, int ex) {
  s64 H = w.H + (s64)((u64)w.L >> 32);
  unsigned lo = (unsigned)w.L;
  const s64 sg = H >> 63;
  H ^= sg;
  lo ^= (unsigned)sg;  // one's complement: one unit of the sums
  unsigned hi = (unsigned)((u64)H >> 32), mid = (unsigned)H;
  if (hi == 0u) {
    hi = mid;
    mid = lo;
    lo = 0u;
    ex -= 32;
    if (hi == 0u) {
      hi = mid;
      mid = 0u;
      ex -= 32;
    }
  }
  const int lg = fx::floor_log2(hi);
  const int sh = (31 - lg) & 31;
  const u64 U = ((u64)__funnelshift_l(mid, hi, sh) << 32) | __funnelshift_l(lo, mid, sh);  // leading one at bit 63
  const u64 M = ((U >> 1) + 0x1ffull + ((U >> 11) & 1ull)) >> 10;
  u64 r = ((u64)(1023 + 64 + lg + ex - 1) << 52) + M;
  if (lg < 0) r = 0ull;
  return __longlong_as_double((s64)(((u64)sg & 0x8000000000000000ull) | r));
}
// x aligned to the exponent emax: +-m 2^(7 - (emax - E)), rounded to odd (the last bit left is set where a set
// bit drops out), which has no sign and no bias however few bits drop: truncation would take half a unit of
// every smaller value, in every step. Of a zero (E = 0) the shift, at least kMomEmin, clears the hidden bit too.
constexpr int kMomEmin = 128;
constexpr int kMomUnit = 1082;  // a term's unit is 2^(emax - kMomUnit): emax - 1075 - 7
__device__ __forceinline__ s64 mom_term(double x, int emax) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int s = emax - (int)((hi & 0x7fffffffu) >> 20);
  const unsigned m = (hi & 0xfffffu) | 0x100000u;
  const unsigned l7 = lo << 7;
  const u64 v = fx::shr_clamped(((u64)__funnelshift_l(lo, m, 7) << 32) | l7, s) |
                (fx::shl_clamped(l7, max(32 - s, 0)) ? 1u : 0u);  // beyond s = 32: the low word's bits will do
  const s64 sg = (s64)((int)hi >> 31);
  return (s64)(v ^ (u64)sg) - sg;
}
struct RingSums {
  s64 S, AX, DX, AY, DY;
};
__device__ __forceinline__ RingSums ring_sums_fx(const double (&x)[8], int emax) {
  s64 t[8];
#pragma unroll
  for (int d = 0; d < 8; ++d) t[d] = mom_term(x[d], emax);
  RingSums r;
  r.S = ((t[0] + t[4]) + (t[2] + t[6])) + ((t[1] + t[5]) + (t[3] + t[7]));
  r.AX = t[7] - t[3];
  r.AY = t[1] - t[5];
  const s64 a = t[0] - t[4], b = t[6] - t[2];
  r.DX = a + b;
  r.DY = a - b;
  return r;
}
// The node's sums: N = sum f; Ax, Dx (Ay, Dy) = sum_k V_k AX_k, DX_k; E = sum_k V_k^2 S_k, V_k = 100 v_k.
struct NodeSums {
  Wide N, Ax, Dx, Ay, Dy, E;
};
__device__ __forceinline__ void add_ring(NodeSums& s, const RingSums& r, int V) {
  wide_add(s.N, r.S, 1);
  wide_add(s.Ax, r.AX, V);
  wide_add(s.Dx, r.DX, V);
  wide_add(s.Ay, r.AY, V);
  wide_add(s.Dy, r.DY, V);
  wide_add(s.E, r.S, V * V);
}
__device__ __forceinline__ Wide times_1e4(const Wide& w) {
  return Wide{fx::mad_small(10000u, w.H, 0), fx::mad_small(10000u, w.L, 0)};
}
// (n, u, T, P) from n, 10^4 n (rounded from the exact sum like n), 100 j and 10^4 sum |v|^2 f
__device__ __forceinline__ Macro macro_of(double n, double n4, double jx, double jy, double e2) {
  Macro o;
  const double i4 = rcp64(n4), ij = 100.0 * i4;
  o.n = n;
  o.ux = jx * ij;
  o.uy = jy * ij;
  const double u2 = fma(o.ux, o.ux, o.uy * o.uy);
  o.T = 0.5 * fma(e2, i4, -u2);
  o.P = n * o.T;
  return o;
}
__device__ __forceinline__ Macro macro_from_sums(const NodeSums& s, int ex) {
  return macro_of(wide_to_f64(s.N, ex), wide_to_f64(times_1e4(s.N), ex),
                  fma(kS, wide_to_f64(s.Dx, ex), wide_to_f64(s.Ax, ex)),
                  fma(kS, wide_to_f64(s.Dy, ex), wide_to_f64(s.Ay, ex)), wide_to_f64(s.E, ex));
}
// Values near the ends of the exponent range (infinities and NaN among them): the sums in FP64.
template <bool COH>
__device__ __noinline__ Macro node_macro_f64(const double* __restrict__ f, long long plane, long long off,
                                             const Coeffs& c) {
  double S[4], X[4], Y[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    double x[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) x[d] = ldf<COH>(f + (long long)(1 + 8 * k + d) * plane + off);
    ring_sums(x, S[k], X[k], Y[k]);
  }
  return to_macro<1>(combine_rings(ldf<COH>(f + off), S, X, Y, c));
}
// The largest sum, 33 x 449^2 times the largest value, stays below 2^1023: its exponent is written without a check.
__device__ __forceinline__ bool mom_range(int emax) { return emax >= kMomEmin && emax < 2047 - 25; }
template <bool COH>
__device__ __forceinline__ Macro node_macro_fx(const double* __restrict__ f, long long plane, long long off,
                                               const Coeffs& c) {
  double x[Q];
  unsigned amax = 0u;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    x[q] = ldf<COH>(f + (long long)q * plane + off);
    amax = max(amax, (unsigned)__double2hiint(x[q]) & 0x7fffffffu);
  }
  const int emax = (int)(amax >> 20);
  if (__builtin_expect(!mom_range(emax), 0)) return node_macro_f64<COH>(f, plane, off, c);
  NodeSums s{};
  wide_add(s.N, mom_term(x[0], emax), 1);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    double g[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) g[d] = x[1 + 8 * k + d];
    add_ring(s, ring_sums_fx(g, emax), speed_c(k));
  }
  return macro_from_sums(s, emax - kMomUnit);
}
// The four lanes of a quad, lane r summing ring r: integer sums, so in any order the same macros.
template <bool COH>
__device__ __forceinline__ Macro quad_macro_fx(const double* __restrict__ f, long long plane, long long off, int r,
                                               const Coeffs& c) {
  const unsigned ALL = 0xffffffffu;
  double x[8];
  const double x0 = ldf<COH>(f + off);
  unsigned amax = (unsigned)__double2hiint(x0) & 0x7fffffffu;
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    x[d] = ldf<COH>(f + (long long)(1 + 8 * r + d) * plane + off);
    amax = max(amax, (unsigned)__double2hiint(x[d]) & 0x7fffffffu);
  }
  amax = max(amax, __shfl_xor_sync(ALL, amax, 1));
  amax = max(amax, __shfl_xor_sync(ALL, amax, 2));
  const int emax = (int)(amax >> 20);
  NodeSums s{};
  if (r == 0) wide_add(s.N, mom_term(x0, emax), 1);
  add_ring(s, ring_sums_fx(x, emax), speed_c(r));
  auto sum = [&](Wide& w) {
#pragma unroll
    for (int lm = 1; lm <= 2; lm <<= 1) {
      w.H += __shfl_xor_sync(ALL, w.H, lm);
      w.L += __shfl_xor_sync(ALL, w.L, lm);
    }
  };
  sum(s.N);
  sum(s.Ax);
  sum(s.Dx);
  sum(s.Ay);
  sum(s.Dy);
  sum(s.E);
  // Lane 1 finishes jx, lane 2 jy, lane 0 n and the energy, lane 3 10^4 n: two conversions each, not seven
  const int ex = emax - kMomUnit;
  const Wide u = r == 1 ? s.Dx : r == 2 ? s.Dy : r == 0 ? s.E : times_1e4(s.N);
  const Wide v = r == 1 ? s.Ax : r == 2 ? s.Ay : s.N;
  const double a = wide_to_f64(u, ex), b = wide_to_f64(v, ex), j = fma(kS, a, b);
  const int q0 = (threadIdx.x & 31) & ~3;
  const double n = __shfl_sync(ALL, b, q0), e2 = __shfl_sync(ALL, a, q0), n4 = __shfl_sync(ALL, a, q0 + 3);
  const double jx = __shfl_sync(ALL, j, q0 + 1), jy = __shfl_sync(ALL, j, q0 + 2);
  if (__builtin_expect(!mom_range(emax), 0)) return node_macro_f64<COH>(f, plane, off, c);
  return macro_of(n, n4, jx, jy, e2);
}

// ---------------------------------------------------------------------------------------------
// The FP64 form of r f_eq of ring K, for nodes outside the fixed-point range: the directions of the mask, into their
// places in f_new (o: the node's entry of the ring's first plane).
__device__ __noinline__ void feq_f64(double n, double ux, double uy, double T, int K, unsigned mask, const Coeffs& c,
                                     double* __restrict__ o, long long plane) {
  EqSite e = eq_site(n, ux, uy, T, c);
  // the weight that the rest velocity's is formed from: another rounding of it would make mass
  e.nF[K] = weight_poly<true>(c.r * n * T, T, K, c);
  const EqRing r = eq_ring(e, K, c);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    double fp, fm;
    eq_pair(r, e.p[t], e.x[t], fp, fm);
    if (mask >> dir_plus(t) & 1u) o[dir_plus(t) * plane] = fp;
    if (mask >> dir_minus(t) & 1u) o[dir_minus(t) * plane] = fm;
  }
}

// The same from the pairs' integers, formed again (q: the lane's powers of the projections, stride between them).
// Out of line: kept for the slow directions in the ring's loop, they cost all others 4%.
__device__ __noinline__ void feq_slow(s64 A0f, int es, int e0, int ea, int ep, unsigned neg, int K, double nF,
                                      unsigned mask, const Coeffs& c, const int4* __restrict__ q, int stride,
                                      double* __restrict__ o, long long plane) {
  const fx::RingFx r = fx::ring_scaled(A0f, es, e0, ea, ep, K, nF, c.fxc[1][K]);
#pragma unroll 1
  for (int t = 0; t < 4; ++t) {
    const int dp = dir_plus(t), dm = dir_minus(t);
    if (!(mask & (1u << dp | 1u << dm))) continue;
    const int4 u = q[2 * t * stride], v = q[(2 * t + 1) * stride];
    s64 NE, NO;
    fx::pair_of<true>(r, fx::Dir{{u.x, u.y}, {u.z, u.w}, {v.x, v.y}, {v.z, v.w}}, NE, NO);
    if (neg >> t & 1u) NO = -NO;
    if (mask >> dp & 1u) o[dp * plane] = fx::to_f64(NE + NO, r.ex);
    if (mask >> dm & 1u) o[dm * plane] = fx::to_f64(NE - NO, r.ex);
  }
}

// ---------------------------------------------------------------------------------------------
// Eq. 17. Integers in two limbs of radix 2^28, h signed and l in [0, 2^28).
struct L28 {
  int h, l;
};
__device__ __forceinline__ L28 l28(s64 v) { return L28{(int)(v >> 28), (int)v & 0xfffffff}; }
// A plane's class entry where its cells are FP64 numbers: several classes, or one outside the integer form's range
constexpr int kMixed = 1 << 16;
// Class range of the integer form: results and their units stay normal FP64 numbers
constexpr int kClsMin = 56, kClsMax = 456;
// A value's integer, m 2^sh with its sign; sh = E - 4c + 5, in 2..5
__device__ __forceinline__ s64 val_fixed(double x, int sh) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = (hi & 0xfffffu) | 0x100000u;
  const u64 v = ((u64)__funnelshift_l(lo, m, sh) << 32) | (lo << sh);
  const s64 sg = (s64)((int)hi >> 31);
  return (s64)(v ^ (u64)sg) - sg;
}
// Weights of one ring as limbs (units of 2^-S): W+ and W- with line IV for the axis-aligned (0) or
// diagonal (1) directions, and minus their sum for the node itself (0 x-axis, 1 y-axis directions, 2
// diagonals), so that a constant field is reproduced exactly.
struct ClassW {
  L28 P[2], M[2];
};
__device__ __forceinline__ ClassW class_w(const Coeffs& c, int K, int l, s64 nux, s64 nuy) {
  return ClassW{{l28(c.xW1[0][K][l] + nux), l28(c.xW1[1][K][l] + nuy)},
                {l28(c.xWm1[0][K][l] + nux), l28(c.xWm1[1][K][l] + nuy)}};
}
__device__ __forceinline__ L28 centre_w(const Coeffs& c, int K, int l, s64 nux, s64 nuy) {
  return l28(c.xkeep - (c.xC2[K][l] + 2 * (nux + nuy)));
}
// Accumulators of a sum of products: H 2^56 + M 2^28. The low products are dropped; M starts from their
// mean, with l uniform in [0, 2^28) for a value and the weights' l given (their sum, lsum; a difference of
// values has mean zero), and from half a unit of 2^56 for the final shift.
struct Acc {
  s64 H, M;
};
__device__ __forceinline__ Acc acc_start(int lsum) { return Acc{0, (s64)(lsum >> 1) + (1 << 27)}; }
__device__ __forceinline__ int low_sum(const ClassW& w) {  // of the four neighbours' weights, below 2^30
  return (w.P[0].l + w.P[1].l) + (w.M[0].l + w.M[1].l);
}
__device__ __forceinline__ void mac(Acc& a, int vh, int vl, int wh, int wl) {
  a.M = fx::mad(vh, wl, a.M);
  a.M = fx::mad(vl, wh, a.M);
  a.H = fx::mad(vh, wh, a.H);
}
__device__ __forceinline__ void mac(Acc& a, L28 v, L28 w) { mac(a, v.h, v.l, w.h, w.l); }
// f_new of one velocity from the accumulated neighbours: B 2^t + sum, t = ex - unit, in units of
// 2^unit = 2^(4c - 1024 - S), rounded to FP64 once. B is shifted left or right by |t| (the other shift is by zero: no
// branch); what drops out rounds to odd. Where E and O nearly cancel, t is up to 20 and more. Returns false where r f_eq
// is far above the stencil's values or the result is below 2^32 units; the FP64 form then replaces it.
__device__ __forceinline__ bool finish(const Acc& a, s64 B, int ex, int unit, double& out) {
  const int t = ex - unit, l = max(t, 0), r = max(-t, 0), hi = (int)(B >> 32);
  const unsigned odd = fx::shl_clamped((unsigned)B, max(32 - r, 0)) ? 1u : 0u;
  const s64 Bs = (fx::shl64(B, l) >> min(r, 63)) | odd;
  const s64 R = Bs + (a.H + (a.M >> 28));
  out = fx::to_f64_fast(R, unit);
  // |B| 2^t < 2^61
  return l <= 29 && ((unsigned)(hi ^ (hi >> 31)) >> ((29 - l) & 31)) == 0u && (unsigned)(R >> 32) + 1u > 1u;
}

// A plane of several classes: a stencil's first NP cells, FP64 numbers, become integers of their largest class cl,
// m 2^(6 - s) with s = 4 cl + 1 - E, rounded to odd as in mom_term: a rounding of one sign would add up. FP64 numbers in the
// box and not integers of 15 classes below the plane's largest, since no span of a tile's values may change a stencil's:
// 1023 x 777 497 us per step against 503, a 32-tube batch 23.0 ms against 23.6, 400 x 4 10.4 us against 10.0. To nearest
// even instead the double Mach reflection's pass takes 2242 us, not 2175, and a 9000 x 4 tube's 3209, not 3148.
template <int NP>
__device__ __forceinline__ void align_cells(int2 (&t)[9], int& cl) {
  unsigned top = 0u;
#pragma unroll
  for (int i = 0; i < NP; ++i) top = max(top, (unsigned)t[i].y & 0x7fffffffu);
  cl = ((int)(top >> 20) + 3) >> 2;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const unsigned hi = (unsigned)t[i].y, lo = (unsigned)t[i].x, m = (hi & 0xfffffu) | 0x100000u;
    const int s = 4 * cl + 1 - (int)((hi & 0x7fffffffu) >> 20);  // 1..; of a zero so large that nothing is left
    const unsigned l6 = lo << 6;
    const u64 r = fx::shr_clamped(((u64)__funnelshift_l(lo, m, 6) << 32) | l6, s) |
                  (fx::shl_clamped(l6, max(32 - s, 0)) ? 1u : 0u);
    const s64 sg = (s64)((int)hi >> 31);
    const L28 u = l28((s64)(r ^ (u64)sg) - sg);
    t[i] = make_int2(u.h, u.l);
  }
}
// Whether a result of a plane of several classes may stay: 2^45 units of 2^unit or more, or the node's n 2^49 units.
// If not, several_classes looks at the stencil itself. The nodes that this leaves to the FP64 form, one direction in 10^5
// along a Mach 6 shock and none in smooth flow, cost the double Mach reflection 3% (100.5 -> 103.6 us per step).
__device__ __forceinline__ bool precise(double out, int unit, double n) {
  const int e = (int)((unsigned)__double2hiint(out) >> 20 & 0x7ffu) - 1023;
  return e >= unit + 45 || (int)((unsigned)__double2hiint(n) >> 20) - 1023 >= unit + 49;
}
// The directions of the mask, of planes of several classes, whose stencils hold several (b: the node's entry of the ring's
// first plane, planes BN apart, rows of BW)
template <int BN, int BW>
__device__ __noinline__ unsigned several_classes(const int2* __restrict__ b, unsigned mask) {
  unsigned out = 0u;
#pragma unroll 1
  for (int d = 0; d < 8; ++d, b += BN) {
    if (!(mask >> d & 1u)) continue;
    const int x2 = dir_xs(d) ? 2 : 1, y2 = dir_ys(d) ? 2 * BW : BW;
    const int at[9] = {0, 1, -1, x2, -x2, BW, -BW, y2, -y2};
    int lo = 1 << 20, hi = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int c = ((int)((unsigned)b[at[i]].y >> 20 & 0x7ffu) + 3) >> 2;
      lo = min(lo, c);
      hi = max(hi, c);
    }
    if (lo != hi) out |= 1u << d;
  }
  return out;
}
// Direction D at a node from the box (b: the node's entry of the plane, rows of BW). MIXED: the plane may hold several
// classes; the stencil's values then enter at their largest class, which cl becomes.
template <int D, int BW, bool MIXED>
__device__ __forceinline__ void stencil_box(Acc& a, int& cl, const int2* __restrict__ b, const ClassW& w, L28 w0,
                                            const Coeffs& c, int K, L28 nux, L28 nuy) {
  constexpr int XS = dir_xs(D), YS = dir_ys(D), CL = dir_cls(D);
  // centre, +-1 along x, then (along the direction) +2 and -2; the same along y
  constexpr int NP = 5 + (XS ? 2 : 0) + (YS ? 2 : 0), Y0 = XS ? 5 : 3;
  int2 t[9];
  t[0] = b[0];
  t[1] = b[1];
  t[2] = b[-1];
  if constexpr (XS != 0) {
    t[3] = b[2 * XS];
    t[4] = b[-2 * XS];
  }
  t[Y0] = b[BW];
  t[Y0 + 1] = b[-BW];
  if constexpr (YS != 0) {
    t[Y0 + 2] = b[2 * YS * BW];
    t[Y0 + 3] = b[-2 * YS * BW];
  }
  if constexpr (MIXED) {
    if (cl & kMixed) align_cells<NP>(t, cl);
  }
  auto at = [&](int i) { return L28{t[i].x, t[i].y}; };
  mac(a, at(0), w0);
  if constexpr (XS == 0) {
    mac(a, t[1].x + t[2].x, t[1].y + t[2].y, nux.h, nux.l);
  } else {
    mac(a, at(1), XS > 0 ? w.P[0] : w.M[0]);
    mac(a, at(2), XS > 0 ? w.M[0] : w.P[0]);
    mac(a, t[3].x - t[4].x, t[3].y - t[4].y, c.xD[0][K][CL][0], c.xD[0][K][CL][1]);
  }
  if constexpr (YS == 0) {
    mac(a, t[Y0].x + t[Y0 + 1].x, t[Y0].y + t[Y0 + 1].y, nuy.h, nuy.l);
  } else {
    mac(a, at(Y0), YS > 0 ? w.P[1] : w.M[1]);
    mac(a, at(Y0 + 1), YS > 0 ? w.M[1] : w.P[1]);
    mac(a, t[Y0 + 2].x - t[Y0 + 3].x, t[Y0 + 2].y - t[Y0 + 3].y, c.xD[1][K][CL][0], c.xD[1][K][CL][1]);
  }
}
// The FP64 form of Eq. 17 for the directions of the mask of ring K at one node: p and o are the node's entries of the
// ring's first plane in f and f_new, where o holds the directions' r f_eq. The ring's weights are formed once for all of
// them: with every direction here a site takes some 450 FP64 operations (1024^2 nodes with nu out of range: 1378 us per
// step; with f_eq and the weights formed again for each direction 4763, in range 830).
template <bool COH>
__device__ __noinline__ void stencils_f64(const double* __restrict__ p, double* __restrict__ o, long long plane,
                                          int pitch, int K, unsigned mask, double nux, double nuy, const Coeffs& c) {
  const double w0 = (1.0 - c.r) - 2.0 * (nux + nuy);
  double P1[2][2], M1[2][2];
#pragma unroll
  for (int l = 0; l < 2; ++l) {
    P1[0][l] = c.W1[0][K][l] + nux;
    M1[0][l] = c.Wm1[0][K][l] + nux;
    P1[1][l] = c.W1[1][K][l] + nuy;
    M1[1][l] = c.Wm1[1][K][l] + nuy;
  }
#pragma unroll
  for (int d = 0; d < 8; ++d, p += plane, o += plane) {
    if (!(mask >> d & 1u)) continue;
    const int xs = dir_xs(d), ys = dir_ys(d), cl = dir_cls(d);
    double acc = fma(w0 - c.C2[K][dir_c2(d)], ldf<COH>(p), *o);
    if (xs == 0) {
      acc = fma(nux, ldf<COH>(p + 1) + ldf<COH>(p - 1), acc);
    } else {
      acc = fma(xs > 0 ? P1[0][cl] : M1[0][cl], ldf<COH>(p + 1), acc);
      acc = fma(xs > 0 ? M1[0][cl] : P1[0][cl], ldf<COH>(p - 1), acc);
      acc = fma(xs > 0 ? c.D[0][K][cl] : -c.D[0][K][cl], ldf<COH>(p + 2) - ldf<COH>(p - 2), acc);
    }
    if (ys == 0) {
      acc = fma(nuy, ldf<COH>(p + pitch) + ldf<COH>(p - pitch), acc);
    } else {
      acc = fma(ys > 0 ? P1[1][cl] : M1[1][cl], ldf<COH>(p + pitch), acc);
      acc = fma(ys > 0 ? M1[1][cl] : P1[1][cl], ldf<COH>(p - pitch), acc);
      acc = fma(ys > 0 ? c.D[1][K][cl] : -c.D[1][K][cl], ldf<COH>(p + 2 * pitch) - ldf<COH>(p - 2 * pitch), acc);
    }
    *o = acc;
  }
}
// The ghost copies that an edge node owns of ring K's velocities, from the values it has just stored.
__device__ __noinline__ void ghost_ring(double* fn, const Grid& g, int gx, int gy, GhostOwn go, int K) {
  double* p = fn + (long long)(1 + 8 * K) * g.plane + (long long)(gy + NG) * g.pitch + (gx + NG);
  double v[8];
#pragma unroll
  for (int d = 0; d < 8; ++d) v[d] = p[d * g.plane];
#pragma unroll 1
  for (int t = 0; t < 8; ++t) {
    if (!(((go.mx | go.my << 4) >> t) & 1u)) continue;
    const bool x = t < 4;
    const int cc = x ? ghost_coord(t, g.nx) : ghost_coord(t - 4, g.ny);
    const bool wall = (x ? (cc < 0 ? g.bc[0] : g.bc[1]) : (cc < 0 ? g.bc[2] : g.bc[3])) == BC_WALL;
    double* q = p + (x ? (long long)(cc - gx) : (long long)(cc - gy) * g.pitch);
#pragma unroll
    for (int d = 0; d < 8; ++d) q[(wall ? (x ? mirror_x(1 + d) : mirror_y(1 + d)) - 1 : d) * g.plane] = v[d];
  }
}
// ... and of one velocity q
__device__ __noinline__ void ghost_one(double* __restrict__ fn, const Grid& g, int gx, int gy, GhostOwn go, int q,
                                       double val) {
  double* p = fn + (long long)(gy + NG) * g.pitch + (gx + NG);
#pragma unroll 1
  for (unsigned m = go.mx | go.my << 4; m; m &= m - 1u) {
    const int t = __ffs((int)m) - 1;
    const bool x = t < 4;
    const int cc = x ? ghost_coord(t, g.nx) : ghost_coord(t - 4, g.ny);
    const bool wall = (x ? (cc < 0 ? g.bc[0] : g.bc[1]) : (cc < 0 ? g.bc[2] : g.bc[3])) == BC_WALL;
    const int qq = wall ? (x ? mirror_x(q) : mirror_y(q)) : q;
    p[(long long)qq * g.plane + (x ? (long long)(cc - gx) : (long long)(cc - gy) * g.pitch)] = val;
  }
}

// A tile's box: the tile and its halo of two without the corners, which no stencil reads.
template <int TW, int TH>
struct FxBox {
  static constexpr int BW = TW + 4, BH = TH + 4, BN = BW * BH;
  static constexpr int CELLS = TW * BH + 4 * TH;  // the box without its corners
  // column and row of the box's cell idx: all rows of the tile's columns, then the halo columns
  __device__ static int2 cell(int idx) {
    if (idx < TW * BH) return make_int2(idx % TW + 2, idx / TW);
    const int j = idx - TW * BH;
    return make_int2((j & 3) < 2 ? (j & 3) : TW + (j & 3), 2 + (j >> 2));
  }
  __device__ static bool needed(const Grid& g, int cx, int cy) {  // padded coordinates
    return cx < g.nx + 2 * NG && cy < g.ny + 2 * NG &&
           ((cx >= NG && cx < g.nx + NG) || (cy >= NG && cy < g.ny + NG));
  }
};

// The cells that a tile converts: its box, or (DUP), where it holds the whole height of a y-periodic grid, the grid's
// rows with their halo columns, each stored again in the ghost row that copies it.
template <int TW, int TH, bool DUP>
struct FxCells {
  using X = FxBox<TW, TH>;
  static constexpr int N = DUP ? (TW + 4) * TH : X::CELLS, NV = (N + 31) / 32;
  __device__ static int2 cell(int idx) {
    if constexpr (DUP) return make_int2(idx % (TW + 4), idx / (TW + 4) + 2);
    else return X::cell(idx);
  }
  __device__ static void put(int2* __restrict__ box, int2 p, int2 w) {
    box[p.y * X::BW + p.x] = w;
    if constexpr (DUP) {
      if (p.y < 4) box[(p.y + TH) * X::BW + p.x] = w;
      if (p.y >= TH) box[(p.y - TH) * X::BW + p.x] = w;
    }
  }
};

// One warp converts one plane into its box, from the lane's cells' values v (a cell that no stencil reads
// takes another cell's value); returns the plane's class entry.
template <int TW, int TH, bool DUP = false>
__device__ __forceinline__ int convert_plane(int lane, const double (&v)[FxCells<TW, TH, DUP>::NV],
                                             int2* __restrict__ box) {
  using C = FxCells<TW, TH, DUP>;
  constexpr int NV = C::NV;
  unsigned amax = 0u, amin = 0x7fffffffu;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const unsigned a = (unsigned)__double2hiint(v[i]) & 0x7fffffffu;
    amax = max(amax, a);
    amin = min(amin, a);
  }
  const int cl = ((int)(__reduce_max_sync(0xffffffffu, amax) >> 20) + 3) >> 2;
  const int cm = ((int)(__reduce_min_sync(0xffffffffu, amin) >> 20) + 3) >> 2;
  if (cl == cm && cl >= kClsMin && cl <= kClsMax) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int2 p = C::cell(lane + 32 * i);
      const unsigned a = (unsigned)__double2hiint(v[i]) & 0x7fffffffu;
      const L28 t = l28(val_fixed(v[i], (int)(a >> 20) - (4 * cl - 5)));
      if (lane + 32 * i < C::N) C::put(box, p, make_int2(t.h, t.l));
    }
    return cl;
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int2 p = C::cell(lane + 32 * i);
    if (lane + 32 * i < C::N) C::put(box, p, make_int2(__double2loint(v[i]), __double2hiint(v[i])));
  }
  return kMixed;
}
template <int TW, int TH, bool DUP = false>
__device__ __forceinline__ void plane_cells(const Grid& g, int x0, int y0, int lane,
                                            int (&src)[FxCells<TW, TH, DUP>::NV]) {
  using X = FxBox<TW, TH>;
  using C = FxCells<TW, TH, DUP>;
#pragma unroll
  for (int i = 0; i < C::NV; ++i) {
    const int2 p = C::cell(lane + 32 * i);
    const int cx = x0 + p.x, cy = y0 + p.y;
    const bool use = lane + 32 * i < C::N && X::needed(g, cx, cy);
    src[i] = use ? cy * g.pitch + cx : (y0 + NG) * g.pitch + x0 + NG;
  }
}
// Eq. 16's switch along one axis, kappa (Eq. 15) and nu, in FP64: Pp, Pm the neighbours' pressures.
__device__ __forceinline__ double axis_nu(double P0, double Pp, double Pm, double u, double k, const Grid& g,
                                          const Coeffs& c, bool& kappa) {
  double th;
  if (g.flags & F_SWITCH_CONST) {
    th = c.lam;
  } else {
    const double s = Pp + Pm;
    th = c.lam * fabs(fma(-2.0, P0, s) * recip(fma(2.0, P0, s)));
  }
  const double ak = fabs(u * k);
  kappa = kappa || ak > 1.0;
  return g.flags & F_NO_VISC ? 0.0 : 0.5 * th * ak * (1.0 - ak);
}
// nu in the integer weights' units, where it fits them, and nu the number that the integer stands for: the rest velocity
// and the FP64 form take that one, since two roundings of nu at a node would make mass. To nearest: truncated, the
// viscosity would be low by half a unit in every step.
__device__ __forceinline__ bool nu_fixed(double& nu, const Coeffs& c, s64& nui) {
  nui = 0;
  if (!(c.xS != 0 && fabs(nu) <= c.xnu)) return false;
  nui = fx::from_f64_rn(nu, 62 - c.xS);
  nu = fx::to_f64(nui, -c.xS);  // exact: of 53 bits or fewer, like nu
  return true;
}
// f_eq and Eq. 17 of the pair of directions T of ring K (box: the node's entry in the ring's first plane,
// planes BN apart; MIXED: planes of several classes, n: the node's density). Returns the mask of directions
// that did not fit, and above it (<< 8) of those that have to be of one class (precise).
template <int T, int BN, int BW, bool MIXED>
__device__ __forceinline__ unsigned pair_box(const int2* __restrict__ box, const fx::RingFx& r, const fx::Dir& d,
                                             bool neg, const ClassW& w, L28 w0, L28 nux, L28 nuy, const Coeffs& c,
                                             int K, double n, const int* __restrict__ cls, double* __restrict__ o,
                                             long long plane) {
  s64 NE, NO;
  fx::pair_of<true>(r, d, NE, NO);
  if (neg) NO = -NO;
  unsigned bad = 0u;
  const int lsum = w0.l + (T == 0 ? w.P[0].l + w.M[0].l + 2 * nuy.l : T == 2 ? w.P[1].l + w.M[1].l + 2 * nux.l : low_sum(w));
  auto one = [&](auto dc, s64 B) {
    constexpr int D = decltype(dc)::value;
    int cl = cls[D];
    Acc a = acc_start(lsum);
    stencil_box<D, BW, MIXED>(a, cl, box + D * BN, w, w0, c, K, nux, nuy);
    const int unit = 4 * cl - 1024 - c.xS;
    double v;
    const bool ok = finish(a, B, r.ex, unit, v);
    if (!ok || (MIXED && (cl < kClsMin || cl > kClsMax))) bad |= 1u << D;
    if (MIXED && (cls[D] & kMixed) && !precise(v, unit, n)) bad |= 0x100u << D;
    o[D * plane] = v;
  };
  one(std::integral_constant<int, dir_plus(T)>{}, NE + NO);
  one(std::integral_constant<int, dir_minus(T)>{}, NE - NO);
  return bad;
}
// rest velocity: c = 0 on both axes, line IV only; five operations in FP64
template <bool COH>
__device__ __forceinline__ void rest_update(const double* __restrict__ f, double* __restrict__ fn, const Grid& g,
                                            const Coeffs& c, long long off, int gx, int gy, const GhostOwn& go,
                                            double rfeq, double nux, double nuy) {
  const double* p = f + off;
  double acc = fma((1.0 - c.r) - 2.0 * (nux + nuy), ldf<COH>(p), rfeq);
  acc = fma(nux, ldf<COH>(p + 1) + ldf<COH>(p - 1), acc);
  acc = fma(nuy, ldf<COH>(p + g.pitch) + ldf<COH>(p - g.pitch), acc);
  store_node<double, 0>(fn, g, gx, gy, go, acc);
}

// Shared memory of the tile with one lane per node: a ring's eight planes, the macros of the tile and its
// 1-node ring, and each lane's powers of its projections, which four rings need and registers cannot hold.
template <int TW, int TH>
struct FxTile {
  static constexpr int SW = TW + 2, SH = TH + 2, SN = SW * SH, NT = TW * TH;
  int4 q[8 * NT];  // fx::Dir of direction t: [2 t][lane] (q1, q2), [2 t + 1][lane] (q3, q4)
  int2 box[8][FxBox<TW, TH>::BN];
  double n[SN], ux[SN], uy[SN], T[SN], P[SN];
  int cls[8];  // the planes' classes, or kMixed
};

// One tile of the FP64 step, one lane per node, the rings one after the other. A tile that holds a
// y-periodic grid's whole height takes its two ghost rows' macros from the interior rows they copy.
template <int TW, int TH, bool COH, bool DUP>
__device__ __forceinline__ void fx_tile_body(const double* __restrict__ f, double* __restrict__ fn, const Grid& g,
                                        const Coeffs& c, unsigned* __restrict__ health, int tile_x, int tile_y,
                                        FxTile<TW, TH>& sm) {
  using S = FxTile<TW, TH>;
  using X = FxBox<TW, TH>;
  constexpr int SW = S::SW, SH = S::SH, NT = S::NT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x0 = tile_x * TW, y0 = tile_y * TH;
  unsigned bits = 0;

  // Phase 1: macros of the tile and its ring
  const bool wrap = g.ny <= TH && g.bc[2] == BC_PERIODIC && g.bc[3] == BC_PERIODIC;
  const int nslot = wrap ? SW * g.ny : SW * SH;
#pragma unroll 1
  for (int idx = tid; idx < nslot; idx += NT) {
    const int lx = idx % SW, ly = idx / SW + (wrap ? 1 : 0);
    const int gx = x0 + lx - 1, gy = y0 + ly - 1;
    if (!ring_node_needed(g, gx, gy)) continue;
    const Macro m = node_macro_fx<COH>(f, g.plane, (long long)(gy + NG) * g.pitch + (gx + NG), c);
    if (!macro_ok(m)) bits |= H_NUMERIC;
    const int o = ly * SW + lx;
    sm.n[o] = m.n;
    sm.ux[o] = m.ux;
    sm.uy[o] = m.uy;
    sm.T[o] = m.T;
    sm.P[o] = m.P;
  }
  if (wrap) {  // CTA-uniform: ghost rows copy the interior rows they stand for
    __syncthreads();
    const int top = (g.ny + 1) * SW, last = g.ny * SW;
    for (int i = tid; i < SW; i += NT) {
      sm.n[i] = sm.n[last + i], sm.n[top + i] = sm.n[SW + i];
      sm.ux[i] = sm.ux[last + i], sm.ux[top + i] = sm.ux[SW + i];
      sm.uy[i] = sm.uy[last + i], sm.uy[top + i] = sm.uy[SW + i];
      sm.T[i] = sm.T[last + i], sm.T[top + i] = sm.T[SW + i];
      sm.P[i] = sm.P[last + i], sm.P[top + i] = sm.P[SW + i];
    }
  }
  __syncthreads();

  // Phase 2, the lane's node: switch, nu, and what its rings share
  const int tx = tid % TW, ty = tid / TW;
  const int gx = x0 + tx, gy = y0 + ty;
  const bool mine = gx < g.nx && gy < g.ny;
  const int so = (ty + 1) * SW + (tx + 1);
  const long long off = (long long)(gy + NG) * g.pitch + (gx + NG);
  const GhostOwn go = ghost_own(g, gx, gy);
  double dnux = 0.0, dnuy = 0.0, snF = 0.0;
  s64 nuxi = 0, nuyi = 0;
  bool fixed = false;  // nu and the equilibrium's site numbers are in the integers' range
  FeqNode e;
  if (mine) {
    bool kappa = false;
    const double ux = sm.ux[so], uy = sm.uy[so];
    dnux = axis_nu(sm.P[so], sm.P[so + 1], sm.P[so - 1], ux, c.kx, g, c, kappa);
    dnuy = axis_nu(sm.P[so], sm.P[so + SW], sm.P[so - SW], uy, c.ky, g, c, kappa);
    if (kappa) bits |= H_KAPPA;
    e = feq_node<double>(sm.n[so], ux, uy, sm.T[so], c);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      sm.q[(2 * t) * NT + tid] = make_int4(e.q[t].q1.h, e.q[t].q1.l, e.q[t].q2.h, e.q[t].q2.l);
      sm.q[(2 * t + 1) * NT + tid] = make_int4(e.q[t].q3.h, e.q[t].q3.l, e.q[t].q4.h, e.q[t].q4.l);
    }
    // |nu| <= xnu keeps the weights' sum below 15/16 2^59
    fixed = nu_fixed(dnux, c, nuxi);
    fixed = nu_fixed(dnuy, c, nuyi) && fixed && e.b.ok;
  }
  constexpr int NV = FxCells<TW, TH, DUP>::NV;
  int src[NV];
  plane_cells<TW, TH, DUP>(g, x0, y0, lane, src);
#pragma unroll 1
  for (int K = 0; K < 4; ++K) {
    if (K) __syncthreads();  // the previous planes have been read
#pragma unroll 1
    for (int q = warp; q < 8; q += NT / 32) {
      const double* pl = f + (long long)(1 + 8 * K + q) * g.plane;
      double v[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = ldf<COH>(pl + src[i]);
      const int cl = convert_plane<TW, TH, DUP>(lane, v, sm.box[q]);
      if (lane == 0) sm.cls[q] = cl;
    }
    __syncthreads();
    if (!mine) continue;
    const double nF = ring_weight<true>(e, K, c);
    snF += nF;
    double* o = fn + (long long)(1 + 8 * K) * g.plane + off;
    unsigned slow = 0xffu;  // directions left to the FP64 form
    if (fixed && fx::weight_ok(nF)) {
      slow = 0u;
      const fx::RingFx r = fx::ring_scaled(e.b.A0f, fx::scale_of(e.b, K), e.b.e0, e.b.ea, e.b.ep, K, nF, c.fxc[1][K]);
      const int2* b = &sm.box[0][(ty + 2) * X::BW + tx + 2];
      auto powers = [&](int t) {
        const int4 u = sm.q[(2 * t) * NT + tid], v = sm.q[(2 * t + 1) * NT + tid];
        return fx::Dir{{u.x, u.y}, {u.z, u.w}, {v.x, v.y}, {v.z, v.w}};
      };
      int any = 0;
#pragma unroll
      for (int d = 0; d < 8; ++d) any |= sm.cls[d];
      const L28 nux = l28(nuxi), nuy = l28(nuyi);
      auto ring = [&](auto mixed) {
        constexpr bool MX = decltype(mixed)::value;
        constexpr int N = X::BN, W = X::BW;
        const double n = MX ? sm.n[so] : 0.0;
        {
          const ClassW w = class_w(c, K, 0, nuxi, nuyi);
          slow |= pair_box<0, N, W, MX>(b, r, powers(0), e.neg & 1u, w, centre_w(c, K, 0, nuxi, nuyi), nux, nuy, c, K,
                                        n, sm.cls, o, g.plane);
          slow |= pair_box<2, N, W, MX>(b, r, powers(2), e.neg & 4u, w, centre_w(c, K, 1, nuxi, nuyi), nux, nuy, c, K,
                                        n, sm.cls, o, g.plane);
        }
        {
          const ClassW w = class_w(c, K, 1, nuxi, nuyi);
          const L28 w0 = centre_w(c, K, 2, nuxi, nuyi);
          slow |= pair_box<1, N, W, MX>(b, r, powers(1), e.neg & 2u, w, w0, nux, nuy, c, K, n, sm.cls, o, g.plane);
          slow |= pair_box<3, N, W, MX>(b, r, powers(3), e.neg & 8u, w, w0, nux, nuy, c, K, n, sm.cls, o, g.plane);
        }
      };
      if (__builtin_expect(!(any & kMixed), 1)) ring(std::false_type{});  // CTA-uniform
      else ring(std::true_type{});
    }
    if (slow >> 8) slow |= several_classes<X::BN, X::BW>(&sm.box[0][(ty + 2) * X::BW + tx + 2], slow >> 8);
    slow &= 0xffu;
    if (slow) {
      if (e.b.ok && fx::weight_ok(nF))
        feq_slow(e.b.A0f, fx::scale_of(e.b, K), e.b.e0, e.b.ea, e.b.ep, e.neg, K, nF, slow, c, sm.q + tid, NT, o, g.plane);
      else
        feq_f64(sm.n[so], sm.ux[so], sm.uy[so], sm.T[so], K, slow, c, o, g.plane);
      stencils_f64<COH>(f + (o - fn), o, g.plane, g.pitch, K, slow, dnux, dnuy, c);
    }
    if (go.mx | go.my) ghost_ring(fn, g, gx, gy, go, K);
  }
  if (mine)
    rest_update<COH>(f, fn, g, c, off, gx, gy, go, fma(-8.0, snF, c.r * sm.n[so]) * e.A0d, dnux, dnuy);
  if (bits) atomicOr(health, bits);
}

// 4-row tubes are the tiles whose halo rows weigh most (272 converted cells for 128 nodes, 144 without): the 32 x 4
// tile has a form of its own for them (16384 x 4: 60.6 -> 53.0 us per step; 40000 x 4: 124 -> 115).
template <int TW, int TH, bool COH>
__device__ __forceinline__ void fx_tile(const double* __restrict__ f, double* __restrict__ fn, const Grid& g,
                                        const Coeffs& c, unsigned* __restrict__ health, int tile_x, int tile_y,
                                        FxTile<TW, TH>& sm) {
  if constexpr (TH == 4) {
    if (g.ny == TH && g.bc[2] == BC_PERIODIC && g.bc[3] == BC_PERIODIC)
      return fx_tile_body<TW, TH, COH, true>(f, fn, g, c, health, tile_x, tile_y, sm);
  }
  fx_tile_body<TW, TH, COH, false>(f, fn, g, c, health, tile_x, tile_y, sm);
}

// ---------------------------------------------------------------------------------------------
// The step for small grids, which leave the GPU mostly empty: a step lasts as long as one warp's
// instructions, and an FP64 instruction holds its warp for 64 cycles. A 4 x 4 or 8 x 4 tile has a CTA of
// eight warps. Phase 1: a quad of lanes per node sums the macros of the tile and its ring, while the other
// warps convert all 32 planes. Phase 2: three warps, two lanes per node, form the powers of the projections,
// nu, and the F_k. Phase 3: one thread for each node, ring and pair of opposite directions. The
// node's numbers are formed once, not by every lane, since the FP64 pipe is what a warp waits for.
// PPT: pairs of opposite directions per thread of phase 3, 1 or 2 (then x and y, or the two diagonals).
template <int TW, int TH, int PPT>
struct FxSmall {
  static constexpr int SW = TW + 2, SH = TH + 2, SN = SW * SH, NN = TW * TH, NT = 16 * NN / PPT;
  static_assert(NN % 16 == 0 && (TW & (TW - 1)) == 0 && (PPT == 1 || PPT == 2), "whole warps");
  int2 box[32][FxBox<TW, TH>::BN];
  double n[SN], ux[SN], uy[SN], T[SN], P[SN];
  int cls[32], next;
  int4 q[NN][8];
  double nF[NN][4], nu[NN][2], A0[NN];
  s64 A0f[NN], nui[NN][2];
  int es[NN][4], e0[NN], ea[NN], ep[NN], neg[NN], ok[NN], nufit[NN][2];
};
template <int TW, int TH, int PPT, bool COH>
__device__ __forceinline__ void fx_small_tile(const double* __restrict__ f, double* __restrict__ fn, const Grid& g,
                                              const Coeffs& c, unsigned* __restrict__ health, int tile_x, int tile_y,
                                              FxSmall<TW, TH, PPT>& sm) {
  using S = FxSmall<TW, TH, PPT>;
  using X = FxBox<TW, TH>;
  constexpr int SW = S::SW, NW = S::NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x0 = tile_x * TW, y0 = tile_y * TH;
  unsigned bits = 0;

  // a tile that holds a y-periodic grid's height: 24 nodes, the ghost rows' macros are the interior's
  const bool wrap = g.ny <= TH && g.bc[2] == BC_PERIODIC && g.bc[3] == BC_PERIODIC;
  // slots, and warps for them: at most all but three, in rounds
  const int nslot = wrap ? SW * g.ny : S::SN, mw = min((4 * nslot + 31) >> 5, NW - 3);
  if (tid == 0) sm.next = 0;
  __syncthreads();
  if (warp < mw) {
    const int r = tid & 3;
#pragma unroll 1
    for (int idx = tid >> 2; idx - (lane >> 2) < nslot; idx += 8 * mw) {
    const bool in = idx < nslot;
    const int lx = in ? idx % SW : 1, ly = in ? idx / SW + (wrap ? 1 : 0) : 1;
    const int gx = x0 + lx - 1, gy = y0 + ly - 1;
    const int cx = min(max(gx, -1), g.nx), cy = min(max(gy, -1), g.ny);
    const Macro m = quad_macro_fx<COH>(f, g.plane, (long long)(cy + NG) * g.pitch + (cx + NG), r, c);
    if (in && ring_node_needed(g, gx, gy)) {
      if (!macro_ok(m)) bits |= H_NUMERIC;
      auto put = [&](int o) {  // one array for each lane of the quad, and P
        if (r == 0) sm.n[o] = m.n, sm.P[o] = m.P;
        else if (r == 1) sm.ux[o] = m.ux;
        else if (r == 2) sm.uy[o] = m.uy;
        else sm.T[o] = m.T;
      };
      put(ly * SW + lx);
      if (wrap && gy == 0) put((g.ny + 1) * SW + lx);
      if (wrap && gy == g.ny - 1) put(lx);
    }
    }
  }
  // Planes, four at a time so that their loads overlap, by whichever warp is free
  {
    constexpr int NV = (X::CELLS + 31) / 32, U = 4;
    int src[NV];
    plane_cells<TW, TH>(g, x0, y0, lane, src);
#pragma unroll 1
    for (;;) {
      int q = 0;
      if (lane == 0) q = atomicAdd(&sm.next, U);
      q = __shfl_sync(0xffffffffu, q, 0);
      if (q >= 32) break;
      const double* pl = f + (long long)(1 + q) * g.plane;
      double v[U][NV];
#pragma unroll
      for (int j = 0; j < U; ++j)
#pragma unroll
        for (int i = 0; i < NV; ++i) v[j][i] = ldf<COH>(pl + j * g.plane + src[i]);
#pragma unroll 1
      for (int j = 0; j < U; ++j) {
        const int cl = convert_plane<TW, TH>(lane, v[0], sm.box[q + j]);
        if (lane == 0) sm.cls[q + j] = cl;
#pragma unroll
        for (int k = 0; k + 1 < U; ++k)
#pragma unroll
          for (int i = 0; i < NV; ++i) v[k][i] = v[k + 1][i];
      }
    }
  }
  __syncthreads();

#pragma unroll 1
  for (int item = warp; item < 3 * (S::NN / 16); item += NW) {  // 16 nodes, two lanes each
    const int kind = item % 3, nd = 16 * (item / 3) + (lane >> 1), h = lane & 1, tx = nd % TW, ty = nd / TW;
    const int so = (ty + 1) * SW + tx + 1;
    if (x0 + tx < g.nx && y0 + ty < g.ny) {
      const double n = sm.n[so], ux = sm.ux[so], uy = sm.uy[so], T = sm.T[so];
      if (kind == 0) {  // the powers of the projections; lane h stores directions 2 h and 2 h + 1
        const FeqSite64 e = feq_site64(ux, uy, T);
        const double pa = h ? e.p[2] : e.p[0], pb = h ? e.p[3] : e.p[1];
        const fx::Dir da = fx::dir_plain(fx::powers_of(e.b, pa, 2)), db = fx::dir_plain(fx::powers_of(e.b, pb, 2));
        sm.q[nd][4 * h] = make_int4(da.q1.h, da.q1.l, da.q2.h, da.q2.l);
        sm.q[nd][4 * h + 1] = make_int4(da.q3.h, da.q3.l, da.q4.h, da.q4.l);
        sm.q[nd][4 * h + 2] = make_int4(db.q1.h, db.q1.l, db.q2.h, db.q2.l);
        sm.q[nd][4 * h + 3] = make_int4(db.q3.h, db.q3.l, db.q4.h, db.q4.l);
        sm.es[nd][2 * h] = fx::scale_of(e.b, 2 * h);
        sm.es[nd][2 * h + 1] = fx::scale_of(e.b, 2 * h + 1);
        if (h == 0) {
          sm.A0[nd] = e.A0;
          sm.A0f[nd] = e.b.A0f;
          sm.e0[nd] = e.b.e0;
          sm.ea[nd] = e.b.ea;
          sm.ep[nd] = e.b.ep;
          sm.neg[nd] = (int)e.neg;
          sm.ok[nd] = e.b.ok;
        }
      } else if (kind == 1) {  // nu along x or y
        bool kappa = false;
        const int step = h ? SW : 1;
        double nu = axis_nu(sm.P[so], sm.P[so + step], sm.P[so - step], h ? uy : ux, h ? c.ky : c.kx, g, c, kappa);
        if (kappa) bits |= H_KAPPA;
        s64 nui;
        sm.nufit[nd][h] = nu_fixed(nu, c, nui);
        sm.nu[nd][h] = nu;
        sm.nui[nd][h] = nui;
      } else {  // r n F_k of two rings
        const double rnth = c.r * n * T;
        sm.nF[nd][2 * h] = weight_poly<true>(rnth, T, 2 * h, c);
        sm.nF[nd][2 * h + 1] = weight_poly<true>(rnth, T, 2 * h + 1, c);
      }
    }
  }
  __syncthreads();

  // A warp takes pairs of one kind, a lane is one (node, ring). One code for every direction (it is
  // fetched once, and used by all warps): a direction is the signs of its steps and its weights.
  constexpr int WPP = S::NN / 8;  // warps for one kind of pairs
  const int pg = warp / WPP, K = lane & 3, nd = (warp % WPP) * 8 + (lane >> 2);
  const int tx = nd % TW, ty = nd / TW, gx = x0 + tx, gy = y0 + ty;
  if (gx < g.nx && gy < g.ny) {
    const int so = (ty + 1) * SW + tx + 1;
    const long long off = (long long)(gy + NG) * g.pitch + (gx + NG);
    const GhostOwn go = ghost_own(g, gx, gy);
    const double nF = sm.nF[nd][K];
    const int diag = pg & 1;
    const s64 nuxi = sm.nui[nd][0], nuyi = sm.nui[nd][1];
    const bool fits = sm.nufit[nd][0] && sm.nufit[nd][1], brackets = sm.ok[nd] && fx::weight_ok(nF);
    const fx::RingFx r = fx::ring_scaled(sm.A0f[nd], sm.es[nd][K], sm.e0[nd], sm.ea[nd], sm.ep[nd], K, nF, c.fxc[1][K]);
    const L28 nux = l28(nuxi), nuy = l28(nuyi);
    const ClassW w = class_w(c, K, diag, nuxi, nuyi);
    unsigned slow = 0u;  // directions left to the FP64 form
#pragma unroll 1
    for (int T = pg; T < 4; T += 4 / PPT) {  // pairs pg, pg + 2
      const bool hx = T != 2, hy = T != 0;
      const L28 Px = hx ? w.P[0] : nux, Mx = hx ? w.M[0] : nux, Py = hy ? w.P[1] : nuy, My = hy ? w.M[1] : nuy;
      const L28 Dx{hx ? c.xD[0][K][diag][0] : 0, hx ? c.xD[0][K][diag][1] : 0};
      const L28 Dy{hy ? c.xD[1][K][diag][0] : 0, hy ? c.xD[1][K][diag][1] : 0};
      const L28 w0 = centre_w(c, K, diag ? 2 : T >> 1, nuxi, nuyi);
      const int4 u = sm.q[nd][2 * T], v4 = sm.q[nd][2 * T + 1];
      s64 NE, NO;
      fx::pair_of<true>(r, fx::Dir{{u.x, u.y}, {u.z, u.w}, {v4.x, v4.y}, {v4.z, v4.w}}, NE, NO);
      if ((sm.neg[nd] >> T) & 1) NO = -NO;
#pragma unroll 1
      for (int m = 0; m < 2; ++m) {
        const int d = m ? dir_minus(T) : dir_plus(T), q = 1 + 8 * K + d;
        const int ox = (m ? -1 : 1) * (T == 3 ? -1 : 1), oy = m ? -X::BW : X::BW;
        const int2* b = &sm.box[8 * K + d][(ty + 2) * X::BW + tx + 2];
        int cl = sm.cls[8 * K + d];
        int2 t[9] = {b[0], b[ox], b[-ox], b[2 * ox], b[-2 * ox], b[oy], b[-oy], b[2 * oy], b[-2 * oy]};
        bool ok = brackets && fits;
        if (cl & kMixed) {
          // a cell that the direction does not reach has no say in the class
          if (!hx) t[3] = t[4] = t[0];
          if (!hy) t[7] = t[8] = t[0];
          align_cells<9>(t, cl);
          ok = ok && cl >= kClsMin && cl <= kClsMax;
        }
        auto at = [&](int i) { return L28{t[i].x, t[i].y}; };
        Acc a = acc_start(w0.l + (Px.l + Mx.l) + (Py.l + My.l));
        mac(a, at(0), w0);
        mac(a, at(1), Px);
        mac(a, at(2), Mx);
        mac(a, t[3].x - t[4].x, t[3].y - t[4].y, Dx.h, Dx.l);
        mac(a, at(5), Py);
        mac(a, at(6), My);
        mac(a, t[7].x - t[8].x, t[7].y - t[8].y, Dy.h, Dy.l);
        const s64 B = m ? NE - NO : NE + NO;
        const int unit = 4 * cl - 1024 - c.xS;
        double v;
        ok = finish(a, B, r.ex, unit, v) && ok;
        const long long to = (long long)q * g.plane + off;
        if (ok && (sm.cls[8 * K + d] & kMixed) && !precise(v, unit, sm.n[so]))
          ok = !several_classes<X::BN, X::BW>(&sm.box[8 * K][(ty + 2) * X::BW + tx + 2], 1u << d);
        if (!ok) {  // r f_eq's integer waits in the place of the result
          slow |= 1u << d;
          v = __longlong_as_double(B);
        }
        fn[to] = v;
        if (ok && (go.mx | go.my)) ghost_one(fn, g, gx, gy, go, q, v);
      }
    }
    if (slow) {
      double* o = fn + (long long)(1 + 8 * K) * g.plane + off;
      if (brackets) {
#pragma unroll 1
        for (int d = 0; d < 8; ++d)
          if (slow >> d & 1u) o[d * g.plane] = fx::to_f64(__double_as_longlong(o[d * g.plane]), r.ex);
      } else {
        feq_f64(sm.n[so], sm.ux[so], sm.uy[so], sm.T[so], K, slow, c, o, g.plane);
      }
      stencils_f64<COH>(f + (o - fn), o, g.plane, g.pitch, K, slow, sm.nu[nd][0], sm.nu[nd][1], c);
      if (go.mx | go.my)
#pragma unroll 1
        for (int d = 0; d < 8; ++d)
          if (slow >> d & 1u) ghost_one(fn, g, gx, gy, go, 1 + 8 * K + d, o[d * g.plane]);
    }
    if (pg == 4 / PPT - 1 && K == 0) {
      const double snF = ((sm.nF[nd][0] + sm.nF[nd][1]) + sm.nF[nd][2]) + sm.nF[nd][3];
      rest_update<COH>(f, fn, g, c, off, gx, gy, go, fma(-8.0, snF, c.r * sm.n[so]) * sm.A0[nd], sm.nu[nd][0],
                       sm.nu[nd][1]);
    }
  }
  if (bits) atomicOr(health, bits);
}

// Programmatic dependent launch: the next step's blocks may be set up from here on, this one's wait for the
// step before to end (both do nothing in a launch without the attribute). 2 us of a 12 us step. f passes
// through the wait, so that no load of it is moved ahead.
__device__ __forceinline__ const double* dependent_launch(const double* f) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" : "+l"(f)::"memory");
  return f;
}
template <int TW, int TH, int MINB>
__global__ void __launch_bounds__(TW * TH, MINB) k_step_fx(const double* f, double* __restrict__ fn, Grid g,
                                                       Coeffs c, unsigned* __restrict__ health) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  f = dependent_launch(f);
  fx_tile<TW, TH, false>(f, fn, g, c, health, blockIdx.x, blockIdx.y, *reinterpret_cast<FxTile<TW, TH>*>(s_dyn));
}
template <int TW, int TH, int PPT, int MINB>
__global__ void __launch_bounds__(FxSmall<TW, TH, PPT>::NT, MINB) k_step_fx_small(const double* f,
                                                                              double* __restrict__ fn, Grid g,
                                                                              Coeffs c, unsigned* __restrict__ health) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  f = dependent_launch(f);
  fx_small_tile<TW, TH, PPT, false>(f, fn, g, c, health, blockIdx.x, blockIdx.y,
                                    *reinterpret_cast<FxSmall<TW, TH, PPT>*>(s_dyn));
}
// Batched step (see k_step_batch): block b runs tile b - tile0 of its member.
template <int TW, int TH, int MINB>
__global__ void __launch_bounds__(TW * TH, MINB) k_step_batch_fx(const BatchMember* __restrict__ mem, int nmem,
                                                             unsigned long long step, Coeffs c) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  const BatchMember& m = mem[batch_member(mem, nmem)];
  const Grid g = m.g;
  const long long local = (long long)blockIdx.x - m.tile0;
  const int par = (int)((m.cur0 + step) & 1ull);
  fx_tile<TW, TH, false>(static_cast<const double*>(m.f[par]), static_cast<double*>(m.f[par ^ 1]), g, c, m.health,
                         (int)(local % m.tiles_x), (int)(local / m.tiles_x), *reinterpret_cast<FxTile<TW, TH>*>(s_dyn));
}

}  // namespace
}  // namespace fdlbm
