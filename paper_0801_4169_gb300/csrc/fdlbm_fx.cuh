#pragma once
// fdlbm_fx.cuh -- 62-bit fixed-point arithmetic on the integer pipes, for the parts of the step that
// would otherwise issue on the FP64 pipe.
//
// What bounds these kernels is FP64 issue: a warp-wide FP64 instruction holds its scheduler's FP64
// pipe for 64 cycles (16 cycles per SM and warp instruction, measured: 16-20), where a 32-bit integer
// instruction takes 0.5 cycles per SM, and so does a 32 x 32 + 64 -> 64-bit multiply-add (0.53
// measured, and on the FMA pipe beside the ALU). A 62-bit fractional product is three of those and a
// 64-bit shift, about 2.5 cycles, and it carries 9 bits more than FP64's significand.
//
// A fixed-point number is a 64-bit integer v that stands for v 2^-62 times a power of two that the
// caller keeps, |v| < 2^62. For a product it is split into limbs h 2^31 + l, 0 <= l < 2^31, h signed,
// so that every partial product is a signed 32 x 32-bit one. The low product l l' (below one unit of
// the result) is dropped.
//
// Every function is also compiled for the host, where the tests compare it with wider arithmetic.
#include <cmath>
#include <cstdint>
#include <cstring>

#ifndef FX_HD
#define FX_HD __host__ __device__ __forceinline__
#endif

namespace fdlbm {
namespace fx {

typedef long long s64;
typedef unsigned long long u64;

struct Limb {
  int h, l;
};
FX_HD Limb limb(s64 v) { return Limb{(int)(v >> 31), (int)(v & 0x7fffffff)}; }
// One wide multiply-add. Written out: from a * b + c on 64-bit integers the compiler makes a product and
// a separate 64-bit addition (2.5 cycles per SM and warp instruction, against 0.53).
FX_HD s64 mad(int a, int b, s64 c) {
#ifdef __CUDA_ARCH__
  s64 d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (s64)a * (s64)b + c;
#endif
}
FX_HD s64 mad_u(unsigned a, unsigned b, s64 c) {  // the unsigned form
#ifdef __CUDA_ARCH__
  s64 d;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (s64)((u64)a * (u64)b + (u64)c);
#endif
}
// a v + c modulo 2^64 for a small factor a >= 0
FX_HD s64 mad_small(unsigned a, s64 v, s64 c) {
#ifdef __CUDA_ARCH__
  s64 d;
  asm("{\n .reg .u32 l, h, dl, dh;\n .reg .b64 t;\n mov.b64 {l, h}, %2;\n mad.wide.u32 t, l, %1, %3;\n"
      " mov.b64 {dl, dh}, t;\n mad.lo.u32 dh, h, %1, dh;\n mov.b64 %0, {dl, dh};\n}\n"
      : "=l"(d) : "r"(a), "l"(v), "l"(c));
  return d;
#else
  return (s64)((u64)a * (u64)v + (u64)c);
#endif
}
// The dropped low product l l' 2^-62 is between 0 and 1 unit (1/4 in the mean, 1/3 of a square), and a shift
// drops up to one more; the products below start from the mean of what they drop, so that rounding has no
// sign: a bias would add up over the steps of a solve, where a rounding error only spreads.
constexpr s64 kMean = 3ll << 29, kMeanSq = (5ll << 30) / 3;
constexpr s64 kMeanShift = 1ll << 29;  // without the half unit: for a result that shr_round or a larger half follows
// a b 2^-62, within 2 units; start in units of 2^-31
FX_HD s64 mul(Limb a, Limb b, s64 start = kMean) {
  const s64 m = mad(a.h, b.l, mad(a.l, b.h, start));
  return mad(a.h, b.h, m >> 31);
}
// (a b + c d) 2^-62, within 3 units; the cross products of both pairs share one accumulator, so
// |a.h b.l| + |a.l b.h| + |c.h d.l| + |c.l d.h| must stay below 2^63. start: the mean of what drops out, half
// a unit and, unless b and d have signed low limbs, a quarter for each pair.
FX_HD s64 mul2(Limb a, Limb b, Limb c, Limb d, s64 start) {
  s64 m = mad(a.h, b.l, start);
  m = mad(a.l, b.h, m);
  m = mad(c.h, d.l, m);
  m = mad(c.l, d.h, m);
  return mad(a.h, b.h, mad(c.h, d.h, m >> 31));
}

FX_HD u64 bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 u;
  std::memcpy(&u, &x, 8);
  return u;
#endif
}
FX_HD double double_of(u64 u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((s64)u);
#else
  double x;
  std::memcpy(&x, &u, 8);
  return x;
#endif
}
FX_HD float float_of(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  std::memcpy(&x, &u, 4);
  return x;
#endif
}
FX_HD unsigned bits_of(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  unsigned u;
  std::memcpy(&u, &x, 4);
  return u;
#endif
}
FX_HD unsigned abs_hi(double x) { return (unsigned)(bits_of(x) >> 32) & 0x7fffffffu; }
// v >> s with 0 for s >= 64 (the shift instruction clamps its amount)
FX_HD u64 shr_clamped(u64 v, int s) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
#else
  return s < 64 ? v >> s : 0;
#endif
}
// v 2^-s rounded, |v| < 2^62, s in 0..63
FX_HD s64 shr_round(s64 v, int s) { return (v + (s64)((1ull << s) >> 1)) >> s; }
FX_HD s64 shl64(s64 v, int s) {  // 0 for s >= 64
#ifdef __CUDA_ARCH__
  s64 r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
#else
  return s < 64 ? (s64)((u64)v << s) : 0;
#endif
}
FX_HD unsigned shl_clamped(unsigned v, int s) {  // 0 for s >= 32
#ifdef __CUDA_ARCH__
  unsigned r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
  return r;
#else
  return s < 32 ? v << s : 0u;
#endif
}
// floor(log2 x) of a 32-bit integer, -127 for 0. From the exponent of x rounded towards zero to FP32:
// that conversion issues at full rate, the count of leading zeros at an eighth of it.
FX_HD int floor_log2(unsigned x) {
#ifdef __CUDA_ARCH__
  return (int)(__float_as_uint(__uint2float_rz(x)) >> 23) - 127;
#else
  return x ? 31 - __builtin_clz(x) : -127;
#endif
}
FX_HD int imax(int a, int b) { return a > b ? a : b; }
FX_HD int imin(int a, int b) { return a < b ? a : b; }
// |x| 2^(62 - e), truncated; |x| < 2^e. 0 for zero and far smaller values.
FX_HD s64 from_f64(double x, int e) {
  const u64 b = bits_of(x);
  const unsigned hi = (unsigned)(b >> 32) & 0x7fffffffu;
  const int E = (int)(hi >> 20);
  const u64 m = ((u64)((hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)b;
  const int s = 1022 + e - E;  // >= 0
  return (s64)((m << 9) >> (s < 63 ? s : 63));
}
// ... with its sign, rounded to nearest even; |x| < 2^(e - 1)
FX_HD s64 from_f64_rn(double x, int e) {
  const u64 b = bits_of(x);
  const unsigned hi = (unsigned)(b >> 32) & 0x7fffffffu;
  const u64 m = ((u64)((hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)b, v = m << 9;
  const int s = imin(1022 + e - (int)(hi >> 20), 63);  // >= 1; of a zero 63, which leaves nothing
  const u64 r = (v + ((1ull << (s - 1)) - 1ull) + ((v >> s) & 1ull)) >> s;
  return b >> 63 ? -(s64)r : (s64)r;
}
// e with |x| < 2^e (x normal)
FX_HD int exp_of(unsigned abs_hi_word) { return (int)(abs_hi_word >> 20) - 1022; }

// R 2^ex rounded to nearest even FP64, |R| < 2^63, the result a normal number or zero. The magnitude
// is shifted until its leading one is bit 62, and rounded at bit 10.
FX_HD double to_f64(s64 R, int ex) {
  const s64 sg = R >> 63;
  const u64 A = (u64)((R ^ sg) - sg);
  unsigned hi = (unsigned)(A >> 32), lo = (unsigned)A;
  if (hi == 0u) {  // below 2^32
    hi = lo >> 1;
    lo <<= 31;
    ex -= 31;
  }
  const int lg = floor_log2(hi);  // 0..30; negative for 0 and 1
  const u64 U = (((u64)hi << 32) | lo) << ((30 - lg) & 31);
  const u64 M = (U + 0x1ffull + ((U >> 10) & 1ull)) >> 10;
  // the leading one of M (bit 52) adds the last 1 to the exponent; a carry to 2^53 adds one more
  u64 r = ((u64)(1023 + 32 + lg + ex - 1) << 52) + M;
  if (lg < 0) r = lo ? (u64)(1023 + 31 + ex) << 52 : 0ull;
  return double_of(((u64)sg & 0x8000000000000000ull) | r);
}

// R 2^ex rounded to nearest even FP64 (a tie is not rare: a few bits drop), for 2^32 <= |R| < 2^62 and a normal result
FX_HD double to_f64_fast(s64 R, int ex) {
  const s64 sg = R >> 63;
  const u64 A = (u64)((R ^ sg) - sg);
  const int lg = floor_log2((unsigned)(A >> 32));
  const u64 U = A << ((30 - lg) & 31);
  const u64 M = (U + 0x1ffull + (unsigned)((unsigned)U >> 10 & 1u)) >> 10;
  const unsigned hi = (unsigned)(M >> 32) + ((unsigned)(1023 + 31 + lg + ex) << 20);
  return double_of(((u64)(hi | ((unsigned)(sg >> 32) & 0x80000000u)) << 32) | (unsigned)M);
}

// ---------------------------------------------------------------------------------------------
// The opposite-direction pairs of Eq. 10. With p_t = (e_t . u)/theta the projection on direction t
// (x, diagonal, y, anti-diagonal), A0 = 1 - b + b^2/2, A1 = 1 - b:
//   f+- = nF_k (E +- O),  E = A0 + (v_k^2/2) A1 p^2 + (v_k^4/24) p^4,  O = v_k A1 p + (v_k^3/6) p^3.
// A node's projections share one scale, p = P 2^ep with |P| < 1, and ring k's brackets come in units of
// 2^es, where 2^es is 8 to 128 times a bound of |E| and |O| over the directions. The four powers of p are
// formed once per direction, and the ring's five constants, scaled and multiplied by the significand of
// nF_k, once per ring, so that a bracket is four (cross) plus two (high) multiply-adds. It carries an
// error of a few 2^-56 of its bound at most, where FP64 rounds each of its operations to 2^-53.
FX_HD constexpr int exp_c1(int k) { return k == 0 ? 0 : k == 1 ? 2 : k == 2 ? 3 : 4; }
FX_HD constexpr int exp_c2(int k) { return k == 0 ? -4 : k == 1 ? 0 : k == 2 ? 2 : 5; }
FX_HD constexpr int exp_c3(int k) { return k == 0 ? 1 : k == 1 ? 2 : k == 2 ? 2 : 3; }
FX_HD constexpr int exp_c4(int k) { return k == 0 ? -2 : k == 1 ? 1 : k == 2 ? 3 : 5; }
FX_HD unsigned umax(unsigned a, unsigned b) { return a > b ? a : b; }
// an FP32 number at or just above |x| from its FP64 high word (|x| in the FP32 normal range)
FX_HD float f32_above(unsigned ah) { return float_of(((ah - (896u << 20)) << 3) + 8u); }
// Scales of one node. ok is false where the numbers lie outside the range that they can hold
// (infinities and NaN among them): the caller then takes the FP64 form.
struct Base {
  int ep, ea, e0;
  s64 A1f, A0f;  // A1 2^-ea and A0 2^-e0 with their signs
  unsigned a0;   // high word of |A0|
  float a1, pf;  // bounds of |A1| and of the largest |p|
  bool ok;
};
FX_HD Base base_of(double A0, double A1, double p0, double p1, double p2, double p3) {
  Base b;
  b.a0 = abs_hi(A0);
  const unsigned a1 = umax(abs_hi(A1), (1023u - 40u) << 20);
  const unsigned pm = umax(umax(umax(abs_hi(p0), abs_hi(p1)), umax(abs_hi(p2), abs_hi(p3))), (1023u - 40u) << 20);
  b.ep = exp_of(pm);
  b.ea = exp_of(a1);
  // |p| < 2^10 and 2^-60 < |A0| < 2^40, |A1| < 2^40 keep every scale and FP32 bound inside its range
  b.ok = pm < (1023u + 10u) << 20 && a1 < (1023u + 40u) << 20 && b.a0 < (1023u + 40u) << 20 &&
         b.a0 > (1023u - 60u) << 20;
  b.a1 = f32_above(a1);
  b.pf = f32_above(pm);
  b.A1f = from_f64(A1, b.ea);
  if (bits_of(A1) >> 63) b.A1f = -b.A1f;
  b.e0 = exp_of(b.a0);
  b.A0f = from_f64(A0, b.e0);
  if (bits_of(A0) >> 63) b.A0f = -b.A0f;
  return b;
}
// A weight nF_k that the fixed-point form can take. FP64 results: 2^-700 < |nF_k| < 2^700. Its exponent is part of
// the results' scale alone, an integer; the limits keep the results normal.
FX_HD bool weight_ok(double nF) { return abs_hi(nF) - ((1023u - 700u) << 20) < 1400u << 20; }
// ... for FP32 results, in units of 2^ex: those whose scale 2^(ex + 36) beside narrow_f32 is an FP32 number
FX_HD bool unit_ok_f32(int ex) { return (unsigned)(ex + 36 + 149) <= 149u + 127u; }
// es of ring k
FX_HD int scale_of(const Base& b, int k) {
  const float v = k == 0 ? 1.0f : k == 1 ? 1.92f : k == 2 ? 2.99f : 4.49f;
  const float vp = v * b.pf, x = vp * vp;
  const float E = f32_above(b.a0) + 0.5f * b.a1 * x + (1.0f / 24.0f) * x * x;
  const float O = b.a1 * vp + (1.0f / 6.0f) * x * vp;
  // 2^(es - 3) > max(E, O); the factor covers the FP32 roundings
  const int es = (int)(bits_of((E > O ? E : O) * 1.0001f) >> 23) - 126 + 3;
  // ... and the scaled constants stay below 2^62
  return imax(imax(es, imax(b.ea + 2 * b.ep + exp_c1(k), 4 * b.ep + exp_c2(k)) + 2),
              imax(b.ea + b.ep + exp_c3(k), 3 * b.ep + exp_c4(k)) + 2);
}
// One direction's A1 p^2, p^4, A1 p, p^3 (of |p|), as fractions of 2^(ea + 2 ep), 2^(4 ep), ...
struct Powers {
  s64 ax, x2, ap, p3;
};
// half: added to the results, in units of 2^-62: half of what a later shift drops (0 or more)
FX_HD Powers powers_of(const Base& b, double p, int half) {
  const Limb P = limb(from_f64(p, b.ep));
  const Limb A = limb(b.A1f);
  const Limb X = limb(mul(P, P, kMeanSq));
  const s64 m = half ? kMeanShift + ((s64)half << 31) : kMean, sq = m + (kMeanSq - kMean);
  return Powers{mul(A, X, m), mul(X, X, sq), mul(A, P, m), mul(P, X, m)};
}
struct Dir {
  Limb q1, q2, q3, q4;
};
// One ring's constants times the significand of nF_k; brackets come in units of 2^ex.
struct RingFx {
  s64 A0;
  Limb c1, c2, c3, c4;
  int ex;
};
FX_HD Limb significand(double nF, int e) {  // with its sign
  const s64 v = from_f64(nF, e);
  return limb(bits_of(nF) >> 63 ? -v : v);
}
// FP64 results: the powers stay as they are (two bits down, so that the cross products of a bracket
// fit one accumulator; powers_of has added the half of them; the low limb is signed, so that what mul2 drops
// has mean zero, and is zero for a projection of zero) and each ring scales its constants. c: v^2/2 2^-exp_c1, v^4/24 2^-exp_c2,
// v 2^-exp_c3, v^3/6 2^-exp_c4 of ring k as 62-bit integers.
FX_HD Dir dir_plain(const Powers& w) {
  auto down2 = [](s64 v) {
    const int u = (int)(unsigned)(v >> 2);
    return Limb{((int)(v >> 32) + 1) >> 1, (int)((unsigned)u << 1) >> 1};
  };
  return Dir{down2(w.ax), down2(w.x2), down2(w.ap), down2(w.p3)};
}
// es, e0, ea, ep and A0f: scale_of(b, k) and the fields of Base
FX_HD RingFx ring_scaled(s64 A0f, int es, int e0, int ea, int ep, int k, double nF, const s64* c) {
  RingFx r;
  const int e = exp_of(abs_hi(nF));
  const Limb m = significand(nF, e);
  r.ex = es + e - 62;
  // shifted after the product: a constant shifted first would keep one error for all steps of a solve
  r.A0 = shr_round(mul(limb(A0f), m, kMeanShift), imin(es - e0, 63));
  r.c1 = limb(shr_round(mul(limb(c[0]), m, kMeanShift), imin(es - ea - 2 * ep - exp_c1(k) - 2, 63)));
  r.c2 = limb(shr_round(mul(limb(c[1]), m, kMeanShift), imin(es - 4 * ep - exp_c2(k) - 2, 63)));
  r.c3 = limb(shr_round(mul(limb(c[2]), m, kMeanShift), imin(es - ea - ep - exp_c3(k) - 2, 63)));
  r.c4 = limb(shr_round(mul(limb(c[3]), m, kMeanShift), imin(es - 3 * ep - exp_c4(k) - 2, 63)));
  return r;
}
// FP32 results: one scale, ring 4's, for all rings: the powers are scaled once, and a ring only
// multiplies. That costs the slower rings up to 15 bits and leaves them 20 more than the FP32 number
// they are rounded to. c: the constants of ring k by ring 4's powers of two.
FX_HD Dir dir_shared(const Powers& w, const Base& b, int es) {
  return Dir{limb(w.ax >> imin(es - b.ea - 2 * b.ep - exp_c1(3), 63)), limb(w.x2 >> imin(es - 4 * b.ep - exp_c2(3), 63)),
             limb(w.ap >> imin(es - b.ea - b.ep - exp_c3(3), 63)), limb(w.p3 >> imin(es - 3 * b.ep - exp_c4(3), 63))};
}
FX_HD RingFx ring_shared(Limb A0, int es, double nF, const s64* c) {
  RingFx r;
  const int e = exp_of(abs_hi(nF));
  const Limb m = significand(nF, e);
  r.ex = es + e - 62;
  r.A0 = mul(A0, m);
  r.c1 = limb(mul(limb(c[0]), m));
  r.c2 = limb(mul(limb(c[1]), m));
  r.c3 = limb(mul(limb(c[2]), m));
  r.c4 = limb(mul(limb(c[3]), m));
  return r;
}
// nF_k E and nF_k O of one pair, for |p|: integers below 2^60 in units of 2^ex
template <bool PLAIN>  // from dir_plain, or from dir_shared
FX_HD void pair_of(const RingFx& r, const Dir& d, s64& NE, s64& NO) {
  constexpr s64 start = PLAIN ? 1ll << 30 : 1ll << 31;
  NE = r.A0 + mul2(r.c1, d.q1, r.c2, d.q2, start);
  NO = mul2(r.c3, d.q3, r.c4, d.q4, start);
}
// R as an FP32 number in units of 2^36, |R| < 2^60: R = hi 2^36 + lo 2^4 with hi exact in FP32, so one rounding of
// R's leading bits (and one of lo, 2^-24 of 2^36 units). The caller's scale 2^(ex + 36) then changes no bit.
FX_HD float narrow_f32(s64 R) {
  const int hi = (int)(R >> 32) >> 4;
  const unsigned lo = (unsigned)(R >> 4);
#ifdef __CUDA_ARCH__
  return __fmaf_rn(__uint2float_rn(lo), 0x1p-32f, __int2float_rn(hi));
#else
  return std::fma((float)lo, 0x1p-32f, (float)hi);
#endif
}
// 2^e, e in -149..127
FX_HD float pow2_f32(int e) { return float_of(e >= -126 ? (unsigned)(e + 127) << 23 : 1u << ((e + 149) & 31)); }

}  // namespace fx
}  // namespace fdlbm
