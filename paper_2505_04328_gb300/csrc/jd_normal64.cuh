// jd_normal64.cuh -- the double-precision Box-Muller transform of the generator's 23-bit
// uniforms (jd_device.cuh: U(w) = ((w >> 9) + 1/2) 2^-23).
//
// FP64 is this part's scarcest unit: 2 lanes per clock and SM, so a warp instruction holds
// the pipe for 16 clocks, and log, sincospi and the products around them were three quarters
// of a step's FP64 instructions.  The arguments here are 23-bit integers, so the reductions
// are integer operations, and table entries with a short polynomial take the rest:
//
//   log    u = m 2^-E with m in [1, 2) by a count of leading zeros; i = m's first 8 bits below
//          the leading one; with g_i ~ 1/c_i rounded to 28 bits, r = m g_i - 1 is exact and
//          |r| <= 2^-9 (the table method of P. T. P. Tang, ACM TOMS 16(4), 1990), and
//          -2 log m = 2 log g_i - 2 log1p(r), the last by its Taylor series in s = -2 r.
//          For m >= sqrt 2 the entry holds 2 log(2 g_i) and E is one less; c_255 = 2, whose
//          entry is 0, so the result keeps its relative accuracy as u -> 1.
//   angle  the nearest of 1024 points of the circle (256 of a quarter turn, turned by the
//          quadrant) and the rest |b| <= 1.5 pi 2^-10 by the Taylor series of sin and cos.
//
// Every table value is split into a leading part and a remainder that joins the small terms,
// so each result has one rounding of its own size.  Largest error over all 2^23 arguments in
// units of the last place (and root mean square relative error), the CUDA library's functions
// -> here: radius sqrt(-2 log u) 0.852 -> 0.852 (5.27e-17 -> 5.27e-17), cosine and sine 1.476
// -> 0.998 (5.47e-17 -> 4.27e-17).  The chunked FP64 store sweep of d = 2 at M = 2^17, N_t =
// 400, lambda dt = 0.025: 14.6 -> 10.7 ms; without jumps 1.17 -> 0.79 (M = 2^15, N_t = 160).
#pragma once

#include <cstdint>

namespace jd {
namespace n64 {

// Double-double arithmetic for the tables, evaluated by the compiler.
struct DD {
  double h, l;
};
constexpr DD quick(double a, double b) {
  const double s = a + b;
  return {s, b - (s - a)};
}
constexpr DD two_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
constexpr DD two_prod(double a, double b) {
  const double ca = 134217729.0 * a, cb = 134217729.0 * b;
  const double ah = ca - (ca - a), bh = cb - (cb - b), al = a - ah, bl = b - bh, p = a * b;
  return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD add(DD a, DD b) {
  const DD s = two_sum(a.h, b.h);
  return quick(s.h, s.l + (a.l + b.l));
}
constexpr DD mul(DD a, DD b) {
  const DD p = two_prod(a.h, b.h);
  return quick(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD neg(DD a) { return {-a.h, -a.l}; }
constexpr DD div(DD a, DD b) {   // two corrections of the leading quotient
  const double q0 = a.h / b.h;
  DD r = add(a, neg(mul(b, DD{q0, 0.0})));
  const double q1 = r.h / b.h;
  r = add(r, neg(mul(b, DD{q1, 0.0})));
  const DD q = quick(q0, q1);
  return add(q, DD{r.h / b.h, 0.0});
}
constexpr DD kPi{3.141592653589793116, 1.2246467991473532e-16};

// log x = 2 atanh((x - 1) / (x + 1)) for x in [1/2, 2].
constexpr DD log_dd(double x) {
  const DD z = div(two_sum(x, -1.0), two_sum(x, 1.0)), z2 = mul(z, z);
  DD t = z, s = z;
  for (int k = 3; k <= 71; k += 2) {
    t = mul(t, z2);
    s = add(s, div(t, DD{(double)k, 0.0}));
  }
  return {2.0 * s.h, 2.0 * s.l};
}
// Leading part of v on the grid 2^-42 (sums of a few of them below 64 are exact).
constexpr double on_grid(double v) {
  const double magic = 1536.0;   // 1.5 2^10: its last place is 2^-42
  return (v + magic) - magic;
}

constexpr int NLOG = 256, NEXP = 25, NANG = 256;
struct alignas(16) Tables {
  double lg[NLOG][4];    // -2 g_i, 2 log g_i (or 2 log 2 g_i): grid part, remainder, unused
  double ex[NEXP][2];    // 2 E log 2: grid part, remainder
  double sc[NANG][4];    // sin, its remainder, cos, its remainder of j pi / 512
};
constexpr int FOLD = 106;   // first index with m >= sqrt 2

constexpr Tables make_tables() {
  Tables t{};
  for (int i = 0; i < NLOG; ++i) {
    const double c = i == NLOG - 1 ? 2.0 : 1.0 + (i + 0.5) / 256.0;
    // 1/c on the grid 2^-28
    const double g = ((1.0 / c) + 25165824.0) - 25165824.0;
    const DD v = log_dd(i >= FOLD ? 2.0 * g : g);
    t.lg[i][0] = -2.0 * g;
    t.lg[i][1] = on_grid(2.0 * v.h);
    t.lg[i][2] = (2.0 * v.h - t.lg[i][1]) + 2.0 * v.l;
  }
  const DD ln2 = log_dd(2.0);
  for (int e = 0; e < NEXP; ++e) {
    const DD v = mul(ln2, DD{2.0 * e, 0.0});
    t.ex[e][0] = on_grid(v.h);
    t.ex[e][1] = (v.h - t.ex[e][0]) + v.l;
  }
  for (int j = 0; j < NANG; ++j) {
    // sin and cos of j pi / 512 (at most pi / 2) by their Taylor series
    const DD x = mul(kPi, DD{j / 512.0, 0.0}), x2 = neg(mul(x, x));
    DD s = x, c{1.0, 0.0}, ts = x, tc{1.0, 0.0};
    for (int k = 1; k <= 14; ++k) {
      tc = div(mul(tc, x2), DD{(double)((2 * k - 1) * (2 * k)), 0.0});
      ts = div(mul(ts, x2), DD{(double)((2 * k) * (2 * k + 1)), 0.0});
      c = add(c, tc);
      s = add(s, ts);
    }
    t.sc[j][0] = s.h;
    t.sc[j][1] = s.l;
    t.sc[j][2] = c.h;
    t.sc[j][3] = c.l;
  }
  return t;
}
__device__ constexpr Tables kTab = make_tables();

// pi = PI_HI + PI_LO, PI_HI on the grid 2^-36
constexpr double PI_HI = (kPi.h + 98304.0) - 98304.0, PI_LO = (kPi.h - PI_HI) + kPi.l;

// The double with integer value n < 2^32 above 2^52.
__device__ __forceinline__ double above_2p52(uint32_t n) { return __hiloint2double(0x43300000, (int)n); }

// -2 log u, u = ((w >> 9) + 1/2) 2^-23.
__device__ __forceinline__ double neg2_log(uint32_t w) {
  const uint32_t X = (w >> 9) * 2u + 1u;   // u = X 2^-24
  const int lz = __clz((int)X);
  const uint32_t m32 = X << lz;            // m 2^31
  const int i = (int)((m32 >> 23) & 255u);
  const int E = lz - 7 - (i >= FOLD ? 1 : 0);
  const double m = __hiloint2double((int)(0x3ff00000u | ((m32 >> 11) & 0xfffffu)), (int)(m32 << 21));
  const double2 a = __ldg(reinterpret_cast<const double2 *>(kTab.lg[i]));
  const double lo = __ldg(&kTab.lg[i][2]);
  const double2 e = __ldg(reinterpret_cast<const double2 *>(kTab.ex[E]));
  const double s = __fma_rn(m, a.x, 2.0);   // -2 r, exact
  // -2 log1p(r) = s + s^2 (1/4 + s/12 + s^2/32 + s^3/80 + s^4/192)
  double q = __fma_rn(s, 1.0 / 192.0, 1.0 / 80.0);
  q = __fma_rn(s, q, 1.0 / 32.0);
  q = __fma_rn(s, q, 1.0 / 12.0);
  q = __fma_rn(s, q, 0.25);
  // H + s with its rounding error (|s| <= |H| or H = 0), which joins the small terms
  const double H = __dadd_rn(a.y, e.x);   // exact
  const double t = __dadd_rn(H, s), err = __dadd_rn(__dsub_rn(H, t), s);
  return __dadd_rn(t, __fma_rn(__dmul_rn(s, s), q, __dadd_rn(__dadd_rn(lo, e.y), err)));
}

// cos and sin of 2 pi ((w >> 9) + 1/2) 2^-23.
__device__ __forceinline__ void cos_sin_2pi(uint32_t w, double &c, double &s) {
  const uint32_t v = w >> 9;
  uint32_t p = (v + 4096u) >> 13;          // nearest of 1024 points
  int n = (int)v - (int)(p << 13);         // -4096 .. 4095
  // beside the axes the axis' point serves half a step more: no sum below cancels by half
  const int up = ((p & 255u) == 255u && n >= 2048) - ((p & 255u) == 1u && n < -2048);
  p += (uint32_t)up;
  n -= up * 8192;
  const double2 sn = __ldg(reinterpret_cast<const double2 *>(kTab.sc[p & 255u]));
  const double2 cs = __ldg(reinterpret_cast<const double2 *>(kTab.sc[p & 255u]) + 1);
  // b = k pi 2^-23, k = 2 n + 1 (14 bits): the product by pi's first 38 bits is exact
  const double k = __dadd_rn(above_2p52((uint32_t)(2 * n + 1 + 16384)), -(4503599627370496.0 + 16384.0));
  const double b = __fma_rn(k, PI_HI / 8388608.0, __dmul_rn(k, PI_LO / 8388608.0));
  const double b2 = __dmul_rn(b, b);
  const double sb = __fma_rn(__dmul_rn(b, b2), __fma_rn(b2, 1.0 / 120.0, -1.0 / 6.0), b);   // sin b
  const double cb = __dmul_rn(b2, __fma_rn(b2, 1.0 / 24.0, -0.5));                          // cos b - 1
  const double S = __dadd_rn(sn.x, __fma_rn(cs.x, sb, __fma_rn(sn.x, cb, sn.y)));
  const double C = __dadd_rn(cs.x, __fma_rn(-sn.x, sb, __fma_rn(cs.x, cb, cs.y)));
  // turn by the quadrant: (C, S), (-S, C), (-C, -S), (S, -C)
  const uint32_t quad = (p >> 8) & 3u;
  const double a = (quad & 1u) ? S : C, d = (quad & 1u) ? C : S;
  c = __hiloint2double(__double2hiint(a) ^ (int)(((quad + 1u) & 2u) << 30), __double2loint(a));
  s = __hiloint2double(__double2hiint(d) ^ (int)((quad & 2u) << 30), __double2loint(d));
}

}  // namespace n64
}  // namespace jd
