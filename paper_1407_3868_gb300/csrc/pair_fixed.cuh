// The Hankel sequence of one disc pair in 64-bit fixed point, for the FP64 translation on the tensor
// cores (translate_f64_tc.cu).
//
// This GPU issues 2 FP64 operations per SM and clock against 64 to 128 integer ones, so the
// sequence of a far pair is formed in integers: FP64 gives the distance, its reciprocal and the
// phase (about 40 operations), everything after them is fixed point.  With z = k rho >= 26 and
// s <= 2p <= z - 4 every quantity is bounded (|J_s|, |Y_s| < 0.22, |2s/z| < 2), so fixed point loses
// nothing: products keep 62 to 65 fractional bits, FP64 would keep 53.
//
// Notation: Qn is a signed 64-bit integer with n fractional bits.  All functions also compile for
// the host, where the tests of the arithmetic run.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "fixed64.cuh"

// Constants of a layer (host: pair_consts).
struct PairConsts {
  double turn_hi, turn_lo;   // k / (2 pi) as a sum of two doubles
  double inv_k;              // 1 / k
  double amp;                // sqrt(2 / (pi k)) / R, see PairState
  float near_r2;             // pairs with r^2 below this are left out (summed from the near-pair list)
};

// H_0 / R, H_1 / R (Q65), e^{i phi} (Q62) and 2/z (Q62) of a pair.
struct PairSeed {
  int64_t j0, y0, j1, y1, c, s, w;
};

namespace {

LSMS_HD int64_t to_fixed(double x) {
#ifdef __CUDA_ARCH__
  return __double2ll_rn(x);
#else
  return llrint(x);
#endif
}

// c0 + x (c1 + x (c2 + ... + x c5)) in Q62 for x = 1/z^2 <= 26^-2 given in Q72: the tail from c2 on
// in 32 bits (c2 in Q31, then 8 fractional bits less per step: the mulhi of a Q40 gives 8 back).
LSMS_HD int64_t series(int64_t x, int64_t c0, int64_t c1, int32_t c2, int32_t c3, int32_t c4, int32_t c5) {
  const int32_t h = hi_s32(x);
  const int32_t r = c2 + mulhi_s32(h, c3 + mulhi_s32(h, c4 + mulhi_s32(h, c5)));
  return c0 + (mulq(x, c1 + (mul_wide(h, r) >> 9)) >> 8);  // Q71 -> Q62, Q70 -> Q62
}

#define LSMS_Q(x, n) ((int64_t)((x) * (double)(1LL << ((n) / 2)) * (double)(1LL << ((n) - (n) / 2))))
#define LSMS_Q32(x, n) ((int32_t)((x) * (double)(1LL << (n))))

// Hankel's expansion (Abramowitz & Stegun 9.2.5-9.2.10), P_n = 1 + x P(x), Q_n = Q(x) / z, x = 1/z^2,
// as polynomials of degree 5 interpolated at Chebyshev nodes on [0, 26^-2] (within 4e-18 of P_n, Q_n).
LSMS_HD int64_t series_p0(int64_t x) {
  return series(x, LSMS_Q(-0.0703124999999995114, 62), LSMS_Q(0.112152099585567959, 62), LSMS_Q32(-0.572501232228554015, 31),
                LSMS_Q32(6.07349164755919553, 23), LSMS_Q32(-109.284463061588291, 15), LSMS_Q32(2577.61909601392639, 7));
}
LSMS_HD int64_t series_q0(int64_t x) {
  return series(x, LSMS_Q(-0.124999999999999923, 62), LSMS_Q(0.0732421874962389523, 62), LSMS_Q32(-0.227107971911088272, 31),
                LSMS_Q32(1.72764073954614824, 23), LSMS_Q32(-24.2653379847043508, 15), LSMS_Q32(479.362753445535456, 7));
}
LSMS_HD int64_t series_p1(int64_t x) {
  return series(x, LSMS_Q(0.117187499999999474, 62), LSMS_Q(-0.144195556615006151, 62), LSMS_Q32(0.676592385323675246, 31),
                LSMS_Q32(-6.88332211536600019, 23), LSMS_Q32(120.809715149211668, 15), LSMS_Q32(-2807.11788473847159, 7));
}
LSMS_HD int64_t series_q1(int64_t x) {
  return series(x, LSMS_Q(0.374999999999999916, 62), LSMS_Q(-0.102539062495930361, 62), LSMS_Q32(0.277576414291913122, 31),
                LSMS_Q32(-1.99343786532250002, 23), LSMS_Q32(27.1242252388828417, 15), LSMS_Q32(-526.022190652616016, 7));
}

// The same float decision everywhere a pair is classified.
LSMS_HD bool pair_is_near(double r2, const PairConsts& q) { return (float)r2 < q.near_r2; }

// Seed of the pair offset (dx, dy) = x_l - x_m, r2 = dx^2 + dy^2.  table[i] = (cos, sin) of
// 2 pi i / 256 - pi / 4 in Q62.
template <typename Table>
LSMS_HD void pair_seed(double dx, double dy, double r2, const PairConsts& q, const Table* table, PairSeed& o) {
  // v = r2^(-1/4), y = 1/rho, rho: one step of third order from a float start
#ifdef __CUDA_ARCH__
  double v = (double)rsqrtf(sqrtf((float)r2));
#else
  double v = (double)(1.0f / sqrtf(sqrtf((float)r2)));
#endif
  const double v2 = v * v;
  const double e = fma(-r2, v2 * v2, 1.0);
  v = fma(v * e, fma(e, 0.15625, 0.25), v);
  double y = v * v;
  double rho = r2 * y;
  rho = fma(fma(-rho, rho, r2), 0.5 * y, rho);
  y = fma(y, fma(-rho, y, 1.0), y);
  // phase z / (2 pi) modulo 1
  const double t = rho * q.turn_hi;
  const double tl = fma(rho, q.turn_lo, fma(rho, q.turn_hi, -t));
  const double f = (t - rint(t)) + tl;
  const int64_t phase = shl(to_fixed(f * 9223372036854775808.0 * 0.5), 2);   // Q64, modulo 1
  const int64_t u = to_fixed(y * (q.inv_k * 73786976294838206464.0));        // 1/z, Q66
  const int64_t amp = to_fixed(v * (q.amp * 36893488147419103232.0));        // sqrt(2 / (pi z)), Q65
  const double ys = y * 4611686018427387904.0;
  o.c = to_fixed(dx * ys);
  o.s = to_fixed(dy * ys);
  o.w = u >> 3;                                                              // 2/z, Q62
  // e^{i (z - pi/4)}: table entry and the remainder theta = 2 pi delta, |theta| <= 2 pi / 512
  const int idx = (int)((uint32_t)((uint64_t)(phase + (1LL << 55)) >> 56));
  const int64_t delta = phase - shl(idx, 56);
  const int64_t th = mulq(shl(delta, 7), LSMS_Q(6.283185307179586476925, 60));   // Q67
  const int64_t t2 = shl(mulq(th, th), 5);                                       // theta^2, Q75
  const int32_t t2h = hi_s32(t2);                                                // Q43
  const int32_t kc = LSMS_Q32(1.0 / 24.0, 35) - mulhi_s32(t2h, LSMS_Q32(1.0 / 720.0, 24));
  const int64_t gc = (mul_wide(t2h, kc) >> 16) - (1LL << 61);                  // -1/2 + theta^2/24 - ..., Q62
  const int64_t cm = mulq(t2, gc) >> 9;                                          // cos theta - 1, Q64
  const int64_t gs = (mul_wide(t2h, LSMS_Q32(1.0 / 120.0, 37)) >> 18) - LSMS_Q(1.0 / 6.0, 62);
  const int64_t sv = mulq(t2, gs);                                               // sin theta / theta - 1, Q73
  const int64_t sn = (th >> 3) + (mulq(th, sv) >> 12);                           // Q64
  const auto tab = table[idx];
  const int64_t ec = tab.x + mulq2(tab.x, cm, tab.y, -sn);                       // Q62
  const int64_t es = tab.y + mulq2(tab.y, cm, tab.x, sn);
  const int64_t ac = shl(mulq(ec, amp), 2), as = shl(mulq(es, amp), 2);          // Q65
  // H_0 = amp e (P_0 + i Q_0), H_1 = -i amp e (P_1 + i Q_1)
  const int64_t x = shl(mulq(u, u), 4);                                          // 1/z^2, Q72
  const int64_t p0 = mulq(x, series_p0(x)) >> 6, q0 = mulq(u, series_q0(x));     // Q64
  const int64_t p1 = mulq(x, series_p1(x)) >> 6, q1 = mulq(u, series_q1(x));
  o.j0 = ac + mulq2(ac, p0, as, -q0);
  o.y0 = as + mulq2(as, p0, ac, q0);
  o.j1 = as + mulq2(as, p1, ac, q1);
  o.y1 = -(ac + mulq2(ac, p1, as, -q1));
}

// The sequence around an even order s: sigma_s J_s and sigma_{s-1} J_{s-1}, the same of Y (Q63), R e^{i s phi}
// (Q63; the radius R = 1 - 2^-30 keeps them below 1, the amplitude of the seed carries 1 / R), 2s/z and
// -2(s+1)/z (Q62).  The signs sigma = + + - - (s mod 4) turn the recurrence's subtraction into an
// addition, which a multiply-add does by itself: with f = 2s/z, sigma_{s+1} J_{s+1} =
// +-f sigma_s J_s + sigma_{s-1} J_{s-1}, plus for even s, minus for odd s.
struct PairState {
  int64_t je, jo, ye, yo, c, s, fe, fo;
};
// Factors that stay the same along the orders: e^{i phi} (Q62) and minus its sine.
struct PairStep {
  Factor c, s, ns;
  int64_t w2;                // 4/z
};
constexpr int64_t kRadius = ((int64_t)1 << 62) - ((int64_t)1 << 32);   // R / 2 in Q63

// Order 0: J_{-1} = -J_1, sigma_{-1} = -1.
LSMS_HD void pair_start(const PairSeed& o, PairState& a, PairStep& t) {
  a.je = o.j0 >> 2; a.jo = o.j1 >> 2; a.ye = o.y0 >> 2; a.yo = o.y1 >> 2;
  a.c = shl(kRadius, 1); a.s = 0; a.fe = 0; a.fo = -o.w;
  t.c = factor(o.c); t.s = factor(o.s); t.ns = factor(-o.s);
  t.w2 = shl(o.w, 1);
}
// v[0..3] = bias + sigma_s (J cos, J sin, Y cos, Y sin of s phi) (Q64) of the order with J_s = j, Y_s = y,
// then e^{i (s+1) phi}, and jn, yn from order s - 1 to s + 1 with the factor f.
LSMS_HD void pair_order(int64_t j, int64_t y, int64_t& jn, int64_t& yn, int64_t fs, PairState& a, const PairStep& t,
                        int64_t bias, int64_t* v) {
  const Factor jf = factor(shl(j, 2)), yf = factor(shl(y, 2));         // Q65
  const Factor c = factor(a.c), s = factor(a.s), f = factor(fs);
  v[0] = madq(jf, c, bias);
  v[1] = madq(jf, s, bias);
  v[2] = madq(yf, c, bias);
  v[3] = madq(yf, s, bias);
  jn = madq(jf, f, jn);                                          // Q63
  yn = madq(yf, f, yn);
  a.c = shl(mulq2(c, t.c, s, t.ns), 2);
  a.s = shl(mulq2(s, t.c, c, t.s), 2);
}
// The products of the even order s (v[0..3]) and of s + 1 (v[4..7]), then on to s + 2.
LSMS_HD void pair_two_orders(PairState& a, const PairStep& t, int64_t bias, int64_t* v) {
  pair_order(a.je, a.ye, a.jo, a.yo, a.fe, a, t, bias, v);
  pair_order(a.jo, a.yo, a.je, a.ye, a.fo, a, t, bias, v + 4);
  a.fe += t.w2;
  a.fo -= t.w2;
}

#undef LSMS_Q
#undef LSMS_Q32

}  // namespace

// Host: the constants of wavenumber k, pairs with k rho < z_near left out.
inline PairConsts pair_consts(double k, double z_near) {
  const long double pi = 3.14159265358979323846264338327950288L;
  PairConsts q;
  const long double t = (long double)k / (2.0L * pi);
  q.turn_hi = (double)t;
  q.turn_lo = (double)(t - (long double)q.turn_hi);
  q.inv_k = (double)(1.0L / (long double)k);
  q.amp = (double)(sqrtl(2.0L / (pi * (long double)k)) / (1.0L - 0x1p-30L));   // 1 / R of PairState
  q.near_r2 = (float)((z_near / k) * (z_near / k));
  return q;
}
// Smallest k rho of the pairs formed in fixed point: Hankel's expansion from 26 on, and 2p orders
// that stay within the oscillating range.
inline double pair_z_near(int p) { return p <= 11 ? 26.0 : 2.0 * p + 4.0; }
