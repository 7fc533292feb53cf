// exp(-x) and 1 - exp(-x) in FP64 for 2^-6 <= x < 8 by table and series.
//
// x = i/64 + s with |s| <= 1/128: exp(-x) = E_i (1 + e), e = expm1(-s) by its
// Taylor series through s^6 (the rest is below 2^-61), and 1 - exp(-x) = P_i - E_i e
// with P_i = 1 - E_i tabulated on its own.  Eight FP64 instructions, where the
// library's expm1 takes a multiple: the FP64 step is bound by their number (one
// warp instruction every 19 clocks per SM).  The index is formed in FP32 and integer
// arithmetic, which costs nothing beside them.
//
// The table is computed at compile time in double-double arithmetic: exp(i/64) by
// repeated multiplication with exp(1/64) (its Taylor series), then one division.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

struct DD { double h, l; };

constexpr DD dd_two_sum(double a, double b) {
  const double s = a + b, bb = s - a;
  return DD{s, (a - (s - bb)) + (b - bb)};
}
constexpr DD dd_two_prod(double a, double b) {   // Dekker's product
  const double c = 134217729.0;
  const double ac = c * a, ah = ac - (ac - a), al = a - ah;
  const double bc = c * b, bh = bc - (bc - b), bl = b - bh;
  const double p = a * b;
  return DD{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD dd_add(DD a, DD b) {
  const DD s = dd_two_sum(a.h, b.h);
  return dd_two_sum(s.h, s.l + (a.l + b.l));
}
constexpr DD dd_mul(DD a, DD b) {
  const DD p = dd_two_prod(a.h, b.h);
  return dd_two_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD dd_inv(DD a) {   // 1/a, one Newton step on the rounded quotient
  const double y = 1.0 / a.h;
  const DD r = dd_add(DD{1.0, 0.0}, dd_mul(a, DD{-y, 0.0}));
  return dd_two_sum(y, y * (r.h + r.l));
}

constexpr int kExpEntries = 512;   // x in [0, 8), 1/64 apart
struct ExpTable {
  double2 v[kExpEntries];   // E_i = exp(-i/64), P_i = 1 - E_i
};
constexpr ExpTable make_exp_table() {
  ExpTable t{};
  // exp(1/64) by its Taylor series, the terms from the smallest up
  DD e1{1.0, 0.0};
  for (int k = 14; k >= 1; --k) {
    // e1 = 1 + e1 / (64 k)
    const DD inv = dd_inv(DD{64.0 * k, 0.0});
    e1 = dd_add(DD{1.0, 0.0}, dd_mul(e1, inv));
  }
  DD x{1.0, 0.0};
  for (int i = 0; i < kExpEntries; ++i) {
    const DD E = dd_inv(x);
    const DD P = dd_add(DD{1.0, 0.0}, DD{-E.h, -E.l});
    t.v[i].x = E.h;
    t.v[i].y = P.h;
    x = dd_mul(x, e1);
  }
  return t;
}
static __device__ constexpr ExpTable kExpTab = make_exp_table();

// exp(-x) (ONE_MINUS: 1 - exp(-x)) for 2^-6 <= x < 7.99; the caller keeps other
// arguments away (exp_arg_ok)
__device__ __forceinline__ bool exp_arg_ok(double x) {
  // 2^-6 = 0x3F900000.., 7.9921875 = 0x401FF800..
  return (unsigned)(__double2hiint(x) - 0x3F900000) < 0x401FF800u - 0x3F900000u;
}
template <bool ONE_MINUS>
__device__ __forceinline__ double exp_neg_table(double x) {
  // x to float by its bits (truncated to 20 bits of mantissa), rounded to i/64
  const float xf = __int_as_float((__double2hiint(x) - 0x38000000) << 3);
  const float m = __fmaf_rn(xf, 64.0f, 12582912.0f);            // 1.5 2^23: i in the low bits
  const int i = __float_as_int(m) & 0x3ff;
  const float c = __fmul_rn(__fsub_rn(m, 12582912.0f), 0.015625f);   // i/64, exact; i >= 1
  const double ci = __hiloint2double((__float_as_int(c) >> 3) + 0x38000000, 0);
  const double2 t = kExpTab.v[i];
  const double s = __dsub_rn(ci, x);   // -s of the text: exp(-x) = E exp(s)
  double h = __fma_rn(s, 1.0 / 720.0, 1.0 / 120.0);
  h = __fma_rn(s, h, 1.0 / 24.0);
  h = __fma_rn(s, h, 1.0 / 6.0);
  h = __fma_rn(s, h, 0.5);
  const double e = __fma_rn(__dmul_rn(s, s), h, s);             // expm1(s)
  return ONE_MINUS ? __fma_rn(-t.x, e, t.y) : __fma_rn(t.x, e, t.x);
}

}  // namespace lbm
