// A number held as the unevaluated sum of two floats, h + l with |l| <= ulp(h) / 2: 48
// significant bits out of FP32 instructions, by the error-free transformations of Dekker
// (1971) and Knuth (The Art of Computer Programming 2, 4.2.2).  The mixed mode's D-solves
// run in it.  In double, an instruction costs a warp 64 cycles on this chip's
// half-lane-per-cycle FP64 units, and the 140 of them a link (the rank-one update of the
// articulated inertia with its 42 conversions, 1/D and the products with it) were nearly all
// of its step: rollout + adjoint of 8192 quadrupeds over 60 steps 9.2 ms in double, 4.7 in
// pairs; of 4096 7-link chains over 100 steps 6.5 and 1.1 (with the implicit-form adjoint).
//
// Precision: every use rounds its result to float from at least 44 bits of its largest term,
// so it differs from double's in about one rounding of 2^20, and the errors against 64 bits
// are double's (0.66e-6, 0.63e-6 and, for 333 16-link chains, 0.81e-6; in double 0.68e-6,
// 0.63e-6, 0.85e-6).  Range: a pair has float's exponents.  Its low half is lost below 2^-101
// of the largest term, where float's own rounding is all that is left of double's advantage;
// products of several factors are formed one at a time so that none leaves float's range.
// Masses scaled by 1e-33 to 1e32 give double's errors throughout (tests/mixed_scale.cpp).
#pragma once

#include "spatial.cuh"

namespace abasim {

struct FF {
  float h, l;
  FF() = default;
  SD FF(float x) : h(x), l(0.0f) {}
  SD FF(float hi, float lo) : h(hi), l(lo) {}
  SD explicit operator float() const { return h + l; }
};

// single rounded operations, never contracted
#ifdef __CUDA_ARCH__
SD float ff_mul(float a, float b) { return __fmul_rn(a, b); }
SD float ff_add(float a, float b) { return __fadd_rn(a, b); }
SD float ff_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
SD float ff_mul(float a, float b) { volatile float r = a * b; return r; }
SD float ff_add(float a, float b) { volatile float r = a + b; return r; }
SD float ff_fma(float a, float b, float c) { return std::fma(a, b, c); }
#endif

// a + b exactly (any order of magnitude); for |a| >= |b|
SD FF ff_two_sum(float a, float b) {
  const float s = ff_add(a, b), bb = ff_add(s, -a);
  return FF(s, ff_add(ff_add(a, -ff_add(s, -bb)), ff_add(b, -bb)));
}
SD FF ff_fast_sum(float a, float b) {
  const float s = ff_add(a, b);
  return FF(s, ff_add(b, -ff_add(s, -a)));
}
SD FF operator-(FF a) { return FF(-a.h, -a.l); }
SD FF operator+(FF a, FF b) {
  const FF s = ff_two_sum(a.h, b.h);
  return ff_fast_sum(s.h, ff_add(s.l, ff_add(a.l, b.l)));
}
SD FF operator-(FF a, FF b) { return a + (-b); }
SD FF operator*(FF a, FF b) {
  const float p = ff_mul(a.h, b.h);
  return ff_fast_sum(p, ff_fma(a.h, b.l, ff_fma(a.l, b.h, ff_fma(a.h, b.h, -p))));
}
SD FF operator/(FF a, FF b) {
  const float r = 1.0f / b.h, q = ff_mul(a.h, r);
  const FF rest = a - b * FF(q);
  return ff_fast_sum(q, ff_mul(rest.h, r));
}
SD FF ff_sqrt(FF a) {
  const float s = sqrtf(a.h);
  const FF rest = a - FF(s) * FF(s);
  return ff_fast_sum(s, rest.h / (2.0f * s));
}
SD FF& operator+=(FF& a, FF b) { return a = a + b; }
SD FF& operator-=(FF& a, FF b) { return a = a - b; }
SD FF& operator*=(FF& a, FF b) { return a = a * b; }

// i - x u rounded once (an infinite or NaN part leaves the plain sum's value)
SD float ff_minus_product(float i, FF x, float u) {
  const float p = ff_mul(x.h, u);
  const FF s = ff_two_sum(i, -p);
  const float rest = ff_fma(-x.l, u, ff_add(s.l, -ff_fma(x.h, u, -p)));
  const float r = ff_add(s.h, rest);
  return r == r ? r : s.h;
}

}  // namespace abasim
