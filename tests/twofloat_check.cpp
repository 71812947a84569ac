// Float-pair arithmetic of the mixed mode's D-solves (csrc/twofloat.cuh) against double
// and long double, host build.  Prints: name, worst error relative to the largest term.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_2109_07719_gb300/csrc/aba_step.cuh"

using namespace abasim;
static std::mt19937_64 rng(2109077195);
static float U(double lo, double hi) { return (float)std::uniform_real_distribution<double>(lo, hi)(rng); }
static long double val(FF x) { return (long double)x.h + x.l; }

int main() {
  long double recip = 0, root = 0, mul = 0, add = 0, prod = 0, solve = 0;
  for (int i = 0; i < 300000; ++i) {
    const float s = std::ldexp(1.0f, (int)U(-30, 30));
    const float d = s * U(0.01, 2), u = U(-2, 2), v = U(-2, 2), a = (i % 3 == 0) ? u * v / d : U(-2, 2) / s;
    const FF di = FF(1) / FF(d), x = di * FF(u);
    recip = std::fmax(recip, std::fabs(val(di) * d - 1));
    root = std::fmax(root, std::fabs(val(ff_sqrt(FF(d))) / sqrtl(d) - 1));
    if (u != 0) mul = std::fmax(mul, std::fabs(val(x) / (val(di) * u) - 1));
    add = std::fmax(add, std::fabs(val(x + di) - (val(x) + val(di))) / (std::fabs(val(x)) + val(di)));
    const long double want = (long double)a - val(x) * v;
    const float got = minus_product<float, FF>(a, x, v);
    // past the rounding to float: what is left, relative to the larger of the two terms
    const long double ulp = std::ldexp(1.0L, std::ilogb((double)got + 1e-300) - 24);
    prod = std::fmax(prod, (std::fabs(got - want) - ulp) / (std::fabs(a) + std::fabs(val(x) * v)));
  }
  for (int t = 0; t < 2000; ++t) {
    float A[6][6], M[6][6];
    for (auto& r : A)
      for (float& y : r) y = U(-2, 2);
    for (int i = 0; i < 6; ++i)
      for (int j = 0; j < 6; ++j) {
        double s = i == j ? 0.1 : 0;
        for (int k = 0; k < 6; ++k) s += (double)A[i][k] * A[j][k];
        M[i][j] = (float)s;
      }
    SI<float> I;
    I.A = S3<float>{M[0][0], M[1][1], M[2][2], M[0][1], M[0][2], M[1][2]};
    I.C = S3<float>{M[3][3], M[4][4], M[5][5], M[3][4], M[3][5], M[4][5]};
    for (int i = 0; i < 9; ++i) I.B.a[i] = M[i / 3][3 + i % 3];
    const SV<float> b{{U(-1, 1), U(-1, 1), U(-1, 1)}, {U(-1, 1), U(-1, 1), U(-1, 1)}};
    const SV<float> p = spd_solve<float, FF>(I, b), q = spd_solve<float, double>(I, b), e = p - q;
    solve = std::fmax(solve, std::sqrt(dot(e, e) / dot(q, q)));
  }
  const float inf = INFINITY;
  const bool special = minus_product<float, FF>(inf, FF(1), 2) == inf && minus_product<float, FF>(1, FF(inf), 2) == -inf &&
                       std::isnan(minus_product<float, FF>(NAN, FF(1), 2));
  std::printf("reciprocal %.3Le\nsqrt %.3Le\nproduct %.3Le\nsum %.3Le\nminus_product %.3Le\nsolve %.3Le\nspecial %d\n", recip,
              root, mul, add, prod, solve, special ? 1 : 0);
  return 0;
}
