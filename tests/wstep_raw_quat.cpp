// Host FP64 check of the world-aligned step with a free root (csrc/wstep.cuh, csrc/wjvp.cuh)
// on states whose quaternion is not of unit length: the step takes R(quat) as it is given,
// as the link-frame step (csrc/aba_step.cuh) does, so states, gradients and tangents agree
// to rounding there too.  Prints per case: the quaternion's length, error of the new state,
// of the gradients in q, qd and tau, and of the JVP against the adjoint (the dot product),
// each relative to the largest entry.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2109_07719_gb300/csrc/tree_order.h"
#include "../paper_2109_07719_gb300/csrc/wjvp.cuh"

using namespace abasim;
using D = double;
using Vec = std::vector<D>;
using C = Col<const D>;

static std::mt19937_64 rng(77);
static D U(D lo = -1, D hi = 1) { return std::uniform_real_distribution<D>(lo, hi)(rng); }
static Col<D> col(Vec& v) { return Col<D>{v.data(), 1}; }
static C ccol(const Vec& v) { return C{v.data(), 1}; }
static D err(const Vec& a, const Vec& b) {
  D e = 0, m = 0;
  for (size_t i = 0; i < a.size(); ++i) {
    if (!std::isfinite(b[i])) return 1e300;
    e = std::max(e, std::fabs(a[i] - b[i]));
    m = std::max(m, std::fabs(a[i]));
  }
  return e / m;
}
static D inner(const Vec& a, const Vec& b) {
  D s = 0;
  for (size_t i = 0; i < a.size(); ++i) s += a[i] * b[i];
  return s;
}

int main() {
  const int n = 5, par[n] = {-1, 0, 1, 0, 3};
  const TreeOrder to = tree_order(par, n);
  for (D length : {0.8, 1.0 - 6e-8, 1.0, 1.0 + 1e-3, 1.5}) {
    for (int integ : {I_SEMI_IMPLICIT, I_EXPLICIT}) {
      Vec prm(n * NPRM * LANES, 0.0), tp(n * NTAPE * LANES), ad(n * NADJ * LANES), wt(n * NWT * LANES, NAN);
      Vec wa(n * NWJ * LANES, NAN), stk((to.depth + 1) * WSW * LANES, NAN), root(NWF * LANES, NAN);
      std::vector<int> meta(n * LANES);
      int nq = 0, nv = 0;
      for (int l = 0; l < n; ++l) {
        auto P = [&](int f) -> D& { return prm[(l * NPRM + f) * LANES]; };
        D q4[4], nn = 0;
        for (D& x : q4) { x = U(); nn += x * x; }
        nn = std::sqrt(nn);
        const M3<D> E = quat_R(q4[0] / nn, q4[1] / nn, q4[2] / nn, q4[3] / nn);
        for (int i = 0; i < 9; ++i) P(P_E + i) = E.a[i];
        for (int i = 0; i < 3; ++i) {
          P(P_R + i) = U(-0.4, 0.4);
          P(P_C + i) = U(-0.2, 0.2);
          P(P_IC + i) = U(0.05, 0.15);
          P(P_IC + 3 + i) = U(-0.01, 0.01);
        }
        P(P_M) = U(0.5, 2.0);
        meta[l * LANES] = make_meta(to.parent[l], l ? J_REVOLUTE : J_FREE, to.branch[l], nq, nv, to.lastsib[l]);
        nq += l ? 1 : 7;
        nv += l ? 1 : 6;
      }
      const V3<D> g{0.3, -1.0, -9.81};
      const D dt = 0.1;
      Vec q(nq), qd(nv), tau(nv), gq(nq), gqd(nv), dq(nq), dqd(nv), dtau(nv);
      for (Vec* v : {&q, &qd, &tau, &gq, &gqd, &dq, &dqd, &dtau})
        for (D& x : *v) x = U();
      D nn = 0;
      for (int i = 3; i < 7; ++i) nn += q[i] * q[i];
      for (int i = 3; i < 7; ++i) q[i] *= length / std::sqrt(nn);
      Sys<D> s{prm.data(), meta.data(), tp.data(), ad.data(), n};
      Vec xa = q, va = qd, gqa = gq, gqda = gqd, gta(nv), gma(n, 0.0);
      aba_forward<D, D, true>(s, ccol(q), ccol(qd), ccol(tau), g);
      step_adjoint<D, D>(s, ccol(q), ccol(qd), col(gqa), col(gqda), col(gta), col(gma), g, dt, integ);
      integrate<D>(s, col(xa), col(va), dt, integ);
      WSys<D> w{prm.data(), meta.data(), wt.data(), wa.data(), n};
      w.stk = stk.data();
      w.root = root.data();
      Vec xb(nq), vb(nv), gqb = gq, gqdb = gqd, gtb(nv), gmb(n, 0.0);
      wstep_forward<D, D, true, true, true>(w, ccol(q), ccol(qd), ccol(tau), g, dt, integ, col(xb), col(vb));
      wstep_adjoint<D, D, true>(w, col(gqb), col(gqdb), col(gtb), col(gmb), dt, integ, g);
      wstep_forward<D, D, true, false, true>(w, ccol(q), ccol(qd), ccol(tau), g, dt, integ, Col<D>{nullptr, 0},
                                             Col<D>{nullptr, 0});
      Vec xj(nq), vj(nv), dxj(nq), dvj(nv);
      wstep_jvp<D, D, true>(w, ccol(q), ccol(qd), ccol(dq), ccol(dqd), ccol(dtau), g, dt, integ, col(xj), col(vj),
                            col(dxj), col(dvj));
      const D fwd = inner(gq, dxj) + inner(gqd, dvj), rev = inner(gqa, dq) + inner(gqda, dqd) + inner(gta, dtau);
      std::printf("%.9f %.3e %.3e %.3e %.3e %.3e\n", length, std::max({err(xa, xb), err(va, vb), err(xa, xj), err(va, vj)}),
                  err(gqa, gqb), err(gqda, gqdb), err(gta, gtb), std::fabs(fwd - rev) / std::fabs(rev));
    }
  }
  return 0;
}
