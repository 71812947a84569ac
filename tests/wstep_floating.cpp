// Host FP64 check of the world-aligned step with a free root (csrc/wstep.cuh, FR)
// against the link-frame step and its adjoint (csrc/aba_step.cuh) on random floating
// trees of 1 to 12 links, both integrators, gravity in a general direction: two
// formulations of the same step and gradient, so they agree to rounding.  The stack
// is exactly as deep as the order says with NaN guard entries after it, and every
// adjoint word starts as NaN.  Prints per tree: links, error of the new state, of
// the gradients in q, qd, tau and the masses, of four steps by the fused pass against whole
// steps (each relative to the largest entry), and
// whether the guards are intact.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2109_07719_gb300/csrc/tree_order.h"
#include "../paper_2109_07719_gb300/csrc/wstep.cuh"

using namespace abasim;
using D = double;
using Vec = std::vector<D>;

static std::mt19937_64 rng(2109077194);
static D U(D lo = -1, D hi = 1) { return std::uniform_real_distribution<D>(lo, hi)(rng); }

static D err(const Vec& a, const Vec& b) {
  D e = 0, m = 0;
  for (size_t i = 0; i < a.size(); ++i) {
    if (!std::isfinite(b[i])) return 1e300;
    e = std::max(e, std::fabs(a[i] - b[i]));
    m = std::max(m, std::fabs(a[i]));
  }
  return e / m;
}

int main() {
  for (int trial = 0; trial < 24; ++trial) {
    const int n = 1 + trial % 12, integ = trial % 2 ? I_EXPLICIT : I_SEMI_IMPLICIT;
    std::vector<int> par{-1};
    for (int i = 1; i < n; ++i) par.push_back((int)(U(0, 1) * i) % i);
    const TreeOrder to = tree_order(par.data(), n);
    Vec prm(n * NPRM * LANES, 0.0), tp(n * NTAPE * LANES), ad(n * NADJ * LANES);
    Vec wt(n * NWT * LANES, NAN), wa(n * NWA * LANES, NAN), stk((to.depth + 2) * WSW * LANES, NAN);
    Vec root(NWF * LANES, NAN);
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
      P(P_DAMP) = l ? U(0, 0.5) : 0.0;
      meta[l * LANES] = make_meta(to.parent[l], l ? J_REVOLUTE : J_FREE, to.branch[l], nq, nv, to.lastsib[l]);
      nq += l ? 1 : 7;
      nv += l ? 1 : 6;
    }
    const V3<D> g{0.3, -1.0, -9.81};
    const D dt = 0.5;  // large, so that the step's own part of the gradients is not small
    Vec q(nq), qd(nv), tau(nv), gq(nq), gqd(nv);
    for (Vec* v : {&q, &qd, &tau, &gq, &gqd})
      for (D& x : *v) x = U();
    D nn = 0;
    for (int i = 3; i < 7; ++i) nn += q[i] * q[i];
    for (int i = 3; i < 7; ++i) q[i] /= std::sqrt(nn);
    const Col<const D> qc{q.data(), 1}, qdc{qd.data(), 1}, tc{tau.data(), 1};
    Sys<D> s{prm.data(), meta.data(), tp.data(), ad.data(), n};
    Vec xa = q, va = qd, gqa = gq, gqda = gqd, gta(nv), gma(n, 0.0);
    aba_forward<D, D, true>(s, qc, qdc, tc, g);
    step_adjoint<D, D>(s, qc, qdc, Col<D>{gqa.data(), 1}, Col<D>{gqda.data(), 1}, Col<D>{gta.data(), 1},
                       Col<D>{gma.data(), 1}, g, dt, integ);
    integrate<D>(s, Col<D>{xa.data(), 1}, Col<D>{va.data(), 1}, dt, integ);
    WSys<D> w{prm.data(), meta.data(), wt.data(), wa.data(), n};
    w.stk = stk.data();
    w.root = root.data();
    Vec xb = q, vb = qd, gqb = gq, gqdb = gqd, gtb(nv), gmb(n, 0.0);
    wstep_forward<D, D, false, true, true>(w, Col<const D>{xb.data(), 1}, Col<const D>{vb.data(), 1}, tc, g, dt, integ,
                                           Col<D>{xb.data(), 1}, Col<D>{vb.data(), 1});
    std::fill(wt.begin(), wt.end(), NAN);
    wstep_forward<D, D, true, false, true>(w, qc, qdc, tc, g, dt, integ, Col<D>{nullptr, 0}, Col<D>{nullptr, 0});
    wstep_adjoint<D, D, true>(w, Col<D>{gqb.data(), 1}, Col<D>{gqdb.data(), 1}, Col<D>{gtb.data(), 1},
                              Col<D>{gmb.data(), 1}, dt, integ, g);
    // a rollout's fused pass (accelerations of one step, pose of the next) against whole steps
    Vec qf = q, vf = qd, qs = q, vs = qd;
    const Col<D> qfc{qf.data(), 1}, vfc{vf.data(), 1};
    const Col<const D> qfr{qf.data(), 1}, vfr{vf.data(), 1};
    const D h = 1e-2;
    for (int t = 0; t < 4; ++t) {
      if (t == 0)
        wpass_pose<D, D, false, true>(w, qfr, vfr);
      else
        wpass_accel_pose<D, D, true>(w, qfr, vfr, g, h, integ, qfc, vfc);
      wpass_inward<D, D, false, true>(w, vfr, tc);
    }
    wpass_accel<D, D, false, true, true>(w, qfr, vfr, g, h, integ, qfc, vfc);
    for (int t = 0; t < 4; ++t)
      wstep_forward<D, D, false, true, true>(w, Col<const D>{qs.data(), 1}, Col<const D>{vs.data(), 1}, tc, g, h, integ,
                                             Col<D>{qs.data(), 1}, Col<D>{vs.data(), 1});
    const D fused = std::max(err(qs, qf), err(vs, vf));
    bool guards = true;
    for (size_t i = (size_t)to.depth * WSW * LANES; i < stk.size(); ++i) guards &= std::isnan(stk[i]);
    std::printf("%d %.3e %.3e %.3e %.3e %.3e %.3e %d\n", n, std::max(err(xa, xb), err(va, vb)), err(gqa, gqb),
                err(gqda, gqdb), err(gta, gtb), err(gma, gmb), fused, guards ? 1 : 0);
  }
  return 0;
}
