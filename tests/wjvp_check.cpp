// Host FP64 check of the implicit-form JVP (csrc/wjvp.cuh) against the link-frame step
// run on dual numbers (csrc/dual.cuh): chains, branched trees, a forest and floating
// bases, damping, both integrators, gravity in a general direction.  Prints per model:
// links, error of x' and of its tangent (relative to the largest entry), stack guards.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2109_07719_gb300/csrc/tree_order.h"
#include "../paper_2109_07719_gb300/csrc/wjvp.cuh"

using namespace abasim;
using D = double;
using DD = Dual<double>;
using Vec = std::vector<D>;

static std::mt19937_64 rng(2109077196);
static D U(D lo = -1, D hi = 1) { return std::uniform_real_distribution<D>(lo, hi)(rng); }

template <bool FR> static void run(int trial) {
  const int n = 1 + trial % 11, integ = trial % 2 ? I_EXPLICIT : I_SEMI_IMPLICIT;
  std::vector<int> par{-1};
  for (int i = 1; i < n; ++i)
    par.push_back(trial % 3 == 0 ? i - 1 : (!FR && i % 5 == 4) ? -1 : (int)(U(0, 1) * i) % i);
  const TreeOrder to = tree_order(par.data(), n);
  Vec prm(n * NPRM * LANES, 0.0), wt(n * NWT * LANES, NAN), wj(n * NWJ * LANES, NAN);
  Vec stk((to.depth + 2) * WSW * LANES, NAN), root(NWF * LANES, NAN);
  std::vector<DD> tp(n * NTAPE * LANES);
  std::vector<int> meta(n * LANES);
  int nq = 0, nv = 0;
  for (int l = 0; l < n; ++l) {
    auto P = [&](int f) -> D& { return prm[(l * NPRM + f) * LANES]; };
    const bool fr = FR && l == 0;
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
    P(P_DAMP) = fr ? 0.0 : U(0, 0.5);
    meta[l * LANES] = make_meta(to.parent[l], fr ? J_FREE : J_REVOLUTE, to.branch[l], nq, nv, to.lastsib[l]);
    nq += fr ? 7 : 1;
    nv += fr ? 6 : 1;
  }
  const V3<D> g{0.3, -1.0, -9.81};
  const D dt = 0.5;  // large, so that the accelerations' part of the tangents is not small
  Vec q(nq), qd(nv), tau(nv), dq(nq), dqd(nv), dtau(nv);
  for (Vec* v : {&q, &qd, &tau, &dq, &dqd, &dtau})
    for (D& x : *v) x = U();
  if (FR) {
    D nn = 0;
    for (int i = 3; i < 7; ++i) nn += q[i] * q[i];
    for (int i = 3; i < 7; ++i) q[i] /= std::sqrt(nn);
  }
  std::vector<DD> xq(nq), xv(nv), xt(nv);
  for (int i = 0; i < nq; ++i) xq[i] = DD(q[i], dq[i]);
  for (int i = 0; i < nv; ++i) { xv[i] = DD(qd[i], dqd[i]); xt[i] = DD(tau[i], dtau[i]); }
  Sys<DD, D> s{prm.data(), meta.data(), tp.data(), nullptr, n, 1};
  aba_forward<DD, DD, false>(s, Col<const DD>{xq.data(), 1}, Col<const DD>{xv.data(), 1}, Col<const DD>{xt.data(), 1},
                             V3<DD>{DD(g.x), DD(g.y), DD(g.z)});
  integrate<DD>(s, Col<DD>{xq.data(), 1}, Col<DD>{xv.data(), 1}, DD(dt), integ);
  WSys<D> w{prm.data(), meta.data(), wt.data(), wj.data(), n};
  w.stk = stk.data();
  w.root = root.data();
  const Col<const D> qc{q.data(), 1}, qdc{qd.data(), 1}, tc{tau.data(), 1};
  Vec q2(nq), v2(nv), dq2(nq), dv2(nv);
  wstep_forward<D, D, true, false, FR>(w, qc, qdc, tc, g, dt, integ, Col<D>{nullptr, 0}, Col<D>{nullptr, 0});
  wstep_jvp<D, D, FR>(w, qc, qdc, Col<const D>{dq.data(), 1}, Col<const D>{dqd.data(), 1},
                      Col<const D>{dtau.data(), 1}, g, dt, integ, Col<D>{q2.data(), 1}, Col<D>{v2.data(), 1},
                      Col<D>{dq2.data(), 1}, Col<D>{dv2.data(), 1});
  D ev = 0, mv = 0, et = 0, mt = 0;
  auto cmp = [](D a, D b, D& e, D& m) {
    e = std::isfinite(b) ? std::max(e, std::fabs(a - b)) : 1e300;
    m = std::max(m, std::fabs(a));
  };
  for (int i = 0; i < nq; ++i) { cmp(xq[i].v, q2[i], ev, mv); cmp(xq[i].d, dq2[i], et, mt); }
  for (int i = 0; i < nv; ++i) { cmp(xv[i].v, v2[i], ev, mv); cmp(xv[i].d, dv2[i], et, mt); }
  bool guards = true;
  for (size_t i = (size_t)to.depth * WSW * LANES; i < stk.size(); ++i) guards &= std::isnan(stk[i]);
  std::printf("%d %d %.3e %.3e %d\n", FR ? 1 : 0, n, ev / mv, et / mt, guards ? 1 : 0);
}

int main() {
  for (int t = 0; t < 33; ++t) run<false>(t);
  for (int t = 0; t < 33; ++t) run<true>(t);
  return 0;
}
