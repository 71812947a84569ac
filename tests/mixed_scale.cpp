// The mixed mode (float storage) with its D-solves in float pairs and in double, over models
// whose masses and inertias are scaled by 1e-33 to 1e32: host builds of one step and its
// adjoint, link frames (free and revolute roots, with and without ground contacts) and
// world-aligned.  Prints: formulation, scale, and the mean error of the worst output against
// an all-FP64 run, pairs then double.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2109_07719_gb300/csrc/contact.cuh"
#include "../paper_2109_07719_gb300/csrc/tree_order.h"
#include "../paper_2109_07719_gb300/csrc/wstep.cuh"

using namespace abasim;
using D = double;
using Vec = std::vector<D>;
static std::mt19937_64 rng;
static D U(D lo = -1, D hi = 1) { return (float)std::uniform_real_distribution<D>(lo, hi)(rng); }

constexpr int N = 7;
static const int kParent[N] = {-1, 0, 1, 0, 3, 0, 5};
static const D kDt = 1e-2;
struct Model {
  std::vector<int> meta;
  Vec prm;
  int nq = 0, nv = 0, depth = 0;
};

static Model build(bool free_root, D scale, bool contact) {
  Model m;
  const TreeOrder to = tree_order(kParent, N);
  m.depth = to.depth;
  m.prm.assign(N * NPRM * LANES, 0.0);
  m.meta.resize(N * LANES);
  for (int l = 0; l < N; ++l) {
    auto P = [&](int f) -> D& { return m.prm[(l * NPRM + f) * LANES]; };
    const bool fr = free_root && l == 0;
    D q[4], nn = 0;
    for (D& x : q) { x = U(); nn += x * x; }
    for (D& x : q) x /= std::sqrt(nn);
    const M3<D> E = quat_R(q[0], q[1], q[2], q[3]);
    for (int i = 0; i < 9; ++i) P(P_E + i) = (float)E.a[i];
    for (int i = 0; i < 3; ++i) {
      P(P_R + i) = U(-0.3, 0.3);
      P(P_C + i) = U(-0.1, 0.1);
      P(P_IC + i) = (float)(scale * U(0.02, 0.1));
      P(P_IC + 3 + i) = (float)(scale * U(-0.005, 0.005));
      P(P_CP + i) = U(-0.05, 0.05);
    }
    P(P_AX + 2) = fr ? 0 : 1;
    P(P_M) = (float)(scale * U(0.5, 2));
    P(P_CR) = contact && l > 0 && l % 2 == 0 ? 20.0 : -1.0;  // a sphere so large that it always touches
    P(P_LO) = -INFINITY;
    P(P_HI) = INFINITY;
    m.meta[l * LANES] = make_meta(to.parent[l], fr ? J_FREE : J_REVOLUTE, to.branch[l], m.nq, m.nv, to.lastsib[l]);
    m.nq += fr ? 7 : 1;
    m.nv += fr ? 6 : 1;
  }
  return m;
}

struct Inputs6 { Vec q, qd, tau, gq, gqd; };
enum Form { LINK, WORLD, CONTACT };

template <class T> static std::vector<T> cast(const Vec& v) { return std::vector<T>(v.begin(), v.end()); }
template <class T, class DT, Form F, bool FR> static std::vector<Vec> run(const Model& m, const Inputs6& x) {
  auto prm = cast<T>(m.prm), q = cast<T>(x.q), qd = cast<T>(x.qd), tau = cast<T>(x.tau), gq = cast<T>(x.gq), gv = cast<T>(x.gqd);
  const V3<T> g{T(0), T(0), T(-9.81)};
  const T dt = (T)kDt;
  std::vector<T> qo = q, vo = qd, gt(m.nv), gm(N, T(0));
  const Col<const T> qc{q.data(), 1}, vc{qd.data(), 1}, tc{tau.data(), 1};
  const Col<T> a{gq.data(), 1}, b{gv.data(), 1}, c{gt.data(), 1}, d{gm.data(), 1}, o{qo.data(), 1}, p{vo.data(), 1};
  if constexpr (F == WORLD) {
    std::vector<T> wt(N * NWT * LANES), wa(N * NWA * LANES), stk((m.depth + 1) * WSW * LANES), root(NWF * LANES);
    WSys<T> w{prm.data(), m.meta.data(), wt.data(), wa.data(), N};
    w.stk = stk.data();
    w.root = root.data();
    wstep_forward<T, DT, true, true, FR>(w, qc, vc, tc, g, dt, I_SEMI_IMPLICIT, o, p);
    wstep_adjoint<T, DT, FR>(w, a, b, c, d, dt, I_SEMI_IMPLICIT, g);
  } else {
    std::vector<T> tp(N * NTAPE * LANES), ad(N * NADJ * LANES), ct(N * NCT * LANES), cs(NCS * LANES);
    Sys<T> s{prm.data(), m.meta.data(), tp.data(), ad.data(), N};
    aba_forward<T, DT, true>(s, qc, vc, tc, g);
    if constexpr (F == CONTACT) {
      const CView<T> cv{ct.data(), cs.data()};
      const ContactParams<T> cp{T(0.8), T(0.2), 20};
      contact_forward<T, DT, T>(s, cv, qc, vc, dt, cp);
      integrate<T>(s, o, p, dt, I_SEMI_IMPLICIT, (const T*)ct.data());
      for (int l = 0; l < N; ++l) {
        const int mt = s.M(l);
        T qb[6] = {0, 0, 0, 0, 0, 0};
        integrator_adjoint(s, l, meta_jtype(mt), meta_qoff(mt), meta_voff(mt), qc, vc, a, b, dt, I_SEMI_IMPLICIT, qb,
                           (const T*)ct.data());
        for (int i = 0; i < 6; ++i) cv.L(l, C_QDDB + i) = qb[i];
      }
      contact_adjoint<T, DT, T>(s, cv, dt, cp);
      step_adjoint<T, DT>(s, qc, vc, a, b, c, d, g, dt, I_SEMI_IMPLICIT, (const T*)ct.data());
    } else {
      integrate<T>(s, o, p, dt, I_SEMI_IMPLICIT);
      step_adjoint<T, DT>(s, qc, vc, a, b, c, d, g, dt, I_SEMI_IMPLICIT);
    }
  }
  return {Vec(qo.begin(), qo.end()), Vec(vo.begin(), vo.end()), Vec(gq.begin(), gq.end()), Vec(gv.begin(), gv.end()),
          Vec(gt.begin(), gt.end()), Vec(gm.begin(), gm.end())};
}

static D worst(const std::vector<Vec>& want, const std::vector<Vec>& got) {
  D e = 0;
  for (size_t k = 0; k < want.size(); ++k) {
    D d = 0, m = 0;
    for (size_t i = 0; i < want[k].size(); ++i) {
      if (!std::isfinite(got[k][i])) return INFINITY;
      d = std::max(d, std::fabs(want[k][i] - got[k][i]));
      m = std::max(m, std::fabs(want[k][i]));
    }
    e = std::max(e, d / m);
  }
  return e;
}

template <Form F, bool FR> static void scan(const char* name) {
  for (D scale : {1e-33, 1e-28, 1e-22, 1e-18, 1e-9, 1.0, 1e9, 1e18, 1e22, 1e28, 1e32}) {
    if (F == CONTACT && (scale < 1e-30 || scale > 1e30)) continue;  // A of the rows leaves float's range
    rng.seed(2109077198);
    D pairs = 0, dbl = 0;
    const int trials = 40;
    for (int t = 0; t < trials; ++t) {
      const Model m = build(FR, scale, F == CONTACT);
      Inputs6 x{Vec(m.nq), Vec(m.nv), Vec(m.nv), Vec(m.nq), Vec(m.nv)};
      for (Vec* v : {&x.q, &x.qd, &x.gq, &x.gqd})
        for (D& y : *v) y = U();
      for (D& y : x.tau) y = (float)(scale * U());
      if (FR) {
        D nn = 0;
        for (int i = 3; i < 7; ++i) nn += x.q[i] * x.q[i];
        for (int i = 3; i < 7; ++i) x.q[i] = (float)(x.q[i] / std::sqrt(nn));
      }
      const auto want = run<D, D, F, FR>(m, x);
      pairs += worst(want, run<float, FF, F, FR>(m, x)) / trials;
      dbl += worst(want, run<float, D, F, FR>(m, x)) / trials;
    }
    std::printf("%s %.0e %.3e %.3e\n", name, scale, pairs, dbl);
  }
}

int main() {
  scan<LINK, false>("link");
  scan<LINK, true>("link_free");
  scan<WORLD, false>("world");
  scan<WORLD, true>("world_free");
  scan<CONTACT, true>("contact");
}
