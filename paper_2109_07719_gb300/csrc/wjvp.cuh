// Forward-mode derivative of the world-aligned step, by the implicit form: from
// RNEA(q, qd, qdd) + b qd = tau,
//   dqdd = M^-1 (dtau - b dqd - dRNEA(q, qd, qdd)[dq, dqd])  at fixed qdd,
// with the U and 1/D of the step.  The tangents of a link's motions and forces are taken in
// axes that turn with the link (x -> dx - dphi x x), where its inertia, joint axis and COM
// offset are constant: going from a parent to its child subtracts (s dq) x, and back adds it.
// One directional RNEA (vectors only) and one solve take 530 operations a link beside the
// step's 670; the step on dual numbers took three times the link-frame step's 970 and a
// tape of 238 words a link.  In FP64: 700 9-link chains 602 -> 251 us, three trees of 2-30
// links 2180 -> 873 us, errors 2.8e-16 and 1e-16.
#pragma once

#include "dual.cuh"
#include "wstep.cuh"

namespace abasim {

// Per-link record of the tangent passes: the body force F and its tangent.
enum : int { WJ_F = 0, WJ_DF = 6, NWJ = 12 };

// Requires wstep_forward<ADJ = true>(q, qd, tau).  (q, qd) and the tangents (dq, dqd, dtau)
// in, x' and its tangent (dqo, dqdo) out; s.adj: [maxL][NWJ][LANES].
template <class T, class DT, bool FR, bool STG>
SD void wstep_jvp(const WSys<T, STG>& s, Col<const T> q, Col<const T> qd, Col<const T> dq, Col<const T> dqd,
                  Col<const T> dtau, V3<T> grav, T dt, int integ, Col<T> qo, Col<T> qdo, Col<T> dqo, Col<T> dqdo) {
  T* tp = s.tape;
  const int nl = s.nl, walk = s.walk();
  // tangents of the motions and body forces (root -> leaves)
  {
    Records<T, STG, 1, RING_ADJ, W_D, NWT - W_D, P_M, 1> rec(s, walk);
    SV<T> dv_prev = zeroSV<T>(), da_prev = zeroSV<T>();
    int sp = 0;
    for (int l = 0; l < walk; ++l) {
      rec.next();
      if (STG && l >= nl) continue;
      const int m = s.M(l);
      const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
      const bool fr = FR && meta_jtype(m) == J_FREE;
      const V3<T> sx = fld_v3(rec.t, W_S), rw = fld_v3(rec.t, W_RW);
      const SV<T> v = fld_sv(rec.t, W_V), ap = fld_sv(rec.t, W_AP);
      SV<T> a = ap, dv = zeroSV<T>(), da = zeroSV<T>();
      S3<T> Ic;
      if (fr) {  // v = qd, a = qdd + [0; -E g]
        dv = SV<T>{{dqd[vi], dqd[vi + 1], dqd[vi + 2]}, {dqd[vi + 3], dqd[vi + 4], dqd[vi + 5]}};
        Dual<T> x[4];
        for (int i = 0; i < 4; ++i) x[i] = Dual<T>(q[qi + 3 + i], dq[qi + 3 + i]);
        const M3<Dual<T>> Rq = quat_R(x[0], x[1], x[2], x[3]);
        M3<T> dEJ, Et;
        for (int i = 0; i < 9; ++i) {
          dEJ.a[i] = Rq.a[3 * (i % 3) + i / 3].d;
          Et.a[i] = s.P(l, P_E + i);
        }
        da.v = mul(dEJ, mul(Et, zero3<T>() - grav));
        Ic = ws3(s.root, 0, 0, WF_IC);
      } else {
        const T vl = fld(rec.t, W_QD), x = dq[qi], xd = dqd[vi];
        a.w = ap.w + fld(rec.t, W_QDD) * sx;
        Ic = fld_s3(rec.t, W_XY);
        if (par >= 0) {
          SV<T> dvp = dv_prev, dap = da_prev;
          if (par != l - 1) {
            dvp = wsv(s.stk, WSW, sp - 1, 0);
            dap = wsv(s.stk, WSW, sp - 1, 6);
            if (meta_lastsib(m)) --sp;
          }
          const V3<T> d = fld_v3(rec.t, W_D);
          dv = shift_motion(dvp, d);
          da = shift_motion(dap, d);
        }
        const SV<T> e{cross(sx, v.w), cross(sx, v.v)};
        const SV<T> as = ap + vl * e;  // the parent's acceleration handed down: a' less c = -qd e
        dv -= x * e;
        dv.w += xd * sx;
        const V3<T> sq = vl * sx;
        da += SV<T>{cross(dv.w, sq), cross(dv.v, sq)} - xd * e - x * SV<T>{cross(sx, as.w), cross(sx, as.v)};
      }
      // F = I a + v x* I v at the COM and its tangent
      const T mass = fld(rec.p, P_M);
      const V3<T> vc = v.v + cross(v.w, rw), dvc = dv.v + cross(dv.w, rw), Lw = mul(Ic, v.w);
      const V3<T> f = mass * (a.v + cross(a.w, rw) + cross(v.w, vc));
      const V3<T> df = mass * (da.v + cross(da.w, rw) + cross(dv.w, vc) + cross(v.w, dvc));
      wsv(s.adj, NWJ, l, WJ_F, SV<T>{mul(Ic, a.w) + cross(v.w, Lw) + cross(rw, f), f});
      wsv(s.adj, NWJ, l, WJ_DF, SV<T>{mul(Ic, da.w) + cross(dv.w, Lw) + cross(v.w, mul(Ic, dv.w)) + cross(rw, df), df});
      if (meta_treechild(m)) {
        wsv(s.stk, WSW, sp, 0, dv);
        wsv(s.stk, WSW, sp, 6, da);
        ++sp;
      }
      dv_prev = dv;
      da_prev = da;
    }
  }
  // joint force tangents and the inward half of the solve (leaves -> root)
  {
    Records<T, STG, -1, RING_ADJ, 0, W_XY, P_DAMP, 1, 0, NWJ, 0, 0, NWJ> rec(s, walk);
    SV<T> cf = zeroSV<T>(), cd = zeroSV<T>(), cy = zeroSV<T>();
    int sp = 0;
    for (int l = walk - 1; l >= 0; --l) {
      rec.next();
      if (STG && l >= nl) continue;
      const int m = s.M(l);
      const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
      SV<T> f = cf + fld_sv(rec.a, WJ_F), df = cd + fld_sv(rec.a, WJ_DF), y = cy;
      cf = cd = cy = zeroSV<T>();
      if (meta_treechild(m)) {
        --sp;
        f += wsv(s.stk, WSW, sp, 0);
        df += wsv(s.stk, WSW, sp, 6);
        y += wsv(s.stk, WSW, sp, 12);
      }
      if (FR && meta_jtype(m) == J_FREE) {  // dqdd of the root: (I^A)^-1 (dtau - df + y)
        const SV<T> t{{dtau[vi], dtau[vi + 1], dtau[vi + 2]}, {dtau[vi + 3], dtau[vi + 4], dtau[vi + 5]}};
        wsv(s.adj, NWJ, l, WJ_DF, spd_solve<T, DT>(wsi(s.root, 0, 0, WF_IA), t - df + y));
        continue;
      }
      const V3<T> sx = fld_v3(rec.t, W_S);
      const T r = dtau[vi] - dot(sx, df.w) - fld(rec.p, P_DAMP) * dqd[vi];
      const T wb = (T)((DT)(r + dot(sx, y.w)) * fld_wdi<T, DT>(rec.t));
      s.tp(l, W_u) = wb;
      if (par >= 0) {
        const V3<T> d = fld_v3(rec.t, W_D);
        const T x = dq[qi];
        const SV<T> pf = shift_force(f, d);
        const SV<T> pd = shift_force(df + x * SV<T>{cross(sx, f.w), cross(sx, f.v)}, d);
        const SV<T> py = shift_force(y - wb * fld_sv(rec.t, W_U), d);
        if (par == l - 1) {
          cf = pf;
          cd = pd;
          cy = py;
        } else {
          const bool first = meta_lastsib(m);
          if (first) ++sp;
          wsv(s.stk, WSW, sp - 1, 0, first ? pf : wsv(s.stk, WSW, sp - 1, 0) + pf);
          wsv(s.stk, WSW, sp - 1, 6, first ? pd : wsv(s.stk, WSW, sp - 1, 6) + pd);
          wsv(s.stk, WSW, sp - 1, 12, first ? py : wsv(s.stk, WSW, sp - 1, 12) + py);
        }
      }
    }
  }
  // the outward half and the integrator (root -> leaves)
  Records<T, STG, 1, RING_ADJ, 0, W_XY, 0, 0> rec(s, walk);
  SV<T> w_prev = zeroSV<T>();
  int sp = 0;
  for (int l = 0; l < walk; ++l) {
    rec.next();
    if (STG && l >= nl) continue;
    const int m = s.M(l);
    const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
    SV<T> w = zeroSV<T>();
    if (FR && meta_jtype(m) == J_FREE) {
      w = wsv(s.adj, NWJ, l, WJ_DF);
      const T x[6] = {w.w.x, w.w.y, w.w.z, w.v.x, w.v.y, w.v.z};
      Dual<T> nu[6], p[7];
      for (int i = 0; i < 6; ++i) {
        const Dual<T> v0(qd[vi + i], dqd[vi + i]);
        const Dual<T> v1 = v0 + Dual<T>(dt) * Dual<T>(s.root[(WF_QDD + i) * LANES], x[i]);
        qdo[vi + i] = v1.v;
        dqdo[vi + i] = v1.d;
        nu[i] = integ == I_SEMI_IMPLICIT ? v1 : v0;
      }
      for (int i = 0; i < 7; ++i) p[i] = Dual<T>(q[qi + i], dq[qi + i]);
      free_advance(p, nu, Dual<T>(dt));
      for (int i = 0; i < 7; ++i) {
        qo[qi + i] = p[i].v;
        dqo[qi + i] = p[i].d;
      }
    } else {
      if (par >= 0) {
        SV<T> wp = w_prev;
        if (par != l - 1) {
          wp = wsv(s.stk, WSW, sp - 1, 0);
          if (meta_lastsib(m)) --sp;
        }
        w = shift_motion(wp, fld_v3(rec.t, W_D));
      }
      const T x = fld(rec.t, W_u) - (T)((DT)dot(fld_sv(rec.t, W_U), w) * fld_wdi<T, DT>(rec.t));
      w.w += x * fld_v3(rec.t, W_S);
      const T v0 = qd[vi], v1 = v0 + dt * s.tp(l, W_QDD), d0 = dqd[vi], d1 = d0 + dt * x;
      qdo[vi] = v1;
      dqdo[vi] = d1;
      qo[qi] = q[qi] + dt * (integ == I_SEMI_IMPLICIT ? v1 : v0);
      dqo[qi] = dq[qi] + dt * (integ == I_SEMI_IMPLICIT ? d1 : d0);
    }
    if (meta_treechild(m)) {
      wsv(s.stk, WSW, sp, 0, w);
      ++sp;
    }
    w_prev = w;
  }
}

}  // namespace abasim
