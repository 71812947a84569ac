// The ABA step and its adjoint for trees of revolute joints, written in
// world-aligned link frames: link i's spatial quantities are expressed in a
// frame with the world's orientation whose origin is joint i.
//
// The Articulated Body Algorithm holds in any choice of link frames (Sec. 3.1
// takes Featherstone's recursions as given; they only need the transforms
// between neighbouring frames and each joint's motion subspace in its link's
// frame).  Here the transform from a parent's frame to its child's is a pure
// translation by d = R_p r (r: the joint origin in parent coordinates, R_p: the
// parent's orientation), X = (1, d), and the joint's motion subspace is
// S = [s; 0] with s the joint axis in world coordinates (the third column of the
// link's orientation R, since every revolute link turns about its own z axis).
// The price is a rotation of each body's inertia into world axes; the gain is
// that the inward recursion on the articulated inertias (the serial chain of the
// step, Fig. 1) shifts by d instead of rotating and shifting, and the rotation
// moves out of that chain into per-link work.  Same results as the link-frame
// step up to rounding.
//
// Forward step, per link l with parent p (p = -1: the world, R_p = 1):
//   E   = R(e_z, q)^T E_tree                 (parent -> link coordinates)
//   R   = R_p E^T,  d = R_p r_tree,  s = R e_z
//   v   = [v_p.w + s qd; v_p.v - d x v_p.w]  (root: [s qd; 0])
//   c   = v x [s qd; 0]
//   I^W = [R A_j R^T, skew(m R com); -skew(m R com), m 1]
//         with A_j = I_com + m (|com|^2 1 - com com^T) (inertia about the joint)
//   p^A = v x* (I^W v)
//   inward: I^A = I^W + sum_c shift(I^a_c, d_c), p^A += sum_c [p^a_c.w + d_c x p^a_c.v; p^a_c.v]
//           U = I^A S = [A s; B^T s], D = s.U_w, u = tau - b qd - s.p^A_w
//           I^a = I^A - U U^T / D,  p^a = p^A + I^a c + U u / D
//   outward: a' = [a_p.w; a_p.v - d x a_p.w] + c   (a_world = [0; -g])
//            qdd = (u - U.a') / D,  a = a' + [s qdd; 0]
// shift(I, d) = X^T I X with X = (1, d): the congruence by a pure translation.
//
// Adjoint step.  The joint accelerations solve M qdd = tau - b qd - C(q, qd), i.e.
// RNEA(q, qd, qdd) + b qd = tau, so with qddb the adjoint of qdd
//   lambda = M^-1 qddb,  taub = lambda,  (q, qd, m)b = -d(lambda . (RNEA + b qd)) at fixed qdd
// (the implicit-function form of Eq. 3-4).  lambda comes from the U and 1/D the
// step already holds (the bias-force and acceleration passes of a body at rest),
// and lambda . RNEA = sum_l w_l . (I_l a_l + v_l x* I_l v_l) with w the link
// velocities that the joint rates lambda would give: its derivative needs three
// motion-vector adjoints per link (of v, a and w) and no 6x6 adjoint at all, where
// differentiating the articulated-inertia recursion itself carries a 21-word
// adjoint of I^A through the tree (468 against 1666 floating-point operations and 45
// against 90 tape words per link; rollout + adjoint of 4096 7-link chains over 128
// steps in FP32 1.85 -> 1.49 ms, of 1000 over 50 steps in FP64 17.3 -> 11.7 ms, of
// 16384 trees of 2-64 links over 24 steps 15.6 -> 12.5 ms).  With W = -w, L = sum_l W_l . F_l, F_l = I_l a_l + v_l x* (I_l v_l):
//   leaves -> root: wb = (qddb + s.y_w) / D,  y' = y - wb U shifted to the parent
//   root -> leaves: lambda = wb - (U.w') / D, w = w' + [s lambda; 0]
//   leaves -> root: dL/dv, dL/da, dL/dW of each link (its own terms at its COM plus
//     its children's, shifted), then its joint's terms.
// The joint angle: turning link l's subtree about s by dq changes L as turning the
// motions it receives from its parent the other way does, because L is built
// covariantly:  qb = -s . sum over m in {v, a, W} of (m_w x mb_w + m_v x mb_v),
// m the motion handed down by the parent at joint l.  No adjoint of R or d is formed.
//
// Tree data flow.  Links are numbered in depth-first preorder, so a link's first
// child is link l + 1 and its values pass to it in registers; the values a link
// with several children hands to its later children (outward passes), or collects
// from them (leaves -> root passes), live on a per-system stack whose depth is the
// nesting of branchings, not the link count: a branching link pushes, its later
// children read (or add to) the top, and its last child pops (mirrored in the
// passes that run leaves -> root).  No pass reads another link's tape words.
#pragma once

#include "aba_step.cuh"

namespace abasim {

// Per-link tape of the world-aligned step, [link][field][lane]: orientation R, whose
// first two columns give way, when the adjoint will read the tape, to the rotated
// COM inertia R I_com R^T (the third column is the joint axis s); velocity v; U;
// 1/D (hi/lo pair); u, then the adjoint's wb; the joint offset d; and for the adjoint
// a', qdd, the joint rate qd and the COM offset R com.
enum : int {
  W_R = 0, W_V = 9, W_U = 15, W_DI = 21, W_u = 23, W_D = 24, W_AP = 27, W_QDD = 33, W_QD = 34, W_RW = 35, NWT = 38
};
// Record of a free root (FR kernels; link 0 only), [field][lane]: its articulated
// inertia, qdd, and the quaternion and velocity the step started from.  Its link's
// tape words hold R whole, the rotated COM inertia in W_U and its acceleration in W_AP.
enum : int { WF_IA = 0, WF_QDD = 21, WF_Q = 27, WF_QD = 31, NWF = 37 };
// Per-link adjoint record, [link][field][lane]: W = -w and lambda.
enum : int { WA_W = 0, WA_L = 6, NWA = 7 };
// One entry of the stack of parent values, [entry][field][lane]: (R, v), a or W in
// the outward passes, (shift(I^a, d), p^a), y or the adjoints of (v, a, W) in the
// passes that run leaves -> root.
constexpr int WSW = 27;
// model constants a world-aligned kernel reads: fields [0, NPRM_W) of the
// link's record (E_tree, r_tree, the axis slot, mass, COM, I_com, damping)
constexpr int NPRM_W = P_DAMP + 1;

// View of one system for the world-aligned step (pointers at this system's lane).
template <class T> struct WSys {
  const T* prm;     // [maxL][pstride][LANES]
  const int* meta;  // [maxL][LANES] ints, mstride apart
  T* tape;          // [maxL][NWT][LANES]
  T* adj;           // [maxL][NWA][LANES]
  int nl;
  int mstride = 1;
  int pstride = NPRM;
  int pf = 0;  // prm, meta, tape and adj in global memory: prefetch this many links ahead (0: none)
  T* stk = nullptr;  // [entry][WSW][LANES]: the stack of parent values (see the tree data flow above)
  T* root = nullptr; // [NWF][LANES]: the free root's record (FR only)
  SD T P(int l, int f) const { return prm[(l * pstride + f) * LANES]; }
  SD int M(int l) const { return meta[l * LANES * mstride]; }
  SD T& tp(int l, int f) const { return tape[(l * NWT + f) * LANES]; }
  SD T& ad(int l, int f) const { return adj[(l * NWA + f) * LANES]; }
};

// Prefetch into L1 of the cache lines holding fields [f0, f0 + n) of link l of a
// [link][stride][LANES] global array (a warp's 32 lanes share each line).  The
// passes run one thread per system through its links in a fixed order and
// touch the same fields of every link, so they ask for link l +- pf's lines while
// link l computes (pf from sim_set_prefetch, 2 by default): with a global tape, a
// warp then waits for memory once per pass instead of once per link.
SD void pf_line(const void* p) {
#ifdef __CUDA_ARCH__
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
#endif
}
template <class T> SD void pf_fields(const T* base, int stride, int l, int f0, int n) {
  for (int i = 0; i < n; ++i) pf_line(base + (l * stride + f0 + i) * LANES);
}
template <class T> SD void pf_meta(const WSys<T>& s, int l) { pf_line(s.meta + l * LANES * s.mstride); }

template <class T> SD V3<T> wv3(T* base, int stride, int l, int f) {
  const T* p = base + (l * stride + f) * LANES;
  return {p[0], p[LANES], p[2 * LANES]};
}
template <class T> SD void wv3(T* base, int stride, int l, int f, V3<T> v) {
  T* p = base + (l * stride + f) * LANES;
  p[0] = v.x; p[LANES] = v.y; p[2 * LANES] = v.z;
}
template <class T> SD SV<T> wsv(T* base, int stride, int l, int f) {
  return {wv3(base, stride, l, f), wv3(base, stride, l, f + 3)};
}
template <class T> SD void wsv(T* base, int stride, int l, int f, SV<T> v) {
  wv3(base, stride, l, f, v.w);
  wv3(base, stride, l, f + 3, v.v);
}
template <class T> SD M3<T> wm3(T* base, int stride, int l, int f) {
  M3<T> m;
  const T* p = base + (l * stride + f) * LANES;
  for (int i = 0; i < 9; ++i) m.a[i] = p[i * LANES];
  return m;
}
template <class T> SD void wm3(T* base, int stride, int l, int f, const M3<T>& m) {
  T* p = base + (l * stride + f) * LANES;
  for (int i = 0; i < 9; ++i) p[i * LANES] = m.a[i];
}
template <class T> SD S3<T> ws3(T* base, int stride, int l, int f) {
  const T* p = base + (l * stride + f) * LANES;
  return {p[0], p[LANES], p[2 * LANES], p[3 * LANES], p[4 * LANES], p[5 * LANES]};
}
template <class T> SD void ws3(T* base, int stride, int l, int f, const S3<T>& v) {
  T* p = base + (l * stride + f) * LANES;
  p[0] = v.xx; p[LANES] = v.yy; p[2 * LANES] = v.zz; p[3 * LANES] = v.xy; p[4 * LANES] = v.xz; p[5 * LANES] = v.yz;
}
template <class T> SD SI<T> wsi(T* base, int stride, int l, int f) {
  return {ws3(base, stride, l, f), wm3(base, stride, l, f + 6), ws3(base, stride, l, f + 15)};
}
template <class T> SD void wsi(T* base, int stride, int l, int f, const SI<T>& v) {
  ws3(base, stride, l, f, v.A);
  wm3(base, stride, l, f + 6, v.B);
  ws3(base, stride, l, f + 15, v.C);
}

// field helpers of a link: model constants, the joint axis, the rotated COM inertia in
// the first two columns of the tape's R, and 1/D
template <class T> SD V3<T> wprm_v3(const WSys<T>& s, int l, int f) { return {s.P(l, f), s.P(l, f + 1), s.P(l, f + 2)}; }
template <class T> SD M3<T> wprm_m3(const WSys<T>& s, int l, int f) {
  M3<T> m;
  for (int i = 0; i < 9; ++i) m.a[i] = s.P(l, f + i);
  return m;
}
template <class T> SD S3<T> wprm_s3(const WSys<T>& s, int l, int f) {
  return {s.P(l, f), s.P(l, f + 1), s.P(l, f + 2), s.P(l, f + 3), s.P(l, f + 4), s.P(l, f + 5)};
}
template <class T> SD V3<T> wcol2(const T* tp, int l) {
  const T* p = tp + (l * NWT + W_R) * LANES;
  return {p[2 * LANES], p[5 * LANES], p[8 * LANES]};
}
template <class T> SD void pf_col2(const T* tp, int stride, int l) {
  for (int i = 2; i < 9; i += 3) pf_line(tp + (l * stride + W_R + i) * LANES);
}
template <class T> SD void put_inertia(const WSys<T>& s, int l, const S3<T>& v) {
  s.tp(l, W_R) = v.xx; s.tp(l, W_R + 1) = v.yy; s.tp(l, W_R + 3) = v.zz;
  s.tp(l, W_R + 4) = v.xy; s.tp(l, W_R + 6) = v.xz; s.tp(l, W_R + 7) = v.yz;
}
template <class T> SD S3<T> get_inertia(const WSys<T>& s, int l) {
  return {s.tp(l, W_R), s.tp(l, W_R + 1), s.tp(l, W_R + 3), s.tp(l, W_R + 4), s.tp(l, W_R + 6), s.tp(l, W_R + 7)};
}
template <class T, class DT> SD void put_wdi(const WSys<T>& s, int l, DT di) {
  const T hi = (T)di;
  s.tp(l, W_DI) = hi;
  s.tp(l, W_DI + 1) = (T)(di - (DT)hi);
}
template <class T, class DT> SD DT get_wdi(const WSys<T>& s, int l) {
  return (DT)s.tp(l, W_DI) + (DT)s.tp(l, W_DI + 1);
}

// ------------------------------------------------------------------ operators
// third column of a rotation (the joint axis of a link turning about its z axis)
template <class T> SD V3<T> col2(const M3<T>& R) { return {R.a[2], R.a[5], R.a[8]}; }
// R S R^T for symmetric S
template <class T> SD S3<T> rot_sym(const M3<T>& R, const S3<T>& S) {
  const M3<T> F = full(S);
  M3<T> RS;  // R S
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      RS.a[3 * i + j] = R.a[3 * i] * F.a[j] + R.a[3 * i + 1] * F.a[3 + j] + R.a[3 * i + 2] * F.a[6 + j];
  auto e = [&](int i, int j) {
    return RS.a[3 * i] * R.a[3 * j] + RS.a[3 * i + 1] * R.a[3 * j + 1] + RS.a[3 * i + 2] * R.a[3 * j + 2];
  };
  return S3<T>{e(0, 0), e(1, 1), e(2, 2), e(0, 1), e(0, 2), e(1, 2)};
}
// rows of M crossed with d: M skew(d)
template <class T> SD M3<T> mskew(const M3<T>& M, V3<T> d) {
  M3<T> o;
  for (int i = 0; i < 3; ++i) {
    const V3<T> r = cross(V3<T>{M.a[3 * i], M.a[3 * i + 1], M.a[3 * i + 2]}, d);
    o.a[3 * i] = r.x; o.a[3 * i + 1] = r.y; o.a[3 * i + 2] = r.z;
  }
  return o;
}
// skew(d) M: columns of M crossed by d
template <class T> SD M3<T> skewm(V3<T> d, const M3<T>& M) {
  M3<T> o;
  for (int j = 0; j < 3; ++j) {
    const V3<T> c = cross(d, V3<T>{M.a[j], M.a[3 + j], M.a[6 + j]});
    o.a[j] = c.x; o.a[3 + j] = c.y; o.a[6 + j] = c.z;
  }
  return o;
}
// shift(I, d) = X^T I X, X = (1, d): Y_A = A - B K - (B K)^T - K C K, Y_B = B + K C,
// Y_C = C with K = skew(d)
template <class T> SD SI<T> shift(const SI<T>& I, V3<T> d) {
  const M3<T> BK = mskew(I.B, d);
  const M3<T> KC = skewm(d, full(I.C));
  const M3<T> KCK = mskew(KC, d);
  S3<T> A;
  A.xx = I.A.xx - T(2) * BK.a[0] - KCK.a[0];
  A.yy = I.A.yy - T(2) * BK.a[4] - KCK.a[4];
  A.zz = I.A.zz - T(2) * BK.a[8] - KCK.a[8];
  A.xy = I.A.xy - BK.a[1] - BK.a[3] - KCK.a[1];
  A.xz = I.A.xz - BK.a[2] - BK.a[6] - KCK.a[2];
  A.yz = I.A.yz - BK.a[5] - BK.a[7] - KCK.a[5];
  return SI<T>{A, I.B + KC, I.C};
}
// X^T f for X = (1, d): a force at the child's origin seen at the parent's
template <class T> SD SV<T> shift_force(SV<T> f, V3<T> d) { return {f.w + cross(d, f.v), f.v}; }
// X m for X = (1, d): the parent's motion seen at the child's origin
template <class T> SD SV<T> shift_motion(SV<T> m, V3<T> d) { return {m.w, m.v - cross(d, m.w)}; }

// ------------------------------------------------------------------ forward
// a body's own terms: inertia about its joint in world axes and bias force, from its
// COM inertia Ic and COM offset rw in world axes.  With vc the COM velocity the
// momentum about the COM is (Ic w, m vc), and v x* h = [w x Ic w; w x m vc] there.
template <class T> SD void body_terms(T m, V3<T> rw, const S3<T>& Ic, SV<T> v, SI<T>& IA, SV<T>& pA) {
  const V3<T> g = m * rw;
  const T cc = dot(rw, g);
  IA.A = S3<T>{Ic.xx + (cc - rw.x * g.x), Ic.yy + (cc - rw.y * g.y), Ic.zz + (cc - rw.z * g.z),
               Ic.xy - rw.x * g.y, Ic.xz - rw.x * g.z, Ic.yz - rw.y * g.z};
  IA.B = skew(g);
  IA.C = S3<T>{m, m, m, T(0), T(0), T(0)};
  const V3<T> vc = v.v + cross(v.w, rw);
  const V3<T> f = m * cross(v.w, vc);
  pA = SV<T>{cross(v.w, mul(Ic, v.w)) + cross(rw, f), f};
}

// One step for the state (q, qd) and joint force tau.  ADJ: also store what the
// adjoint reads.  INTEG: integrate into (qo, qdo) in the acceleration pass (they may
// alias q, qd: a link's own coordinates are read before they are written, and no
// pass after it reads the state).  FR: link 0 may be a free joint (R = E_tree^T R(quat),
// S = R on both halves, so D = I^A in world axes: one Cholesky solve).
template <class T, class DT, bool ADJ, bool INTEG, bool FR = false>
SD void wstep_forward(const WSys<T>& s, Col<const T> q, Col<const T> qd, Col<const T> tau, V3<T> grav, T dt,
                      int integ, Col<T> qo, Col<T> qdo) {
  T* tp = s.tape;
  const int nl = s.nl;
  // outward: orientation, joint offset, velocity (a root takes R_p = 1, v_p = 0,
  // which gives its values exactly)
  {
    M3<T> R_prev = eye3<T>();
    SV<T> v_prev = zeroSV<T>();
    int sp = 0;  // entries on the stack
    for (int l = 0; l < nl; ++l) {
      if (s.pf > 0 && l + s.pf < nl) {
        pf_meta(s, l + s.pf);
        pf_fields(s.prm, s.pstride, l + s.pf, P_E, 12);
      }
      const int m = s.M(l);
      const int par = meta_parent(m);
      if (FR && meta_jtype(m) == J_FREE) {
        const int qo = meta_qoff(m), vo = meta_voff(m);
        const T qt[4] = {q[qo + 3], q[qo + 4], q[qo + 5], q[qo + 6]};
        T w[6];
        for (int i = 0; i < 6; ++i) w[i] = qd[vo + i];
        R_prev = mTm(wprm_m3(s, l, P_E), quat_R(qt[0], qt[1], qt[2], qt[3]));
        v_prev = SV<T>{mul(R_prev, V3<T>{w[0], w[1], w[2]}), mul(R_prev, V3<T>{w[3], w[4], w[5]})};
        wm3(tp, NWT, l, W_R, R_prev);
        wsv(tp, NWT, l, W_V, v_prev);
        if (ADJ) {
          for (int i = 0; i < 4; ++i) s.root[(WF_Q + i) * LANES] = qt[i];
          for (int i = 0; i < 6; ++i) s.root[(WF_QD + i) * LANES] = w[i];
        }
        if (meta_treechild(m)) {
          wm3(s.stk, WSW, sp, 0, R_prev);
          wsv(s.stk, WSW, sp, 9, v_prev);
          ++sp;
        }
        continue;
      }
      T sn, cs;
      sincos_t(q[meta_qoff(m)], &sn, &cs);
      const T vl = qd[meta_voff(m)];
      const M3<T> E = rotz_T_mm(sn, cs, wprm_m3(s, l, P_E));
      M3<T> Rp = R_prev;
      SV<T> vp = v_prev;
      if (par < 0) {
        Rp = eye3<T>();
        vp = zeroSV<T>();
      } else if (par != l - 1) {
        Rp = wm3(s.stk, WSW, sp - 1, 0);
        vp = wsv(s.stk, WSW, sp - 1, 9);
        if (meta_lastsib(m)) --sp;
      }
      const V3<T> d = mul(Rp, wprm_v3(s, l, P_R));
      const M3<T> R = mmT(Rp, E);
      SV<T> v = shift_motion(vp, d);
      v.w += vl * col2(R);
      wv3(tp, NWT, l, W_D, d);
      wm3(tp, NWT, l, W_R, R);
      wsv(tp, NWT, l, W_V, v);
      if (ADJ) s.tp(l, W_QD) = vl;
      if (meta_treechild(m)) {
        wm3(s.stk, WSW, sp, 0, R);
        wsv(s.stk, WSW, sp, 9, v);
        ++sp;
      }
      R_prev = R;
      v_prev = v;
    }
  }
  // inward: articulated inertias and bias forces, from each link's own terms and its
  // children's contributions
  {
    SI<T> cI = zeroSI<T>();  // link l + 1's contribution when l is its parent
    SV<T> cp = zeroSV<T>();
    bool carry = false;
    int sp = 0;
    for (int l = nl - 1; l >= 0; --l) {
      if (s.pf > 0 && l - s.pf >= 0) {
        pf_fields(tp, NWT, l - s.pf, W_R, 15);
        pf_fields(tp, NWT, l - s.pf, W_D, 3);
        pf_fields(s.prm, s.pstride, l - s.pf, P_M, NPRM_W - P_M);
      }
      const int m = s.M(l);
      const int par = meta_parent(m), vo = meta_voff(m);
      const M3<T> R = wm3(tp, NWT, l, W_R);
      const SV<T> v = wsv(tp, NWT, l, W_V);
      const bool fr = FR && meta_jtype(m) == J_FREE;
      const V3<T> sx = col2(R);
      const T vl = qd[vo];
      const T tl = tau[vo] - s.P(l, P_DAMP) * vl;
      const V3<T> sq = vl * sx;
      const SV<T> c{cross(v.w, sq), cross(v.v, sq)};
      const S3<T> Ic = rot_sym(R, wprm_s3(s, l, P_IC));
      const V3<T> rw = mul(R, wprm_v3(s, l, P_C));
      SI<T> IA;
      SV<T> pA;
      body_terms(s.P(l, P_M), rw, Ic, v, IA, pA);
      if (ADJ) {
        if (fr)
          ws3(tp, NWT, l, W_U, Ic);
        else
          put_inertia(s, l, Ic);
        wv3(tp, NWT, l, W_RW, rw);
      }
      if (carry) {
        IA += cI;
        pA += cp;
      }
      if (meta_treechild(m)) {
        --sp;
        IA += wsi(s.stk, WSW, sp, 0);
        pA += wsv(s.stk, WSW, sp, 21);
      }
      if (fr) {  // D = I^A, u = R tau - p^A
        const SV<T> f{mul(R, V3<T>{tau[vo], tau[vo + 1], tau[vo + 2]}),
                      mul(R, V3<T>{tau[vo + 3], tau[vo + 4], tau[vo + 5]})};
        if (ADJ) wsi(s.root, 0, 0, WF_IA, IA);
        wsv(tp, NWT, l, W_AP, spd_solve<T, DT>(IA, f - pA));
        continue;
      }
      const SV<T> U{mul(IA.A, sx), mulT(IA.B, sx)};
      const DT Di = DT(1) / (DT)dot(sx, U.w);
      const T u = tl - dot(sx, pA.w);
      wsv(tp, NWT, l, W_U, U);
      put_wdi<T, DT>(s, l, Di);
      s.tp(l, W_u) = u;
      // the contribution to the parent (computed for a root too, with d = 0, and dropped)
      V3<T> d = wv3(tp, NWT, l, W_D);
      if (par < 0) d = zero3<T>();
      const SI<T> Ia = minus_scaled_outer<T, DT>(IA, Di, U);
      const SV<T> pa = pA + mul(Ia, c) + (T)((DT)u * Di) * U;
      const SI<T> Y = shift(Ia, d);
      const SV<T> pn = shift_force(pa, d);
      carry = par == l - 1 && par >= 0;
      if (carry) {
        cI = Y;
        cp = pn;
      } else if (par >= 0 && meta_lastsib(m)) {
        wsi(s.stk, WSW, sp, 0, Y);
        wsv(s.stk, WSW, sp, 21, pn);
        ++sp;
      } else if (par >= 0) {
        wsi(s.stk, WSW, sp - 1, 0, wsi(s.stk, WSW, sp - 1, 0) + Y);
        wsv(s.stk, WSW, sp - 1, 21, wsv(s.stk, WSW, sp - 1, 21) + pn);
      }
    }
  }
  // outward: accelerations (and the integrator)
  const SV<T> a0{zero3<T>(), -grav};
  SV<T> a_prev = a0;
  int sp = 0;
  for (int l = 0; l < nl; ++l) {
    if (s.pf > 0 && l + s.pf < nl) {
      pf_fields(tp, NWT, l + s.pf, W_R, W_AP - W_R);
    }
    const int m = s.M(l);
    const int par = meta_parent(m), vi = meta_voff(m);
    if (FR && meta_jtype(m) == J_FREE) {
      const M3<T> R = wm3(tp, NWT, l, W_R);
      const SV<T> a = wsv(tp, NWT, l, W_AP), b = a - a0;
      const V3<T> bw = mulT(R, b.w), bv = mulT(R, b.v);
      const T qdd[6] = {bw.x, bw.y, bw.z, bv.x, bv.y, bv.z};
      if (ADJ)
        for (int i = 0; i < 6; ++i) s.root[(WF_QDD + i) * LANES] = qdd[i];
      if (meta_treechild(m)) {
        wsv(s.stk, WSW, sp, 0, a);
        ++sp;
      }
      if (INTEG) {
        const int qi = meta_qoff(m);
        T nu[6], x[7];
        for (int i = 0; i < 6; ++i) {
          const T v0 = qd[vi + i];
          const T v1 = v0 + dt * qdd[i];
          qdo[vi + i] = v1;
          nu[i] = integ == I_SEMI_IMPLICIT ? v1 : v0;
        }
        for (int i = 0; i < 7; ++i) x[i] = q[qi + i];
        free_advance(x, nu, dt);
        for (int i = 0; i < 7; ++i) qo[qi + i] = x[i];
      }
      a_prev = a;
      continue;
    }
    const V3<T> sx = col2(wm3(tp, NWT, l, W_R));
    const SV<T> v = wsv(tp, NWT, l, W_V);
    const SV<T> U = wsv(tp, NWT, l, W_U);
    const DT Di = get_wdi<T, DT>(s, l);
    const T u = s.tp(l, W_u);
    const T v0 = qd[vi];
    const V3<T> sq = v0 * sx;
    SV<T> ap = a0;
    if (par >= 0) {
      SV<T> apar = a_prev;
      if (par != l - 1) {
        apar = wsv(s.stk, WSW, sp - 1, 0);
        if (meta_lastsib(m)) --sp;
      }
      ap = shift_motion(apar, wv3(tp, NWT, l, W_D));
    }
    ap += SV<T>{cross(v.w, sq), cross(v.v, sq)};
    const T qdd = (T)(((DT)u - (DT)dot(U, ap)) * Di);
    const SV<T> a{ap.w + qdd * sx, ap.v};
    if (ADJ) {
      wsv(tp, NWT, l, W_AP, ap);
      s.tp(l, W_QDD) = qdd;
    }
    if (meta_treechild(m)) {
      wsv(s.stk, WSW, sp, 0, a);
      ++sp;
    }
    if (INTEG) {
      const int qi = meta_qoff(m);
      const T v1 = v0 + dt * qdd;
      const T q1 = q[qi] + dt * (integ == I_SEMI_IMPLICIT ? v1 : v0);
      qdo[vi] = v1;
      qo[qi] = q1;
    }
    a_prev = a;
  }
}

// ------------------------------------------------------------------ adjoint
// the gradients of L_l = W . (I a + v x* (I v)) for one body: dL/dW (the body force F),
// dL/da = I W, dL/dv = -(W x* I v) - I (v x W), and dL/dm.  Formed at the COM, where I
// is block diagonal and the linear part of dL/dv is m W_c x w, then moved to the joint.
template <class T> struct BodyGrad {
  SV<T> F, ab, vb;
  T mb;
};
template <class T> SD BodyGrad<T> body_grad(T m, V3<T> rw, const S3<T>& Ic, SV<T> v, SV<T> a, SV<T> W) {
  const V3<T> vc = v.v + cross(v.w, rw), Wc = W.v + cross(W.w, rw);
  const V3<T> Ac = a.v + cross(a.w, rw) + cross(v.w, vc);  // the COM's acceleration
  const V3<T> Lw = mul(Ic, v.w);
  BodyGrad<T> g;
  const V3<T> f = m * Ac;
  g.F = SV<T>{mul(Ic, a.w) + cross(v.w, Lw) + cross(rw, f), f};
  const V3<T> k = m * Wc;
  g.ab = SV<T>{mul(Ic, W.w) + cross(rw, k), k};
  const V3<T> zv = cross(k, v.w);
  g.vb = SV<T>{cross(rw, zv) - cross(W.w, Lw) - cross(k, vc) - mul(Ic, cross(v.w, W.w)), zv};
  g.mb = dot(Wc, Ac);
  return g;
}

// Requires wstep_forward<ADJ = true>(q, qd, tau) to have filled the tape.  On entry
// (gq, gqd) hold the adjoint of x^{k+1}; on exit that of x^k.  Writes the adjoint
// of tau into gtau and adds dPhi/dm of every link into gm.  FR (link 0 may be a free
// joint) needs the gravity: the only motion a free root's orientation turns against.
template <class T, class DT, bool FR = false>
SD void wstep_adjoint(const WSys<T>& s, Col<T> gq, Col<T> gqd, Col<T> gtau, Col<T> gm, T dt, int integ,
                      V3<T> grav = zero3<T>()) {
  T* tp = s.tape;
  T* ad = s.adj;
  const int nl = s.nl;
  // the integrator's adjoint and the inward half of lambda = M^-1 qddb (leaves -> root)
  {
    SV<T> cy = zeroSV<T>();
    bool carry = false;
    int sp = 0;
    for (int l = nl - 1; l >= 0; --l) {
      if (s.pf > 0 && l - s.pf >= 0) {
        pf_col2(tp, NWT, l - s.pf);
        pf_fields(tp, NWT, l - s.pf, W_U, W_AP - W_U);
      }
      const int m = s.M(l);
      const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
      if (FR && meta_jtype(m) == J_FREE) {  // lambda_root = (I^A)^-1 (R qddb + y)
        T qt[4], nu[6], qddb6[6];
        for (int i = 0; i < 4; ++i) qt[i] = s.root[(WF_Q + i) * LANES];
        for (int i = 0; i < 6; ++i) {
          nu[i] = s.root[(WF_QD + i) * LANES];
          if (integ == I_SEMI_IMPLICIT) nu[i] += dt * s.root[(WF_QDD + i) * LANES];
        }
        free_integrator_adjoint(qt, nu, gq, gqd, qi, vi, dt, integ, qddb6);
        const M3<T> R = wm3(tp, NWT, l, W_R);
        SV<T> y{mul(R, V3<T>{qddb6[0], qddb6[1], qddb6[2]}), mul(R, V3<T>{qddb6[3], qddb6[4], qddb6[5]})};
        if (carry) y += cy;
        carry = false;
        if (meta_treechild(m)) {
          --sp;
          y += wsv(s.stk, WSW, sp, 0);
        }
        const SV<T> w = spd_solve<T, DT>(wsi(s.root, 0, 0, WF_IA), y);
        wsv(ad, NWA, l, WA_W, zeroSV<T>() - w);
        const V3<T> lw = mulT(R, w.w), lv = mulT(R, w.v);
        gtau[vi] = lw.x;
        gtau[vi + 1] = lw.y;
        gtau[vi + 2] = lw.z;
        gtau[vi + 3] = lv.x;
        gtau[vi + 4] = lv.y;
        gtau[vi + 5] = lv.z;
        continue;
      }
      T qddb;
      {
        const T qb = gq[qi], vb = gqd[vi];
        const T vt = vb + dt * qb;
        gqd[vi] = vt;
        qddb = dt * (integ == I_SEMI_IMPLICIT ? vt : vb);
      }
      SV<T> y = carry ? cy : zeroSV<T>();
      carry = false;
      if (meta_treechild(m)) {
        --sp;
        y += wsv(s.stk, WSW, sp, 0);
      }
      const V3<T> sx = wcol2(tp, l);
      const SV<T> U = wsv(tp, NWT, l, W_U);
      const T wb = (T)((DT)(qddb + dot(sx, y.w)) * get_wdi<T, DT>(s, l));
      s.tp(l, W_u) = wb;
      if (par >= 0) {
        const SV<T> yp = shift_force(y - wb * U, wv3(tp, NWT, l, W_D));
        if (par == l - 1) {
          cy = yp;
          carry = true;
        } else if (meta_lastsib(m)) {
          wsv(s.stk, WSW, sp, 0, yp);
          ++sp;
        } else {
          wsv(s.stk, WSW, sp - 1, 0, wsv(s.stk, WSW, sp - 1, 0) + yp);
        }
      }
    }
  }
  // the outward half: lambda, W = -w (root -> leaves)
  {
    SV<T> W_prev = zeroSV<T>();
    int sp = 0;
    for (int l = 0; l < nl; ++l) {
      if (s.pf > 0 && l + s.pf < nl) {
        pf_col2(tp, NWT, l + s.pf);
        pf_fields(tp, NWT, l + s.pf, W_U, W_AP - W_U);
        pf_line(s.prm + ((l + s.pf) * s.pstride + P_DAMP) * LANES);
      }
      const int m = s.M(l);
      const int par = meta_parent(m), vi = meta_voff(m);
      if (FR && meta_jtype(m) == J_FREE) {
        W_prev = wsv(ad, NWA, l, WA_W);
        if (meta_treechild(m)) {
          wsv(s.stk, WSW, sp, 0, W_prev);
          ++sp;
        }
        continue;
      }
      SV<T> W = zeroSV<T>();
      if (par >= 0) {
        SV<T> Wp = W_prev;
        if (par != l - 1) {
          Wp = wsv(s.stk, WSW, sp - 1, 0);
          if (meta_lastsib(m)) --sp;
        }
        W = shift_motion(Wp, wv3(tp, NWT, l, W_D));
      }
      const SV<T> U = wsv(tp, NWT, l, W_U);
      const T lam = s.tp(l, W_u) + (T)((DT)dot(U, W) * get_wdi<T, DT>(s, l));
      W.w = W.w - lam * wcol2(tp, l);
      s.ad(l, WA_L) = lam;
      wsv(ad, NWA, l, WA_W, W);
      gtau[vi] = lam;
      gqd[vi] -= s.P(l, P_DAMP) * lam;
      if (meta_treechild(m)) {
        wsv(s.stk, WSW, sp, 0, W);
        ++sp;
      }
      W_prev = W;
    }
  }
  // the derivative of L (leaves -> root)
  {
    SV<T> cv = zeroSV<T>(), ca = zeroSV<T>(), cw = zeroSV<T>();
    bool carry = false;
    int sp = 0;
    for (int l = nl - 1; l >= 0; --l) {
      if (s.pf > 0 && l - s.pf >= 0) {
        pf_fields(tp, NWT, l - s.pf, W_R, 15);
        pf_fields(tp, NWT, l - s.pf, W_D, NWT - W_D);
        pf_fields(ad, NWA, l - s.pf, 0, NWA);
        pf_line(s.prm + ((l - s.pf) * s.pstride + P_M) * LANES);
      }
      const int m = s.M(l);
      const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
      const bool fr = FR && meta_jtype(m) == J_FREE;
      const V3<T> sx = wcol2(tp, l);
      const SV<T> v = wsv(tp, NWT, l, W_V), ap = wsv(tp, NWT, l, W_AP), W = wsv(ad, NWA, l, WA_W);
      const T vl = fr ? T(0) : s.tp(l, W_QD);
      const T qdd = fr ? T(0) : s.tp(l, W_QDD);
      const SV<T> a{ap.w + qdd * sx, ap.v};
      const S3<T> Ic = fr ? ws3(tp, NWT, l, W_U) : get_inertia(s, l);
      BodyGrad<T> g = body_grad(s.P(l, P_M), wv3(tp, NWT, l, W_RW), Ic, v, a, W);
      gm[l] += g.mb;
      if (carry) {
        g.vb += cv;
        g.ab += ca;
        g.F += cw;
      }
      carry = false;
      if (meta_treechild(m)) {
        --sp;
        g.vb += wsv(s.stk, WSW, sp, 0);
        g.ab += wsv(s.stk, WSW, sp, 6);
        g.F += wsv(s.stk, WSW, sp, 12);
      }
      if (fr) {  // v = R qd, a = R qdd + [0; -g]: only the gravity does not turn with R
        const M3<T> R = wm3(tp, NWT, l, W_R);
        const V3<T> bw = mulT(R, g.vb.w), bv = mulT(R, g.vb.v);
        const T vv[6] = {bw.x, bw.y, bw.z, bv.x, bv.y, bv.z};
        for (int i = 0; i < 6; ++i) gqd[vi + i] += vv[i];
        const M3<T> EJb = mmT(outer(mulT(R, g.ab.v), zero3<T>() - grav), wprm_m3(s, l, P_E));  // E = E_J E_t
        T qb[4] = {T(0), T(0), T(0), T(0)};
        quat_R_adj(s.root[WF_Q * LANES], s.root[(WF_Q + 1) * LANES], s.root[(WF_Q + 2) * LANES],
                   s.root[(WF_Q + 3) * LANES], transpose(EJb), qb);
        for (int i = 0; i < 4; ++i) gq[qi + 3 + i] += qb[i];
        continue;
      }
      // c = v x [s qd; 0] = -qd e with e = [s x v_w; s x v_v]; b = [s x ab_w; s x ab_v]
      const SV<T> e{cross(sx, v.w), cross(sx, v.v)}, b{cross(sx, g.ab.w), cross(sx, g.ab.v)};
      g.vb += vl * b;
      gqd[vi] += dot(sx, g.vb.w) - dot(g.ab, e);
      // the motions handed down by the parent, turned against the subtree (a' less c; the
      // joint's own parts along s drop out)
      gq[qi] += dot(ap + vl * e, b) - dot(e, g.vb) - dot(sx, cross(W.w, g.F.w) + cross(W.v, g.F.v));
      if (par >= 0) {
        const V3<T> d = wv3(tp, NWT, l, W_D);
        cv = shift_force(g.vb, d);
        ca = shift_force(g.ab, d);
        cw = shift_force(g.F, d);
        if (par == l - 1) {
          carry = true;
        } else if (meta_lastsib(m)) {
          wsv(s.stk, WSW, sp, 0, cv);
          wsv(s.stk, WSW, sp, 6, ca);
          wsv(s.stk, WSW, sp, 12, cw);
          ++sp;
        } else {
          wsv(s.stk, WSW, sp - 1, 0, wsv(s.stk, WSW, sp - 1, 0) + cv);
          wsv(s.stk, WSW, sp - 1, 6, wsv(s.stk, WSW, sp - 1, 6) + ca);
          wsv(s.stk, WSW, sp - 1, 12, wsv(s.stk, WSW, sp - 1, 12) + cw);
        }
      }
    }
  }
}

}  // namespace abasim
