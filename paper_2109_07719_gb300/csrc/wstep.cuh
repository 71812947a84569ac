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
// A tree with a free root (FR) is written in the axes of its base instead of the world's:
// R = 1 and v = qd at the root, and only the gravity turns, E g with E = R(quat)^T E_tree.
// The axes need not be the world's, only the same for the whole tree; in the base's own, the
// base's orientation rounds nothing else, and a quaternion that is not of unit length acts as
// in the link-frame step, through the gravity and the position alone.  (In world axes an
// FP32 step's own part of the new state had 3 times the link-frame step's error, of the
// gradient in q 6 times; in the base's axes 2 and 0.9, over random bases of 13 and 23 links.
// A quaternion rounded to float was 1e-7 off in FP64, now 1e-16.)
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

// Per-link tape of the world-aligned step, [link][field][lane]: U; 1/D (hi/lo pair); u,
// then the adjoint's wb; the joint offset d; the orientation R by columns, the joint axis
// s = R e_z first, the other two giving way, when the adjoint will read the tape, to the
// rotated COM inertia R I_com R^T; velocity v; and for the adjoint a', qdd, the joint rate
// qd and the COM offset R com.  Ordered so that what a pass reads is one range (two for
// the acceleration pass).
enum : int {
  W_U = 0, W_DI = 6, W_u = 8, W_D = 9, W_S = 12, W_XY = 15, W_V = 21, W_AP = 27, W_QDD = 33, W_QD = 34, W_RW = 35,
  NWT = 38,
  W_E = 0  // a free root's E, in the words of U, 1/D and u, which it does not have
};
// Record of a free root (FR kernels; link 0 only), [field][lane]: its articulated
// inertia, qdd (its linear part then gives way to that of qddb), the quaternion and velocity
// the step started from and its COM inertia.  Its link's tape words hold E, R = 1 whole and
// its acceleration in W_AP.
enum : int { WF_IA = 0, WF_QDD = 21, WF_QDDB = WF_QDD + 3, WF_Q = 27, WF_QD = 31, WF_IC = 37, NWF = 43 };
// Per-link adjoint record, [link][field][lane]: W = -w.
enum : int { WA_W = 0, NWA = 6 };
// One entry of the stack of parent values, [entry][field][lane]: (R, v), a or W in
// the outward passes, (shift(I^a, d), p^a), y or the adjoints of (v, a, W) in the
// passes that run leaves -> root.
constexpr int WSW = 27;
// model constants a world-aligned kernel reads: fields [0, NPRM_W) of the
// link's record (E_tree, r_tree, the axis slot, mass, COM, I_com, damping)
constexpr int NPRM_W = P_DAMP + 1;

// View of one system for the world-aligned step (pointers at this system's lane).
// STG: the records are in global memory and each pass stages them through `ring`.
template <class T, bool STG = false> struct WSys {
  const T* prm;     // [maxL][pstride][LANES]
  const int* meta;  // [maxL][LANES] ints, mstride apart
  T* tape;          // [maxL][NWT][LANES]
  T* adj;           // [maxL][NWA][LANES]
  int nl;
  int mstride = 1;
  int pstride = NPRM;
  T* stk = nullptr;  // [entry][WSW][LANES]: the stack of parent values (see the tree data flow above)
  T* root = nullptr; // [NWF][LANES]: the free root's record (FR only)
  int links = -1;    // STG: links the warp walks (its longest system's; every lane walks them together)
  T* ring = nullptr; // STG: this warp's ring in shared memory, [rows][LANES], at lane 0
  bool full = true;  // STG: it has three slots of the longest pass, not one
  int lane = 0;
  SD T P(int l, int f) const { return prm[(l * pstride + f) * LANES]; }
  SD int M(int l) const { return meta[l * LANES * mstride]; }
  SD T& tp(int l, int f) const { return tape[(l * NWT + f) * LANES]; }
  SD T& ad(int l, int f) const { return adj[(l * NWA + f) * LANES]; }
  SD int walk() const { return STG ? links : nl; }
};

// Staged records.  A pass walks its links in a fixed order and reads the same fields of
// each, so with the records in global memory the warp copies the next links' rows (32
// systems' words of one field, 128 or 256 bytes) into a shared-memory ring with 16-byte
// cp.async a few links ahead, and the pass reads shared memory.  Prefetching the same
// lines into L1 left the passes waiting for L2 (27 % L1 hits: the tape's lines have been
// written since); with the ring a 64-link chain tile's rollout step went from 123 to 86 us,
// 1500 trees of 2-40 links with segment replay from 17.3 to 12.6 ms over 48 steps.  It
// takes 3 x rows x 128 bytes a warp and a quarter of the instructions (four rows each).
// A pass that reads fewer rows has more slots in the same ring, so a short pass looks as
// far ahead in time as a long one.  The slot filled while link i computes was read at link
// i - 2, so one warp barrier a link orders both the reads and the writes.
// rows of a warp's ring: three slots of its longest pass (the forward passes', the adjoint
// passes', a rollout's with its fused pass); a ring of one slot (staging without looking ahead) is a third of it
constexpr int RING_FWD = 29, RING_ADJ = 36, RING_ROLL = 33;
// producers of the pipelined adjoint at most, each with a tape; in global memory, one stack
// of parent values for each of its warps is beside them
constexpr int WPIPE_TAPES = 3;

#ifdef __CUDACC__
__device__ __forceinline__ void stage_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int NEWER> __device__ __forceinline__ void stage_wait() {  // all but the NEWER newest groups are in place
  asm volatile("cp.async.wait_group %0;\n" ::"n"(NEWER) : "memory");
}
#endif

// The records of one pass over `n` links from link 0 up (DIR 1) or from link n - 1 down
// (DIR -1): tape fields [TF, TF + TN) and [SF, SF + SN), model constants [PF, PF + PN),
// adjoint fields [AF, AF + AN).  next() makes the following link's records readable through
// t (fields of the first range), t2 (the second), p and a, indexed by field, at this lane.
// All lanes of the warp call it together when staging.
template <class T, bool STG, int DIR, int RING, int TF, int TN, int PF, int PN, int AF = 0, int AN = 0, int SF = 0,
          int SN = 0, int ASTRIDE = NWA>
struct Records {
  static constexpr int ROWS = TN + SN + PN + AN, SLOTS = 3 * RING / ROWS, AHEAD = SLOTS - 2;
  static_assert(ROWS <= RING, "ring rows");
  const WSys<T, STG>& s;
  int left;              // links still to fetch (staging)
  const T *st, *sp, *sa;  // the next record to fetch, or the current one
  T *fill, *read;        // ring slots
  const T *t, *t2, *p, *a;
  SD Records(const WSys<T, STG>& sys, int n) : s(sys), left(n) {
    const int first = DIR > 0 ? 0 : n - 1;
    st = s.tape + first * NWT * LANES;
    sp = s.prm + first * s.pstride * LANES;
    sa = AN ? s.adj + first * ASTRIDE * LANES : nullptr;
    if constexpr (STG) {
#ifdef __CUDA_ARCH__
      constexpr int PER = 16 / sizeof(T);
      st += TF * LANES - s.lane + s.lane * PER;  // each lane copies 16 bytes of every LANES x 16
      sp += PF * LANES - s.lane + s.lane * PER;
      if (AN) sa += AF * LANES - s.lane + s.lane * PER;
      fill = read = s.ring;
      __syncwarp();  // the previous pass has read its last slot and written its records
      if (s.full)
        for (int j = 0; j < AHEAD; ++j) fetch();
#endif
    } else {
      st -= DIR * NWT * LANES;
      sp -= DIR * s.pstride * LANES;
      if (AN) sa -= DIR * ASTRIDE * LANES;
    }
  }
  SD void fetch() {
#ifdef __CUDA_ARCH__
    constexpr int CH = LANES * (int)sizeof(T) / 16;  // copies per row
    if (left > 0) {
      copy<TN * CH>(fill, st);
      copy<SN * CH>(fill + TN * LANES, st + (SF - TF) * LANES);
      copy<PN * CH>(fill + (TN + SN) * LANES, sp);
      if (AN) copy<AN * CH>(fill + (TN + SN + PN) * LANES, sa);
      st += DIR * NWT * LANES;
      sp += DIR * s.pstride * LANES;
      if (AN) sa += DIR * ASTRIDE * LANES;
      --left;
    }
    stage_commit();
    if (s.full) fill = fill == s.ring + (SLOTS - 1) * ROWS * LANES ? s.ring : fill + ROWS * LANES;
#endif
  }
  template <int COPIES> SD void copy(T* dst, const T* src) {
#ifdef __CUDA_ARCH__
    constexpr int PER = 16 / sizeof(T);
    dst += s.lane * PER;
#pragma unroll
    for (int c = 0; c < COPIES; c += LANES)
      if (c + LANES <= COPIES || c + s.lane < COPIES) stage_cp16(dst + c * PER, src + c * PER);
#endif
  }
  SD void next() {
    if constexpr (STG) {
#ifdef __CUDA_ARCH__
      if (!s.full) __syncwarp();  // every lane is done with the only slot
      fetch();
      if (s.full)
        stage_wait<AHEAD>();
      else
        stage_wait<0>();
      __syncwarp();
      const T* r = read + s.lane;
      t = r - TF * LANES;
      t2 = r + (TN - SF) * LANES;
      p = r + (TN + SN - PF) * LANES;
      a = r + (TN + SN + PN - AF) * LANES;
      if (s.full) read = read == s.ring + (SLOTS - 1) * ROWS * LANES ? s.ring : read + ROWS * LANES;
#endif
    } else {
      t = t2 = st += DIR * NWT * LANES;
      p = sp += DIR * s.pstride * LANES;
      if (AN) a = sa += DIR * ASTRIDE * LANES;
    }
  }
};

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

// fields of one record (a pointer at this lane, rows LANES apart)
template <class T> SD T fld(const T* r, int f) { return r[f * LANES]; }
template <class T> SD V3<T> fld_v3(const T* r, int f) { return {fld(r, f), fld(r, f + 1), fld(r, f + 2)}; }
template <class T> SD SV<T> fld_sv(const T* r, int f) { return {fld_v3(r, f), fld_v3(r, f + 3)}; }
template <class T> SD S3<T> fld_s3(const T* r, int f) {
  return {fld(r, f), fld(r, f + 1), fld(r, f + 2), fld(r, f + 3), fld(r, f + 4), fld(r, f + 5)};
}
template <class T> SD M3<T> fld_m3(const T* r, int f) {
  M3<T> m;
  for (int i = 0; i < 9; ++i) m.a[i] = fld(r, f + i);
  return m;
}
// the orientation, stored by columns with the joint axis (the third) first
template <class T> SD M3<T> fld_rot(const T* r) {
  const V3<T> s = fld_v3(r, W_S), x = fld_v3(r, W_XY), y = fld_v3(r, W_XY + 3);
  return M3<T>{{x.x, y.x, s.x, x.y, y.y, s.y, x.z, y.z, s.z}};
}
template <class T> SD void put_rot(T* r, const M3<T>& R) {
  for (int i = 0; i < 3; ++i) {
    r[(W_S + i) * LANES] = R.a[3 * i + 2];
    r[(W_XY + i) * LANES] = R.a[3 * i];
    r[(W_XY + 3 + i) * LANES] = R.a[3 * i + 1];
  }
}
template <class T, class DT> SD void put_wdi(T* r, DT di) {
  const T hi = (T)di;
  r[W_DI * LANES] = hi;
  r[(W_DI + 1) * LANES] = (T)(di - (DT)hi);
}
template <class T, class DT> SD DT fld_wdi(const T* r) { return (DT)fld(r, W_DI) + (DT)fld(r, W_DI + 1); }

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

// Per-link scalars of a pass from two coordinate columns (a at the link's position or
// velocity offset, b at its velocity offset), read one link ahead of their use and the
// meta words two ahead, so that no link waits for its own loads.
template <class T, bool STG, bool AQ> struct Inputs {
  const WSys<T, STG>& s;
  Col<const T> ca, cb;
  int l, dir, n, m1, m2;
  T a1, b1;
  int m;   // the link's meta word
  T a, b;  // its scalars
  SD Inputs(const WSys<T, STG>& sys, Col<const T> a_, Col<const T> b_, int first, int dir_, int n_)
      : s(sys), ca(a_), cb(b_), l(first), dir(dir_), n(n_) {
    m1 = m2 = 0;
    a1 = b1 = T(0);
    if (n > 0 && s.nl > 0) {
      m1 = s.M(first);
      m2 = n > 1 ? s.M(first + dir) : m1;
      a1 = ca[AQ ? meta_qoff(m1) : meta_voff(m1)];
      b1 = cb[meta_voff(m1)];
    }
  }
  SD void next() {  // the scalars of the following link
    m = m1;
    a = a1;
    b = b1;
    m1 = m2;
    if (!STG || s.nl > 0) {
      a1 = ca[AQ ? meta_qoff(m1) : meta_voff(m1)];
      b1 = cb[meta_voff(m1)];
    }
    const int l2 = l + 2 * dir;
    if (l2 >= 0 && l2 < n) m2 = s.M(l2);
    l += dir;
  }
};

// ------------------------------------------------------------------ forward
// adds a body's own terms to IA and pA: its inertia about its joint in world axes and its
// bias force, from its COM inertia Ic and COM offset rw in world axes.  With vc the COM
// velocity the momentum about the COM is (Ic w, m vc), and v x* h = [w x Ic w; w x m vc]
// there.  Only the entries a body's inertia has are added (an x + 0 would stay an addition).
template <class T> SD void add_body(T m, V3<T> rw, const S3<T>& Ic, SV<T> v, SI<T>& IA, SV<T>& pA) {
  const V3<T> g = m * rw;
  const T cc = dot(rw, g);
  IA.A += S3<T>{Ic.xx + (cc - rw.x * g.x), Ic.yy + (cc - rw.y * g.y), Ic.zz + (cc - rw.z * g.z),
                Ic.xy - rw.x * g.y, Ic.xz - rw.x * g.z, Ic.yz - rw.y * g.z};
  IA.B.a[1] -= g.z;
  IA.B.a[2] += g.y;
  IA.B.a[3] += g.z;
  IA.B.a[5] -= g.x;
  IA.B.a[6] -= g.y;
  IA.B.a[7] += g.x;
  IA.C.xx += m;
  IA.C.yy += m;
  IA.C.zz += m;
  const V3<T> vc = v.v + cross(v.w, rw);
  const V3<T> f = m * cross(v.w, vc);
  pA += SV<T>{cross(v.w, mul(Ic, v.w)) + cross(rw, f), f};
}

// A free root's rotation from the parent's axes to its own, from the quaternion as it is given.
template <class T> SD M3<T> free_rotation(const T* qt, const M3<T>& Et) {
  return mTm(quat_R(qt[0], qt[1], qt[2], qt[3]), Et);
}

// The passes of a step.  ADJ: also store what the adjoint reads.  FR: link 0 may be a free
// joint (its tree's axes: R = 1, S = 1 on both halves, D = I^A, one Cholesky solve).
template <class T, class DT, bool ADJ, bool FR, bool STG>
SD void wpass_pose(const WSys<T, STG>& s, Col<const T> q, Col<const T> qd) {
  T* tp = s.tape;
  const int nl = s.nl, walk = s.walk();
  // outward: orientation, joint offset, velocity (a root takes R_p = 1, v_p = 0,
  // which gives its values exactly)
  {
    Records<T, STG, 1, RING_FWD, 0, 0, P_E, 12> rec(s, walk);
    Inputs<T, STG, true> in(s, q, qd, 0, 1, walk);
    M3<T> R_prev = eye3<T>();
    SV<T> v_prev = zeroSV<T>();
    int sp = 0;  // entries on the stack
    for (int l = 0; l < walk; ++l) {
      rec.next();
      in.next();
      if (STG && l >= nl) continue;
      const int m = in.m;
      const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
      T* w = tp + l * NWT * LANES;
      M3<T> R;
      SV<T> v;
      if (FR && meta_jtype(m) == J_FREE) {
        const T qt[4] = {q[qi + 3], q[qi + 4], q[qi + 5], q[qi + 6]};
        T x[6];
        for (int i = 0; i < 6; ++i) x[i] = qd[vi + i];
        R = eye3<T>();
        v = SV<T>{{x[0], x[1], x[2]}, {x[3], x[4], x[5]}};
        wm3(w, 0, 0, W_E, free_rotation(qt, fld_m3(rec.p, P_E)));
        if (ADJ) {
          for (int i = 0; i < 4; ++i) s.root[(WF_Q + i) * LANES] = qt[i];
          for (int i = 0; i < 6; ++i) s.root[(WF_QD + i) * LANES] = x[i];
        }
      } else {
        T sn, cs;
        sincos_t(in.a, &sn, &cs);
        const T vl = in.b;
        const M3<T> E = rotz_T_mm(sn, cs, fld_m3(rec.p, P_E));
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
        const V3<T> d = mul(Rp, fld_v3(rec.p, P_R));
        R = mmT(Rp, E);
        v = shift_motion(vp, d);
        v.w += vl * col2(R);
        wv3(w, 0, 0, W_D, d);
        if (ADJ) w[W_QD * LANES] = vl;
      }
      put_rot(w, R);
      wsv(w, 0, 0, W_V, v);
      if (meta_treechild(m)) {
        wm3(s.stk, WSW, sp, 0, R);
        wsv(s.stk, WSW, sp, 9, v);
        ++sp;
      }
      R_prev = R;
      v_prev = v;
    }
  }
}

template <class T, class DT, bool ADJ, bool FR, bool STG>
SD void wpass_inward(const WSys<T, STG>& s, Col<const T> qd, Col<const T> tau) {
  T* tp = s.tape;
  const int nl = s.nl, walk = s.walk();
  // inward: articulated inertias and bias forces, from each link's own terms and its
  // children's contributions
  {
    Records<T, STG, -1, RING_FWD, W_D, W_AP - W_D, P_M, NPRM_W - P_M> rec(s, walk);
    Inputs<T, STG, false> in(s, tau, qd, walk - 1, -1, walk);
    SI<T> cI = zeroSI<T>();  // link l + 1's contribution if l is its parent, else 0
    SV<T> cp = zeroSV<T>();
    int sp = 0;
    for (int l = walk - 1; l >= 0; --l) {
      rec.next();
      in.next();
      if (STG && l >= nl) continue;
      const int m = in.m;
      const int par = meta_parent(m), vo = meta_voff(m);
      T* w = tp + l * NWT * LANES;
      const bool fr = FR && meta_jtype(m) == J_FREE;
      const M3<T> R = fld_rot(rec.t);
      const SV<T> v = fld_sv(rec.t, W_V);
      const V3<T> sx = col2(R);
      const T vl = in.b;
      const T tl = in.a - fld(rec.p, P_DAMP) * vl;
      const V3<T> sq = vl * sx;
      const SV<T> c{cross(v.w, sq), cross(v.v, sq)};
      const S3<T> Ic = rot_sym(R, fld_s3(rec.p, P_IC));
      const V3<T> rw = mul(R, fld_v3(rec.p, P_C));
      SI<T> IA = cI;
      SV<T> pA = cp;
      add_body(fld(rec.p, P_M), rw, Ic, v, IA, pA);
      // the joint offset, 0 for a root (whose contribution to a parent is dropped)
      V3<T> d = fld_v3(rec.t, W_D);
      if (ADJ) {
        if (fr)
          ws3(s.root, 0, 0, WF_IC, Ic);
        else
          ws3(w, 0, 0, W_XY, Ic);
        wv3(w, 0, 0, W_RW, rw);
      }
      if (meta_treechild(m)) {
        --sp;
        IA += wsi(s.stk, WSW, sp, 0);
        pA += wsv(s.stk, WSW, sp, 21);
      }
      if (fr) {  // D = I^A, u = tau - p^A
        const SV<T> f{{tau[vo], tau[vo + 1], tau[vo + 2]}, {tau[vo + 3], tau[vo + 4], tau[vo + 5]}};
        if (ADJ) wsi(s.root, 0, 0, WF_IA, IA);
        wsv(w, 0, 0, W_AP, spd_solve<T, DT>(IA, f - pA));
        continue;
      }
      const SV<T> U{mul(IA.A, sx), mulT(IA.B, sx)};
      const DT Di = DT(1) / (DT)dot(sx, U.w);
      const T u = tl - dot(sx, pA.w);
      wsv(w, 0, 0, W_U, U);
      put_wdi<T, DT>(w, Di);
      w[W_u * LANES] = u;
      if (par < 0) d = zero3<T>();
      const SI<T> Ia = minus_scaled_outer<T, DT>(IA, Di, U);
      const SV<T> pa = pA + mul(Ia, c) + (T)((DT)u * Di) * U;
      const SI<T> Y = shift(Ia, d);
      const SV<T> pn = shift_force(pa, d);
      cI = Y;
      cp = pn;
      if (par != l - 1 || par < 0) {
        cI = zeroSI<T>();
        cp = zeroSV<T>();
        if (par >= 0 && meta_lastsib(m)) {
          wsi(s.stk, WSW, sp, 0, Y);
          wsv(s.stk, WSW, sp, 21, pn);
          ++sp;
        } else if (par >= 0) {
          wsi(s.stk, WSW, sp - 1, 0, wsi(s.stk, WSW, sp - 1, 0) + Y);
          wsv(s.stk, WSW, sp - 1, 21, wsv(s.stk, WSW, sp - 1, 21) + pn);
        }
      }
    }
  }
}

// INTEG: integrate into (qo, qdo), which may alias q, qd: a link's own coordinates are read
// before they are written.
template <class T, class DT, bool ADJ, bool INTEG, bool FR, bool STG>
SD void wpass_accel(const WSys<T, STG>& s, Col<const T> q, Col<const T> qd, V3<T> grav, T dt, int integ, Col<T> qo,
                    Col<T> qdo) {
  T* tp = s.tape;
  const int nl = s.nl, walk = s.walk();
  // outward: accelerations (and the integrator)
  Records<T, STG, 1, RING_FWD, 0, W_XY, 0, 0, 0, 0, W_V, 6> rec(s, walk);
  Inputs<T, STG, true> in(s, q, qd, 0, 1, walk);
  const SV<T> a0{zero3<T>(), -grav};
  SV<T> a_prev = a0;
  int sp = 0;
  for (int l = 0; l < walk; ++l) {
    rec.next();
    in.next();
    if (STG && l >= nl) continue;
    const int m = in.m;
    const int par = meta_parent(m), vi = meta_voff(m);
    T* w = tp + l * NWT * LANES;
    SV<T> a;
    if (FR && meta_jtype(m) == J_FREE) {
      a = wsv(w, 0, 0, W_AP);
      const V3<T> bv = a.v + mul(fld_m3(rec.t, W_E), grav);
      const T qdd[6] = {a.w.x, a.w.y, a.w.z, bv.x, bv.y, bv.z};
      if (ADJ)
        for (int i = 0; i < 6; ++i) s.root[(WF_QDD + i) * LANES] = qdd[i];
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
    } else {
      const V3<T> sx = fld_v3(rec.t, W_S);
      const SV<T> v = fld_sv(rec.t2, W_V);
      const SV<T> U = fld_sv(rec.t, W_U);
      const DT Di = fld_wdi<T, DT>(rec.t);
      const T u = fld(rec.t, W_u);
      const T v0 = in.b;
      const V3<T> sq = v0 * sx;
      SV<T> ap = a0;
      if (par >= 0) {
        SV<T> apar = a_prev;
        if (par != l - 1) {
          apar = wsv(s.stk, WSW, sp - 1, 0);
          if (meta_lastsib(m)) --sp;
        }
        ap = shift_motion(apar, fld_v3(rec.t, W_D));
      }
      ap += SV<T>{cross(v.w, sq), cross(v.v, sq)};
      const T qdd = (T)(((DT)u - (DT)dot(U, ap)) * Di);
      a = SV<T>{ap.w + qdd * sx, ap.v};
      if (ADJ) {
        wsv(w, 0, 0, W_AP, ap);
        w[W_QDD * LANES] = qdd;
      }
      if (INTEG) {
        const int qi = meta_qoff(m);
        const T v1 = v0 + dt * qdd;
        const T q1 = in.a + dt * (integ == I_SEMI_IMPLICIT ? v1 : v0);
        qdo[vi] = v1;
        qo[qi] = q1;
      }
    }
    if (meta_treechild(m)) {
      wsv(s.stk, WSW, sp, 0, a);
      ++sp;
    }
    a_prev = a;
  }
}

// The acceleration pass of one step from (q, qd), integrated into (qo, qdo), which may alias
// them, and the pose pass of the next in one walk: a rollout's two outward passes without the second round of record loads, and
// two independent chains (accelerations; orientations and velocities) in one instruction
// stream (rollout of 16384 trees of 2-64 links 119 -> 98 us a step).
template <class T, class DT, bool FR, bool STG>
SD void wpass_accel_pose(const WSys<T, STG>& s, Col<const T> q, Col<const T> qd, V3<T> grav, T dt, int integ,
                         Col<T> qo, Col<T> qdo) {
  T* tp = s.tape;
  const int nl = s.nl, walk = s.walk();
  Records<T, STG, 1, RING_ROLL, 0, W_XY, P_E, 12, 0, 0, W_V, 6> rec(s, walk);
  Inputs<T, STG, true> in(s, q, qd, 0, 1, walk);
  const SV<T> a0{zero3<T>(), -grav};
  SV<T> a_prev = a0, v_prev = zeroSV<T>();
  M3<T> R_prev = eye3<T>();
  int sp = 0;
  for (int l = 0; l < walk; ++l) {
    rec.next();
    in.next();
    if (STG && l >= nl) continue;
    const int m = in.m;
    const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
    T* w = tp + l * NWT * LANES;
    SV<T> a, v;
    M3<T> R;
    if (FR && meta_jtype(m) == J_FREE) {
      R = eye3<T>();
      a = wsv(w, 0, 0, W_AP);
      const V3<T> bv = a.v + mul(fld_m3(rec.t, W_E), grav);
      const T qdd[6] = {a.w.x, a.w.y, a.w.z, bv.x, bv.y, bv.z};
      T v1[6], nu[6], x[7];
      for (int i = 0; i < 6; ++i) {
        const T v0 = qd[vi + i];
        v1[i] = v0 + dt * qdd[i];
        qdo[vi + i] = v1[i];
        nu[i] = integ == I_SEMI_IMPLICIT ? v1[i] : v0;
      }
      for (int i = 0; i < 7; ++i) x[i] = q[qi + i];
      free_advance(x, nu, dt);
      for (int i = 0; i < 7; ++i) qo[qi + i] = x[i];
      v = SV<T>{{v1[0], v1[1], v1[2]}, {v1[3], v1[4], v1[5]}};
      wm3(w, 0, 0, W_E, free_rotation(x + 3, fld_m3(rec.p, P_E)));
    } else {
      SV<T> apar = a_prev, vp = v_prev;
      M3<T> Rp = R_prev;
      V3<T> d_old = fld_v3(rec.t, W_D);
      if (par < 0) {  // the world: d = 0 in the old step's shift
        apar = a0;
        vp = zeroSV<T>();
        Rp = eye3<T>();
        d_old = zero3<T>();
      } else if (par != l - 1) {
        Rp = wm3(s.stk, WSW, sp - 1, 0);
        vp = wsv(s.stk, WSW, sp - 1, 9);
        apar = wsv(s.stk, WSW, sp - 1, 15);
        if (meta_lastsib(m)) --sp;
      }
      const V3<T> sx = fld_v3(rec.t, W_S);
      const SV<T> vo = fld_sv(rec.t2, W_V);
      const T v0 = in.b;
      const V3<T> sq = v0 * sx;
      const SV<T> ap = shift_motion(apar, d_old) + SV<T>{cross(vo.w, sq), cross(vo.v, sq)};
      const T qdd = (T)(((DT)fld(rec.t, W_u) - (DT)dot(fld_sv(rec.t, W_U), ap)) * fld_wdi<T, DT>(rec.t));
      a = SV<T>{ap.w + qdd * sx, ap.v};
      const T v1 = v0 + dt * qdd;
      const T q1 = in.a + dt * (integ == I_SEMI_IMPLICIT ? v1 : v0);
      qdo[vi] = v1;
      qo[qi] = q1;
      T sn, cs;
      sincos_t(q1, &sn, &cs);
      const V3<T> d = mul(Rp, fld_v3(rec.p, P_R));
      R = mmT(Rp, rotz_T_mm(sn, cs, fld_m3(rec.p, P_E)));
      v = shift_motion(vp, d);
      v.w += v1 * col2(R);
      wv3(w, 0, 0, W_D, d);
    }
    put_rot(w, R);
    wsv(w, 0, 0, W_V, v);
    if (meta_treechild(m)) {
      wm3(s.stk, WSW, sp, 0, R);
      wsv(s.stk, WSW, sp, 9, v);
      wsv(s.stk, WSW, sp, 15, a);
      ++sp;
    }
    R_prev = R;
    v_prev = v;
    a_prev = a;
  }
}

// n steps from the state at x0, each state `stride` after the one before (a replayed segment;
// columns of B systems), q first, qd after nq coordinates.
template <class T, class DT, bool FR, bool STG, class TAU>
SD void wstep_replay(const WSys<T, STG>& s, T* x0, long long stride, long long B, int nq, long long n, TAU&& tau_of, V3<T> grav,
                     T dt, int integ) {
  T* x = x0;
  for (long long t = 0; t < n; ++t, x += stride) {
    const Col<const T> q{x, B}, qd{x + nq * B, B};
    const Col<T> qo{x + stride, B}, qdo{x + stride + nq * B, B};
    if (t == 0) wpass_pose<T, DT, false, FR>(s, q, qd);
    wpass_inward<T, DT, false, FR>(s, qd, tau_of(t));
    if (t + 1 < n)
      wpass_accel_pose<T, DT, FR>(s, q, qd, grav, dt, integ, qo, qdo);
    else
      wpass_accel<T, DT, false, true, FR>(s, q, qd, grav, dt, integ, qo, qdo);
  }
}

// One step for the state (q, qd) and joint force tau.
template <class T, class DT, bool ADJ, bool INTEG, bool FR = false, bool STG = false>
SD void wstep_forward(const WSys<T, STG>& s, Col<const T> q, Col<const T> qd, Col<const T> tau, V3<T> grav, T dt,
                      int integ, Col<T> qo, Col<T> qdo) {
  wpass_pose<T, DT, ADJ, FR>(s, q, qd);
  wpass_inward<T, DT, ADJ, FR>(s, qd, tau);
  wpass_accel<T, DT, ADJ, INTEG, FR>(s, q, qd, grav, dt, integ, qo, qdo);
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
// joint) needs the gravity, all that depends on a free root's orientation.
template <class T, class DT, bool FR = false, bool STG = false>
SD void wstep_adjoint(const WSys<T, STG>& s, Col<T> gq, Col<T> gqd, Col<T> gtau, Col<T> gm, T dt, int integ,
                      V3<T> grav = zero3<T>()) {
  T* tp = s.tape;
  T* ad = s.adj;
  const int nl = s.nl, walk = s.walk();
  // the integrator's adjoint and the inward half of lambda = M^-1 qddb (leaves -> root)
  {
    Records<T, STG, -1, RING_ADJ, 0, W_XY, 0, 0> rec(s, walk);
    SV<T> cy = zeroSV<T>();
    bool carry = false;
    int sp = 0;
    for (int l = walk - 1; l >= 0; --l) {
      rec.next();
      if (STG && l >= nl) continue;
      const int m = s.M(l);
      const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
      SV<T> y = carry ? cy : zeroSV<T>();
      carry = false;
      if (meta_treechild(m)) {
        --sp;
        y += wsv(s.stk, WSW, sp, 0);
      }
      if (FR && meta_jtype(m) == J_FREE) {  // lambda_root = (I^A)^-1 (qddb + y)
        T qt[4], nu[6], qddb6[6];
        for (int i = 0; i < 4; ++i) qt[i] = s.root[(WF_Q + i) * LANES];
        for (int i = 0; i < 6; ++i) {
          nu[i] = s.root[(WF_QD + i) * LANES];
          if (integ == I_SEMI_IMPLICIT) nu[i] += dt * s.root[(WF_QDD + i) * LANES];
        }
        free_integrator_adjoint(qt, nu, gq, gqd, qi, vi, dt, integ, qddb6);
        y += SV<T>{{qddb6[0], qddb6[1], qddb6[2]}, {qddb6[3], qddb6[4], qddb6[5]}};
        for (int i = 0; i < 3; ++i) s.root[(WF_QDDB + i) * LANES] = qddb6[3 + i];
        const SV<T> w = spd_solve<T, DT>(wsi(s.root, 0, 0, WF_IA), y);
        wsv(ad, NWA, l, WA_W, zeroSV<T>() - w);
        const T lam[6] = {w.w.x, w.w.y, w.w.z, w.v.x, w.v.y, w.v.z};
        for (int i = 0; i < 6; ++i) gtau[vi + i] = lam[i];
        continue;
      }
      T qddb;
      {
        const T qb = gq[qi], vb = gqd[vi];
        const T vt = vb + dt * qb;
        gqd[vi] = vt;
        qddb = dt * (integ == I_SEMI_IMPLICIT ? vt : vb);
      }
      const V3<T> sx = fld_v3(rec.t, W_S);
      const SV<T> U = fld_sv(rec.t, W_U);
      const T wb = (T)((DT)(qddb + dot(sx, y.w)) * fld_wdi<T, DT>(rec.t));
      s.tp(l, W_u) = wb;
      if (par >= 0) {
        const SV<T> yp = shift_force(y - wb * U, fld_v3(rec.t, W_D));
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
    Records<T, STG, 1, RING_ADJ, 0, W_XY, P_DAMP, 1> rec(s, walk);
    SV<T> W_prev = zeroSV<T>();
    int sp = 0;
    for (int l = 0; l < walk; ++l) {
      rec.next();
      if (STG && l >= nl) continue;
      const int m = s.M(l);
      const int par = meta_parent(m), vi = meta_voff(m);
      SV<T> W = zeroSV<T>();
      if (FR && meta_jtype(m) == J_FREE) {
        W = wsv(ad, NWA, l, WA_W);
      } else {
        if (par >= 0) {
          SV<T> Wp = W_prev;
          if (par != l - 1) {
            Wp = wsv(s.stk, WSW, sp - 1, 0);
            if (meta_lastsib(m)) --sp;
          }
          W = shift_motion(Wp, fld_v3(rec.t, W_D));
        }
        const SV<T> U = fld_sv(rec.t, W_U);
        const T lam = fld(rec.t, W_u) + (T)((DT)dot(U, W) * fld_wdi<T, DT>(rec.t));
        W.w = W.w - lam * fld_v3(rec.t, W_S);
        wsv(ad, NWA, l, WA_W, W);
        gtau[vi] = lam;
        gqd[vi] -= fld(rec.p, P_DAMP) * lam;
      }
      if (meta_treechild(m)) {
        wsv(s.stk, WSW, sp, 0, W);
        ++sp;
      }
      W_prev = W;
    }
  }
  // the derivative of L (leaves -> root)
  {
    Records<T, STG, -1, RING_ADJ, W_D, NWT - W_D, P_M, 1, WA_W, 6> rec(s, walk);
    SV<T> cv = zeroSV<T>(), ca = zeroSV<T>(), cw = zeroSV<T>();
    bool carry = false;
    int sp = 0;
    for (int l = walk - 1; l >= 0; --l) {
      rec.next();
      if (STG && l >= nl) continue;
      const int m = s.M(l);
      const int par = meta_parent(m), qi = meta_qoff(m), vi = meta_voff(m);
      const bool fr = FR && meta_jtype(m) == J_FREE;
      const V3<T> sx = fld_v3(rec.t, W_S);
      const SV<T> v = fld_sv(rec.t, W_V), ap = fld_sv(rec.t, W_AP), W = fld_sv(rec.a, WA_W);
      const T vl = fr ? T(0) : fld(rec.t, W_QD);
      const T qdd = fr ? T(0) : fld(rec.t, W_QDD);
      const SV<T> a{ap.w + qdd * sx, ap.v};
      const S3<T> Ic = fr ? ws3(s.root, 0, 0, WF_IC) : fld_s3(rec.t, W_XY);
      BodyGrad<T> g = body_grad(fld(rec.p, P_M), fld_v3(rec.t, W_RW), Ic, v, a, W);
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
      if (fr) {  // v = qd, a = qdd + [0; -E g]: only the gravity depends on the orientation
        const T vv[6] = {g.vb.w.x, g.vb.w.y, g.vb.w.z, g.vb.v.x, g.vb.v.y, g.vb.v.z};
        for (int i = 0; i < 6; ++i) gqd[vi + i] += vv[i];
        M3<T> Et;
        for (int i = 0; i < 9; ++i) Et.a[i] = s.P(l, P_E + i);
        // dL/da of the whole tree is -M lambda = -qddb, which the sum over the links only approaches
        const V3<T> qddb{s.root[WF_QDDB * LANES], s.root[(WF_QDDB + 1) * LANES], s.root[(WF_QDDB + 2) * LANES]};
        const M3<T> EJb = mmT(outer(qddb, grav), Et);  // E = E_J E_t
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
        const V3<T> d = fld_v3(rec.t, W_D);
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
