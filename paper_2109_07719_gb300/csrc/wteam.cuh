// The FP64 rollout of serial revolute chains by a team of four warps per 32-system tile, on
// the world-aligned step with everything on chip.
//
// Why: an FP64 instruction keeps a warp's scheduler busy for 64 cycles (its unit is half a
// lane wide), and the link-frame pipelined rollout keeps two of an SM's four schedulers
// busy, one of them with the rotate-and-shift of the articulated inertias.  Here what no
// link waits for from its neighbour (joint rotations, each body's own inertia, bias force
// and velocity products) is taken by the four warps in turn, and the chains are short: a
// translation instead of the congruence for the inertias, with the bias forces on a second
// warp beside them.  Phases, with a block barrier between them:
//   1 (warp 0)  accelerations of the last step and the integrator (root -> leaves)
//   2 (all)     E = R(e_z, q)^T E_tree;  checkpoint and trajectory of x^t (last warp)
//   3 (warp 0)  R, d, v (root -> leaves)
//   4 (all)     each body's inertia about its joint, bias force and c in world axes
//   5 (warp 0)  I^A, U, 1/D, I^a (leaves -> root)
//     (warp 1)  p^A, u, following warp 0 link by link (a named barrier per link)
// 1000 7-link chains 98 -> 66 us a step; one step of
// 64 of them 115 -> 73 us.  Not for two links, whose phases are mostly barriers and
// sin/cos (20.3 us a step pipelined, 26.4 so), nor in FP32, where the barriers and the
// copies between the phases cost what the split gains (4096 7-link chains 4.8 us a step
// pipelined, 5.5 so).
#pragma once

namespace abasim {
namespace host {

constexpr int TEAM = 4;            // warps
constexpr int TEAM_MIN_LINKS = 3;  // below: the pipelined rollout
// Tape words of a link: [0, W_AP) as the world-aligned tape; the body's own inertia (A block,
// m com), the nine words holding E between phases 2 and 3; its bias force; c; I^a.
enum : int { TM_A = W_AP, TM_G = TM_A + 6, TM_P = TM_G + 3, TM_C = TM_P + 6, TM_IA = TM_C + 6, NTM = TM_IA + 21 };

// Scalars per tile: the tape, model constants, meta words, the state and a double buffer of tau.
__host__ __device__ __forceinline__ long long team_smem_per_tile(int maxL, int nx, int nv) {
  return (long long)maxL * (NTM + NPRM_W + 1) + nx + 2LL * nv;
}

template <class T> struct TeamSys {
  const T* prm;     // [maxL][NPRM_W][LANES]
  const int* meta;  // [maxL][LANES], mstride apart
  T* tape;          // [maxL][NTM][LANES]
  int nl, mstride;
  __device__ __forceinline__ T* w(int l) const { return tape + l * NTM * LANES; }
  __device__ __forceinline__ const T* p(int l) const { return prm + l * NPRM_W * LANES; }
  __device__ __forceinline__ int M(int l) const { return meta[l * LANES * mstride]; }
};

// phase 1
template <class T>
__device__ __forceinline__ void team_accelerate(const TeamSys<T>& s, Col<T> q, Col<T> qd, V3<T> grav, T dt, int integ) {
  SV<T> a{zero3<T>(), -grav};
  for (int l = 0; l < s.nl; ++l) {
    const int m = s.M(l);
    const int qi = meta_qoff(m), vi = meta_voff(m);
    const T* w = s.w(l);
    if (l > 0) a = shift_motion(a, fld_v3(w, W_D));
    a += fld_sv(w, TM_C);
    const T qdd = (fld(w, W_u) - dot(fld_sv(w, W_U), a)) * fld_wdi<T, T>(w);
    a.w += qdd * fld_v3(w, W_S);
    const T v0 = qd[vi], v1 = v0 + dt * qdd;
    qd[vi] = v1;
    q[qi] = q[qi] + dt * (integ == I_SEMI_IMPLICIT ? v1 : v0);
  }
}

// phase 2, links first, first + TEAM, ...
template <class T> __device__ __forceinline__ void team_rotations(const TeamSys<T>& s, Col<T> q, int first) {
  for (int l = first; l < s.nl; l += TEAM) {
    T sn, cs;
    sincos_t((T)q[meta_qoff(s.M(l))], &sn, &cs);
    wm3(s.w(l), 0, 0, TM_A, rotz_T_mm(sn, cs, fld_m3(s.p(l), P_E)));
  }
}

// phase 3
template <class T> __device__ __forceinline__ void team_velocities(const TeamSys<T>& s, Col<T> qd) {
  M3<T> R = eye3<T>();
  SV<T> v = zeroSV<T>();
  for (int l = 0; l < s.nl; ++l) {
    T* w = s.w(l);
    const V3<T> d = mul(R, fld_v3(s.p(l), P_R));
    R = mmT(R, fld_m3((const T*)w, TM_A));
    v = shift_motion(v, d);
    v.w += (T)qd[meta_voff(s.M(l))] * col2(R);
    wv3(w, 0, 0, W_D, d);
    put_rot(w, R);
    wsv(w, 0, 0, W_V, v);
  }
}

// phase 4, links first, first + TEAM, ...
template <class T> __device__ __forceinline__ void team_bodies(const TeamSys<T>& s, Col<T> qd, int first) {
  for (int l = first; l < s.nl; l += TEAM) {
    T* w = s.w(l);
    const T* p = s.p(l);
    const M3<T> R = fld_rot((const T*)w);
    const SV<T> v = fld_sv((const T*)w, W_V);
    SI<T> IA = zeroSI<T>();
    SV<T> pA = zeroSV<T>();
    add_body(fld(p, P_M), mul(R, fld_v3(p, P_C)), rot_sym(R, fld_s3(p, P_IC)), v, IA, pA);
    ws3(w, 0, 0, TM_A, IA.A);
    wv3(w, 0, 0, TM_G, V3<T>{IA.B.a[7], IA.B.a[2], IA.B.a[3]});
    wsv(w, 0, 0, TM_P, pA);
    const V3<T> sq = (T)qd[meta_voff(s.M(l))] * col2(R);
    wsv(w, 0, 0, TM_C, SV<T>{cross(v.w, sq), cross(v.v, sq)});
  }
}

// phase 5, warp 0: announces each of the tile's links after its record is written
template <class T> __device__ __forceinline__ void team_inertias(const TeamSys<T>& s, int links) {
  SI<T> IA = zeroSI<T>();
  for (int l = links - 1; l >= 0; --l) {
    if (l < s.nl) {
      T* w = s.w(l);
      const V3<T> sx = fld_v3((const T*)w, W_S), g = fld_v3((const T*)w, TM_G);
      const T mass = fld(s.p(l), P_M);
      IA.A += fld_s3((const T*)w, TM_A);
      IA.B.a[1] -= g.z;
      IA.B.a[2] += g.y;
      IA.B.a[3] += g.z;
      IA.B.a[5] -= g.x;
      IA.B.a[6] -= g.y;
      IA.B.a[7] += g.x;
      IA.C.xx += mass;
      IA.C.yy += mass;
      IA.C.zz += mass;
      const SV<T> U{mul(IA.A, sx), mulT(IA.B, sx)};
      const T Di = T(1) / dot(sx, U.w);
      wsv(w, 0, 0, W_U, U);
      put_wdi<T, T>(w, Di);
      if (l > 0) {  // a root hands nothing on
        const SI<T> Ia = minus_scaled_outer<T, T>(IA, Di, U);
        wsi(w, 0, 0, TM_IA, Ia);
        IA = shift(Ia, fld_v3((const T*)w, W_D));
      }
    }
    __threadfence_block();
    __syncwarp();
    bar_arrive_id(1 + l);
  }
}

// phase 5, warp 1
template <class T>
__device__ __forceinline__ void team_biases(const TeamSys<T>& s, Col<T> qd, Col<const T> tau, int links) {
  SV<T> pA = zeroSV<T>();
  for (int l = links - 1; l >= 0; --l) {
    __syncwarp();
    bar_sync_id(1 + l);
    if (l >= s.nl) continue;
    T* w = s.w(l);
    const int vi = meta_voff(s.M(l));
    pA += fld_sv((const T*)w, TM_P);
    const T u = tau[vi] - fld(s.p(l), P_DAMP) * qd[vi] - dot(fld_v3((const T*)w, W_S), pA.w);
    w[W_u * LANES] = u;
    if (l > 0) {
      pA += mul(wsi(w, 0, 0, TM_IA), fld_sv((const T*)w, TM_C)) + (u * fld_wdi<T, T>((const T*)w)) * fld_sv((const T*)w, W_U);
      pA = shift_force(pA, fld_v3((const T*)w, W_D));
    }
  }
}

template <class T>
__global__ void __launch_bounds__(TEAM* LANES)
k_wrollout_team(DevModel<T> m, const T* __restrict__ q0, const T* __restrict__ qd0, const T* __restrict__ tau,
                long long Tn, int k, T* ckpt, T* qT, T* qdT, T* traj) {
  const int warp = threadIdx.x / LANES, lane = threadIdx.x % LANES;
  const long long B = m.B, L = m.maxL;
  const int nqm = m.nq_max, nvm = m.nv_max, NX = nqm + nvm;
  const V3<T> g{m.g0, m.g1, m.g2};
  constexpr int MS = (int)(sizeof(T) / sizeof(int));
  T* s_tape = reinterpret_cast<T*>(g_smem);
  T* s_prm = s_tape + L * NTM * LANES;
  T* s_meta = s_prm + L * NPRM_W * LANES;
  T* s_state = s_meta + L * LANES;
  T* s_tau = s_state + (long long)NX * LANES;  // [2][nvm][LANES]
  int* meta_l = reinterpret_cast<int*>(s_meta + lane);
  int unit = m.persistent ? next_unit(m.counter) : (int)blockIdx.x;
  while ((long long)unit * LANES < B) {
    const int slot = unit * LANES + lane;
    const bool act = slot < B;
    const int b = act ? m.sys_of_slot[slot] : 0;
    const int nl = act ? m.nl[slot] : 0;
    const int links = __reduce_max_sync(0xffffffffu, nl);
    const T* gprm = m.prm + (long long)unit * L * NPRM * LANES + lane;
    const int* gmeta = m.meta + (long long)unit * L * LANES + lane;
    for (int l = warp; l < nl; l += TEAM) {
      for (int f = 0; f < NPRM_W; ++f) s_prm[(l * NPRM_W + f) * LANES + lane] = gprm[(l * NPRM + f) * LANES];
      meta_l[l * LANES * MS] = gmeta[l * LANES];
    }
    const TeamSys<T> s{s_prm + lane, meta_l, s_tape + lane, nl, MS};
    const Col<T> q{s_state + lane, LANES}, qd{s_state + nqm * LANES + lane, LANES};
    auto fetch_tau = [&](long long t) {  // by warp 2
      if (act && t < Tn)
        for (int d = 0; d < nvm; ++d) cp_async(s_tau + ((t & 1) * nvm + d) * LANES + lane, tau + (t * nvm + d) * B + b);
      cp_commit();
    };
    if (warp == 0 && act) {
      for (int d = 0; d < nqm; ++d) q[d] = q0[d * B + b];
      for (int d = 0; d < nvm; ++d) qd[d] = qd0[d * B + b];
    }
    if (warp == 2) fetch_tau(0);
    auto put = [&](T* x) {  // the state into a [NX][B] array
      if (!act) return;
      for (int d = 0; d < nqm; ++d) x[d * B + b] = q[d];
      for (int d = 0; d < nvm; ++d) x[(nqm + d) * B + b] = qd[d];
    };
    __syncthreads();
    for (long long t = 0; t < Tn; ++t) {
      if (t > 0) {
        if (warp == 0) team_accelerate(s, q, qd, g, m.dt, m.integ);
        __syncthreads();
      }
      if (warp == TEAM - 1) {
        if (traj) put(traj + t * NX * B);
        if (ckpt && t % k == 0) put(ckpt + (t / k) * NX * B);
      }
      team_rotations(s, q, warp);
      __syncthreads();
      if (warp == 0) team_velocities(s, qd);
      if (warp == 2) {  // tau^t in place, tau^{t+1} on its way
        fetch_tau(t + 1);
        cp_wait_all_but_newest();
      }
      __syncthreads();
      team_bodies(s, qd, warp);
      __syncthreads();
      if (warp == 0) team_inertias(s, links);
      if (warp == 1) team_biases(s, qd, Col<const T>{s_tau + (t & 1) * nvm * LANES + lane, LANES}, links);
      __syncthreads();
    }
    if (warp == 2) cp_wait_all();
    if (warp == 0) {
      if (Tn > 0) team_accelerate(s, q, qd, g, m.dt, m.integ);
      if (act) {
        if (traj) put(traj + Tn * NX * B);
        bool ok = true;
        for (int d = 0; d < nqm; ++d) ok &= finite_t((T)q[d]);
        for (int d = 0; d < nvm; ++d) ok &= finite_t((T)qd[d]);
        if (!ok) m.status[b] |= 1;
        for (int d = 0; d < nqm; ++d) qT[d * B + b] = q[d];
        for (int d = 0; d < nvm; ++d) qdT[d * B + b] = qd[d];
      }
    }
    __syncthreads();  // shared memory is reused by the next unit
    if (!m.persistent) break;
    unit = next_unit(m.counter);
  }
}

}  // namespace host
}  // namespace abasim
