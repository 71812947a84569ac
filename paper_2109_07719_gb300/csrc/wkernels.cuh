// Batched rollout and adjoint kernels of the world-aligned step (wstep.cuh) for
// models without contact spheres or joint limits (FR: link 0 may be a free joint).  Thread i handles slot i (systems sorted by link count, longest first);
// the tape and adjoint record are tile-major, [tile][link][field][lane], in
// shared memory when a block's tiles fit (ONCHIP), else in the handle's global
// scratch with the working state and the prefetched input streams still on chip.
#pragma once

#include "wstep.cuh"

namespace abasim {
namespace host {

// Asks for the line at p (a step's inputs, one step ahead) to be brought into L2.
__device__ __forceinline__ void pf_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Scalars per system of one tape: the links' words, then the free root's record.
__host__ __device__ __forceinline__ long long w_tape_words(int maxL, bool fr) {
  return (long long)maxL * NWT + (fr ? NWF : 0);
}

// Scalars per 32-system tile a world-aligned kernel keeps in shared memory: the
// working state (x for the rollout, the state adjoint and the per-link
// mass-gradient sums for the backward pass); with ONCHIP also the tape (and, for
// the adjoint, the adjoint record), the model constants and meta words, the stack
// of parent values (sd scalars per system) and a double buffer for the per-step
// inputs (tau, plus x^t for the adjoint) fetched one step ahead.  Without ONCHIP
// the records are in the handle's global scratch and a ring of `slots` slots stages them
// (wstep.cuh); the stack is here too if the launch has room (sd > 0).
__host__ __device__ __forceinline__ long long w_smem_per_tile(int maxL, int nx, int nv, bool bwd, bool onchip,
                                                              int sd, bool fr, int slots) {
  const long long state = nx + (bwd ? maxL : 0);
  if (!onchip) return state + sd + (long long)slots * (bwd ? RING_ADJ : RING_ROLL);
  return w_tape_words(maxL, fr) + (long long)maxL * ((bwd ? NWA : 0) + NPRM_W + 1) + sd + state +
         2LL * (nv + (bwd ? nx : 0));
}

// Stack `which` (the warp's number in the pipelined adjoint, else 0) of a tile's
// system at `lane` in the handle's global scratch (null when no system branches).
template <class T>
__device__ __forceinline__ T* w_stack(const DevModel<T>& m, int which, long long tile, long long lane) {
  if (!m.stk) return nullptr;
  const long long tiles = (m.B + LANES - 1) / LANES;
  return m.stk + ((long long)which * tiles + tile) * m.wdepth * WSW * LANES + lane;
}

template <class T> struct WTile {
  T* tape;
  T* adj;
  T* prm;
  int* meta;
  T* stk;
  T* ring;  // at lane 0
  T* state;
  T* gm;
  T* stream;
};

template <class T, bool BWD, bool ONCHIP, bool FR>
__device__ __forceinline__ WTile<T> w_tile(const DevModel<T>& m, int lane) {
  const int tb = threadIdx.x / LANES;
  const long long L = m.maxL;
  const int nx = m.nq_max + m.nv_max, sd = ONCHIP ? m.wdepth * WSW : m.sd;
  T* base = reinterpret_cast<T*>(g_smem) +
            (long long)tb * w_smem_per_tile(m.maxL, nx, m.nv_max, BWD, ONCHIP, sd, FR, m.slots) * LANES + lane;
  WTile<T> t{};
  if (ONCHIP) {
    t.tape = base;
    base += w_tape_words(m.maxL, FR) * LANES;
    t.adj = base;
    if (BWD) base += L * NWA * LANES;
    t.prm = base;
    base += L * NPRM_W * LANES;
    t.meta = reinterpret_cast<int*>(base);
    base += L * LANES;
  } else {
    t.ring = base - lane;
    base += (long long)m.slots * (BWD ? RING_ADJ : RING_ROLL) * LANES;
  }
  t.stk = base;
  base += (long long)sd * LANES;
  t.state = base;
  base += (long long)nx * LANES;
  t.gm = base;
  if (BWD) base += L * LANES;
  t.stream = base;
  return t;
}

// The system view of a slot: constants, meta words and tape on chip (copied in here) or
// in global memory.  Every lane of the warp calls it; a lane past the batch has nl = 0.
template <class T, bool BWD, bool ONCHIP, bool FR>
__device__ __forceinline__ WSys<T, !ONCHIP> wsys_of(const DevModel<T>& m, int slot, bool act) {
  const long long tile = slot / LANES, lane = slot % LANES;
  const long long L = m.maxL;
  const T* gprm = m.prm + tile * L * NPRM * LANES + lane;
  const int* gmeta = m.meta + tile * L * LANES + lane;
  const int nl = act ? m.nl[slot] : 0;
  const WTile<T> t = w_tile<T, BWD, ONCHIP, FR>(m, (int)lane);
  if constexpr (ONCHIP) {
    constexpr int MS = (int)(sizeof(T) / sizeof(int));
    for (int l = 0; l < nl; ++l) {
      for (int f = 0; f < NPRM_W; ++f) t.prm[(l * NPRM_W + f) * LANES] = gprm[(l * NPRM + f) * LANES];
      t.meta[l * LANES * MS] = gmeta[l * LANES];
    }
    return WSys<T>{t.prm, t.meta, t.tape, t.adj, nl, MS, NPRM_W, t.stk, t.tape + L * NWT * LANES};
  } else {
    T* tape = m.tape + tile * w_tape_words(m.maxL, FR) * LANES + lane;
    return WSys<T, true>{gprm, gmeta, tape, m.adj + tile * L * NWA * LANES + lane, nl, 1, NPRM,
                         m.sd ? t.stk : w_stack(m, 0, tile, lane), tape + L * NWT * LANES,
                         __reduce_max_sync(0xffffffffu, nl), t.ring, m.slots > 1, (int)lane};
  }
}

// One system's rollout.  Without ONCHIP every lane of a warp takes part (act: the lane has
// a system; the others only help to stage records).
template <class T, class DT, bool ONCHIP, bool FR>
__device__ __forceinline__ void wrollout_one(const DevModel<T>& m, int slot, bool act, const T* __restrict__ q0,
                                             const T* __restrict__ qd0, const T* __restrict__ tau, long long Tn,
                                             int k, T* ckpt, T* qT, T* qdT, T* traj) {
  const int b = act ? m.sys_of_slot[slot] : 0;
  const long long B = m.B;
  const int nqm = m.nq_max, nvm = m.nv_max, NX = nqm + nvm;
  const V3<T> g{m.g0, m.g1, m.g2};
  const WSys<T, !ONCHIP> s = wsys_of<T, false, ONCHIP, FR>(m, slot, act);
  const WTile<T> st = w_tile<T, false, ONCHIP, FR>(m, slot % LANES);
  const Col<T> q{st.state, LANES}, qd{st.state + nqm * LANES, LANES};
  const int nv = act ? m.nqv[slot] >> 16 : 0;
  T* sbuf = st.stream;  // ONCHIP: [2][nvm][LANES], tau one step ahead
  if (ONCHIP) {
    if (Tn > 0)
      for (int d = 0; d < nvm; ++d) cp_async(sbuf + d * LANES, tau + (long long)d * B + b);
    cp_commit();
  }
  for (int d = 0; d < nqm; ++d) q[d] = q0[d * B + b];
  for (int d = 0; d < nvm; ++d) qd[d] = qd0[d * B + b];
  auto put = [&](T* c) {  // the state x into a [NX][B] array
    if (!act) return;
    for (int d = 0; d < nqm; ++d) c[d * B + b] = q[d];
    for (int d = 0; d < nvm; ++d) c[(nqm + d) * B + b] = qd[d];
  };
  const Col<const T> cq{q.p, LANES}, cqd{qd.p, LANES};
  for (long long t = 0; t < Tn; ++t) {
    if (t == 0)
      wpass_pose<T, DT, false, FR>(s, cq, cqd);
    else  // x^t from step t - 1's accelerations, and its pose
      wpass_accel_pose<T, DT, FR>(s, cq, cqd, g, m.dt, m.integ, q, qd);
    if (traj) put(traj + t * NX * B);
    if (ckpt && t % k == 0) put(ckpt + (t / k) * NX * B);
    Col<const T> tau_t{tau + t * nvm * B + b, B};
    if (ONCHIP) {
      if (t + 1 < Tn) {
        T* nb = sbuf + ((t + 1) & 1) * nvm * LANES;
        for (int d = 0; d < nvm; ++d) cp_async(nb + d * LANES, tau + ((t + 1) * nvm + d) * B + b);
      }
      cp_commit();
      cp_wait_all_but_newest();
      tau_t = Col<const T>{sbuf + (t & 1) * nvm * LANES, LANES};
    } else if (t + 1 < Tn && m.slots > 1) {
      for (int d = 0; d < nv; ++d) pf_line(tau + ((t + 1) * nvm + d) * B + b);
    }
    wpass_inward<T, DT, false, FR>(s, cqd, tau_t);
  }
  if (Tn > 0) wpass_accel<T, DT, false, true, FR>(s, cq, cqd, g, m.dt, m.integ, q, qd);
  if (traj) put(traj + Tn * NX * B);
  if (ONCHIP) cp_wait_all();
  if (!act) return;
  bool ok = true;
  for (int d = 0; d < nqm; ++d) ok &= finite_t(q[d]);
  for (int d = 0; d < nvm; ++d) ok &= finite_t(qd[d]);
  if (!ok) m.status[b] |= 1;
  for (int d = 0; d < nqm; ++d) qT[d * B + b] = q[d];
  for (int d = 0; d < nvm; ++d) qdT[d * B + b] = qd[d];
}

template <class T, class DT, bool ONCHIP, bool FR>
__device__ __forceinline__ void wbackward_one(const DevModel<T>& m, int slot, bool act, const T* __restrict__ ckpt,
                                              const T* __restrict__ tau, long long Tn, int k,
                                              const T* __restrict__ gqT, const T* __restrict__ gqdT,
                                              const T* __restrict__ gtraj, T* gq0, T* gqd0, T* gtau, T* gm_acc,
                                              T* ring) {
  const int b = act ? m.sys_of_slot[slot] : 0;
  const long long B = m.B;
  const int nqm = m.nq_max, nvm = m.nv_max, NX = nqm + nvm;
  const int nq = act ? m.nqv[slot] & 0xffff : 0, nv = act ? m.nqv[slot] >> 16 : 0;
  const int rs = act ? slot : 0;  // this lane's column of the replay ring
  const V3<T> g{m.g0, m.g1, m.g2};
  const WSys<T, !ONCHIP> s = wsys_of<T, true, ONCHIP, FR>(m, slot, act);
  const WTile<T> st = w_tile<T, true, ONCHIP, FR>(m, slot % LANES);
  const Col<T> gq{st.state, LANES}, gqd{st.state + nqm * LANES, LANES}, gm{st.gm, LANES};
  T* sbuf = st.stream;  // ONCHIP: [2][NX + nvm][LANES]: x^t and tau^t, one step ahead (k = 1)
  for (int d = 0; d < nqm; ++d) {
    T v = d < nq ? gqT[d * B + b] : T(0);
    if (gtraj && d < nq) v += gtraj[(Tn * NX + d) * B + b];
    gq[d] = v;
  }
  for (int d = 0; d < nvm; ++d) {
    T v = d < nv ? gqdT[d * B + b] : T(0);
    if (gtraj && d < nv) v += gtraj[(Tn * NX + nqm + d) * B + b];
    gqd[d] = v;
  }
  for (int l = 0; l < s.nl; ++l) gm[l] = T(0);
  auto step_back = [&](long long t, Col<const T> q, Col<const T> qd, Col<const T> tau_t) {
    wstep_forward<T, DT, true, false, FR>(s, q, qd, tau_t, g, m.dt, m.integ, Col<T>{nullptr, 0}, Col<T>{nullptr, 0});
    T* gt = gtau + t * nvm * B + b;
    wstep_adjoint<T, DT, FR>(s, gq, gqd, Col<T>{gt, B}, gm, m.dt, m.integ, g);
    if (act)
      for (int d = nv; d < nvm; ++d) gt[d * B] = T(0);
    if (gtraj) {
      const T* gx = gtraj + t * NX * B + b;
      for (int d = 0; d < nq; ++d) gq[d] += gx[d * B];
      for (int d = 0; d < nv; ++d) gqd[d] += gx[(nqm + d) * B];
    }
  };
  auto replay = [&](const T* from, T* to, long long t) {  // one step from state `from` to state `to`
    wstep_forward<T, DT, false, true, FR>(s, Col<const T>{from, B}, Col<const T>{from + nqm * B, B},
                                          Col<const T>{tau + t * nvm * B + b, B}, g, m.dt, m.integ, Col<T>{to, B},
                                          Col<T>{to + nqm * B, B});
  };
  if (k == 1 && ONCHIP) {
    const int W = NX + nvm;
    auto fetch = [&](long long t, int buf) {
      T* dst = sbuf + buf * W * LANES;
      for (int d = 0; d < NX; ++d) cp_async(dst + d * LANES, ckpt + (t * NX + d) * B + b);
      for (int d = 0; d < nvm; ++d) cp_async(dst + (NX + d) * LANES, tau + (t * nvm + d) * B + b);
    };
    if (Tn > 0) fetch(Tn - 1, (int)((Tn - 1) & 1));
    cp_commit();
    for (long long t = Tn - 1; t >= 0; --t) {
      if (t > 0) fetch(t - 1, (int)((t - 1) & 1));
      cp_commit();
      cp_wait_all_but_newest();
      const T* xb = sbuf + (t & 1) * W * LANES;
      step_back(t, Col<const T>{xb, LANES}, Col<const T>{xb + nqm * LANES, LANES},
                Col<const T>{xb + NX * LANES, LANES});
    }
    cp_wait_all();
  } else if (k == 1) {  // inputs straight from global memory, the previous step's lines prefetched
    for (long long t = Tn - 1; t >= 0; --t) {
      if (t > 0 && m.slots > 1) {
        const T* xn = ckpt + (t - 1) * NX * B + b;
        for (int d = 0; d < nq; ++d) pf_line(xn + d * B);
        for (int d = 0; d < nv; ++d) pf_line(xn + (nqm + d) * B);
        for (int d = 0; d < nv; ++d) pf_line(tau + ((t - 1) * nvm + d) * B + b);
      }
      const T* x = ckpt + t * NX * B + b;
      step_back(t, Col<const T>{x, B}, Col<const T>{x + nqm * B, B}, Col<const T>{tau + t * nvm * B + b, B});
    }
  } else {
    const long long nseg = (Tn + k - 1) / k;
    for (long long seg = nseg - 1; seg >= 0; --seg) {
      const long long t0 = seg * k;
      const long long t1 = (t0 + k < Tn) ? t0 + k : Tn;
      const T* xs = ckpt + seg * NX * B + b;
      if (!m.quadratic) {  // replay the segment once, keeping its states (ring by slot)
        T* r0 = ring + rs;
        if (act)
          for (int d = 0; d < NX; ++d) r0[d * B] = xs[d * B];
        wstep_replay<T, DT, FR>(s, r0, NX * B, B, nqm, t1 - t0 - 1,
                                [&](long long j) { return Col<const T>{tau + (t0 + j) * nvm * B + b, B}; }, g, m.dt,
                                m.integ);
      }
      for (long long t = t1 - 1; t >= t0; --t) {
        const T* x = ring + (t - t0) * NX * B + rs;
        if (m.quadratic) {  // recompute x^t from the segment checkpoint: t - t0 steps
          T* cur = ring + rs;
          x = t == t0 ? xs : cur;
          if (t > t0) {
            replay(xs, cur, t0);
            for (long long j = t0 + 1; j < t; ++j) replay(cur, cur, j);
          }
        }
        step_back(t, Col<const T>{x, B}, Col<const T>{x + nqm * B, B}, Col<const T>{tau + t * nvm * B + b, B});
      }
    }
  }
  if (!act) return;
  bool ok = true;
  for (int d = 0; d < nq; ++d) ok &= finite_t(gq[d]);
  for (int d = 0; d < nv; ++d) ok &= finite_t(gqd[d]);
  for (int l = 0; l < s.nl; ++l) ok &= finite_t(gm[l]);
  if (!ok) m.status[b] |= 1;
  for (int d = 0; d < nqm; ++d) gq0[d * B + b] = gq[d];
  for (int d = 0; d < nvm; ++d) gqd0[d * B + b] = gqd[d];
  for (int l = 0; l < s.nl; ++l) gm_acc[l * B + slot] = gm[l];
}

// Runs `...` for every slot of this block's work units.  The lanes of a warp that stages
// records run it together, those past the batch with act false.
#define ABASIM_FOR_EACH_WSLOT(m, ...)                                        \
  int unit = (m).persistent ? next_unit((m).counter) : (int)blockIdx.x;      \
  while ((long long)unit * blockDim.x < (m).B) {                             \
    const int slot = unit * blockDim.x + threadIdx.x;                        \
    const bool act = slot < (m).B;                                           \
    if (ONCHIP ? act : slot / LANES * LANES < (m).B) { __VA_ARGS__; }        \
    if (!(m).persistent) break;                                              \
    unit = next_unit((m).counter);                                           \
  }

template <class T, class DT, bool ONCHIP, bool FR>
__global__ void k_wrollout(DevModel<T> m, const T* __restrict__ q0, const T* __restrict__ qd0,
                           const T* __restrict__ tau, long long Tn, int k, T* ckpt, T* qT, T* qdT, T* traj) {
  ABASIM_FOR_EACH_WSLOT(m, wrollout_one<T, DT, ONCHIP, FR>(m, slot, act, q0, qd0, tau, Tn, k, ckpt, qT, qdT, traj))
}

template <class T, class DT, bool ONCHIP, bool FR>
__global__ void k_wbackward(DevModel<T> m, const T* __restrict__ ckpt, const T* __restrict__ tau, long long Tn,
                            int k, const T* __restrict__ gqT, const T* __restrict__ gqdT,
                            const T* __restrict__ gtraj, T* gq0, T* gqd0, T* gtau, T* gm_acc, T* ring) {
  ABASIM_FOR_EACH_WSLOT(m, wbackward_one<T, DT, ONCHIP, FR>(m, slot, act, ckpt, tau, Tn, k, gqT, gqdT, gtraj, gq0,
                                                            gqd0, gtau, gm_acc, ring))
}

}  // namespace host
}  // namespace abasim
