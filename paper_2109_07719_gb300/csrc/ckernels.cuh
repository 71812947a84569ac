// Rollout and adjoint kernels of models with contact spheres or joint limits (link-frame
// step, tapes in global memory): one to four warps per 32-system tile (contact_warps).  The first warp runs
// the step; the warps share the columns of A = J M^-1 J^T, three to a test pass, and their
// reverse in the adjoint, each with a contact tape of its own.
//
// Why: with feet on the ground the test passes were about half of a step (what the split
// below took away says so), on one warp of an SM's four schedulers (in FP64 each scheduler
// has its own half-lane-per-cycle unit, so one warp reached a quarter of the SM's rate).  A quadruped's four feet are four groups.
// Rollout + adjoint over 12 steps with four feet down: 512 quadrupeds in FP64 46.4 -> 30.6
// ms, 256 in FP32 8.0 -> 6.4, 8192 in the mixed mode 20.2 -> 14.4.  What is left is the first
// warp's: the ABA, the 20 sweeps of 12 dependent updates and their adjoints.
#pragma once

namespace abasim {
namespace host {

// This warp's view of a slot's contact tape and record.
template <class T> __device__ __forceinline__ long long contact_stride(const DevModel<T>& m) {
  return (m.B + LANES - 1) / LANES * m.maxL * NCT * LANES;
}
template <class T> __device__ __forceinline__ CView<T> cview_of(const DevModel<T>& m, long long tile, int lane, int warp) {
  T* ct = m.ctape + tile * m.maxL * NCT * LANES + lane;
  return CView<T>{ct, m.csys + tile * NCS * LANES + lane, warp > 0 ? ct + warp * contact_stride(m) : nullptr};
}

// The team's part of a step: every thread of the block calls it (act: the lane has a
// system).  ADJ as aba_forward's.  Returns the lane's number of active rows to the first
// warp (0 to the others); *any: some system of the tile has one.
template <class T, class DT, bool ADJ>
__device__ __forceinline__ int contact_step(const DevModel<T>& m, const Sys<T>& s, const CView<T>& cv, int warp, bool act,
                                            Col<const T> q, Col<const T> qd, Col<const T> tau_t, V3<T> g, bool* any) {
  const int parts = blockDim.x / LANES;
  int nr = 0;
  if (warp == 0 && act) {
    aba_forward<T, DT, ADJ>(s, q, qd, tau_t, g);
    nr = contact_rows<T, DT, T>(s, cv, q, qd, m.dt, m.cp);
  }
  *any = __syncthreads_or(nr > 0);
  if (*any) {
    if (act) contact_columns<T, DT, T>(s, cv, warp, parts);
    __syncthreads();
    if (nr > 0) contact_solve<T, DT, T>(s, cv, m.cp);
  }
  return nr;
}

// One step x -> x' in place.
template <class T, class DT>
__device__ __forceinline__ void contact_forward_step(const DevModel<T>& m, const Sys<T>& s, const CView<T>& cv, int warp,
                                                     bool act, Col<T> q, Col<T> qd, Col<const T> tau_t, V3<T> g,
                                                     Col<double> xw = Col<double>{nullptr, 0}) {
  bool any;
  const int nr = contact_step<T, DT, false>(m, s, cv, warp, act, Col<const T>{q.p, q.B}, Col<const T>{qd.p, qd.B}, tau_t,
                                            g, &any);
  if (warp == 0 && act) integrate_step<T, DT>(m, s, q, qd, nr > 0 ? (const T*)cv.ct : nullptr, xw);
}

// Recomputes the step from x^t and pulls the state adjoint back through it.  With active
// rows the integrator adjoint runs first for every link (the constraint adjoint needs all
// of qdd's adjoint), then the constraint adjoint, then the ABA adjoint with its terms added.
template <class T, class DT>
__device__ __forceinline__ void contact_adjoint_step(const DevModel<T>& m, const Sys<T>& s, const CView<T>& cv, int warp,
                                                     bool act, Col<const T> q, Col<const T> qd, Col<const T> tau_t,
                                                     Col<T> gq, Col<T> gqd, Col<T> gt, Col<T> gm, V3<T> g) {
  const int parts = blockDim.x / LANES;
  bool any;
  const int nr = contact_step<T, DT, true>(m, s, cv, warp, act, q, qd, tau_t, g, &any);
  if (any) {
    if (nr > 0) {
      for (int l = 0; l < s.nl; ++l) {
        const int mt = s.M(l);
        T qb[6] = {0, 0, 0, 0, 0, 0};
        integrator_adjoint(s, l, meta_jtype(mt), meta_qoff(mt), meta_voff(mt), q, qd, gq, gqd, m.dt, m.integ, qb,
                           (const T*)cv.ct);
        for (int i = 0; i < 6; ++i) cv.L(l, C_QDDB + i) = qb[i];
      }
      contact_adjoint_solve<T, DT, T>(s, cv, m.dt, m.cp);
    } else if (warp > 0 && act) {
      zero_accumulators(s, cv, B_OW);
    }
    __syncthreads();
    if (act) contact_adjoint_columns<T, DT, T>(s, cv, warp, parts);
    __syncthreads();
    if (parts > 1) {
      if (act) contact_adjoint_sum(s, cv, contact_stride(m), warp, parts);
      __syncthreads();
    }
    if (nr > 0) contact_adjoint_finish<T, DT, T>(s, cv, m.dt, m.cp);
  }
  if (warp == 0 && act) {
    if (nr > 0)
      step_adjoint<T, DT>(s, q, qd, gq, gqd, gt, gm, g, m.dt, m.integ, (const T*)cv.ct);
    else
      step_adjoint<T, DT>(s, q, qd, gq, gqd, gt, gm, g, m.dt, m.integ);
  }
}

// What a thread of a contact kernel works on.
template <class T> struct ContactLane {
  int warp, lane, slot, b;
  bool act, lead;  // the lane has a system; it is its first warp's
  Sys<T> s;
  CView<T> cv;
};
template <class T> __device__ __forceinline__ ContactLane<T> contact_lane(const DevModel<T>& m, long long tile) {
  ContactLane<T> c;
  c.warp = threadIdx.x / LANES;
  c.lane = threadIdx.x % LANES;
  c.slot = (int)tile * LANES + c.lane;
  c.act = c.slot < m.B;
  c.lead = c.act && c.warp == 0;
  c.b = c.act ? m.sys_of_slot[c.slot] : 0;
  const long long L = m.maxL;
  c.s = Sys<T>{m.prm + tile * L * NPRM * LANES + c.lane, m.meta + tile * L * LANES + c.lane,
               m.tape + tile * L * NTAPE * LANES + c.lane, m.adj + tile * L * NADJ * LANES + c.lane,
               c.act ? m.nl[c.slot] : 0, 1};
  c.cv = cview_of(m, tile, c.lane, c.warp);
  return c;
}

// T steps of a tile's systems.  The working state lives in (qT, qdT).
template <class T, class DT>
__device__ __forceinline__ void rollout_contact(const DevModel<T>& m, long long tile, const T* __restrict__ q0,
                                                const T* __restrict__ qd0, const T* __restrict__ tau, long long Tn,
                                                int k, T* ckpt, T* qT, T* qdT, T* traj) {
  const ContactLane<T> c = contact_lane(m, tile);
  const long long B = m.B;
  const int b = c.b, nqm = m.nq_max, nvm = m.nv_max, NX = nqm + nvm;
  const V3<T> g{m.g0, m.g1, m.g2};
  const Col<T> q{qT + b, B}, qd{qdT + b, B};
  Col<double> xw{nullptr, 0};
  auto put = [&](T* x) {  // the state into a [NX][B] array
    for (int d = 0; d < nqm; ++d) x[d * B + b] = q[d];
    for (int d = 0; d < nvm; ++d) x[(nqm + d) * B + b] = qd[d];
  };
  if (c.lead) {
    for (int d = 0; d < nqm; ++d) q[d] = q0[d * B + b];
    for (int d = 0; d < nvm; ++d) qd[d] = qd0[d * B + b];
    if constexpr (!std::is_same<T, DT>::value) {
      if (m.x64) {  // FP64 state accumulation, started from the FP32 initial state
        xw = Col<double>{m.x64 + b, B};
        for (int d = 0; d < nqm; ++d) xw[d] = (double)q[d];
        for (int d = 0; d < nvm; ++d) xw[nqm + d] = (double)qd[d];
      }
    }
    if (traj) put(traj);
  }
  for (long long t = 0; t < Tn; ++t) {
    if (c.lead && ckpt && t % k == 0) put(ckpt + (t / k) * NX * B);
    contact_forward_step<T, DT>(m, c.s, c.cv, c.warp, c.act, q, qd, Col<const T>{tau + t * nvm * B + b, B}, g, xw);
    if (c.lead && traj) put(traj + (t + 1) * NX * B);
  }
  if (!c.lead) return;
  bool ok = true;
  for (int d = 0; d < nqm; ++d) ok &= finite_t(q[d]);
  for (int d = 0; d < nvm; ++d) ok &= finite_t(qd[d]);
  if (!ok) m.status[b] |= 1;
}

// Adjoint rollout of a tile's systems.  (gq0, gqd0) carry the running state adjoint.
template <class T, class DT>
__device__ __forceinline__ void backward_contact(const DevModel<T>& m, long long tile, const T* __restrict__ ckpt,
                                                 const T* __restrict__ tau, long long Tn, int k,
                                                 const T* __restrict__ gqT, const T* __restrict__ gqdT,
                                                 const T* __restrict__ gtraj, T* gq0, T* gqd0, T* gtau, T* gm_acc,
                                                 T* ring) {
  const ContactLane<T> c = contact_lane(m, tile);
  const long long B = m.B;
  const int b = c.b, rs = c.act ? c.slot : 0, nqm = m.nq_max, nvm = m.nv_max, NX = nqm + nvm;
  const int nq = c.act ? m.nqv[c.slot] & 0xffff : 0, nv = c.act ? m.nqv[c.slot] >> 16 : 0;
  const V3<T> g{m.g0, m.g1, m.g2};
  const Col<T> gq{gq0 + b, B}, gqd{gqd0 + b, B}, gm{gm_acc + rs, B};
  auto add_seed = [&](const T* gx) {
    for (int d = 0; d < nq; ++d) gq[d] += gx[d * B + b];
    for (int d = 0; d < nv; ++d) gqd[d] += gx[(nqm + d) * B + b];
  };
  if (c.lead) {
    for (int d = 0; d < nqm; ++d) gq[d] = d < nq ? gqT[d * B + b] : T(0);
    for (int d = 0; d < nvm; ++d) gqd[d] = d < nv ? gqdT[d * B + b] : T(0);
    if (gtraj) add_seed(gtraj + Tn * NX * B);
    for (int l = 0; l < c.s.nl; ++l) gm[l] = T(0);
  }
  auto tau_of = [&](long long t) { return Col<const T>{tau + t * nvm * B + b, B}; };
  auto copy_state = [&](const T* from, T* to) {
    if (c.lead)
      for (int d = 0; d < NX; ++d) to[d * B] = from[d * B];
  };
  auto step_in_place = [&](T* x, long long t) {
    contact_forward_step<T, DT>(m, c.s, c.cv, c.warp, c.act, Col<T>{x, B}, Col<T>{x + nqm * B, B}, tau_of(t), g);
  };
  for (long long seg = (Tn + k - 1) / k - 1; seg >= 0; --seg) {
    const long long t0 = seg * k, t1 = t0 + k < Tn ? t0 + k : Tn;
    const T* xs = ckpt + seg * NX * B + b;
    if (k > 1 && !m.quadratic) {  // replay the segment once, keeping its states (ring by slot)
      copy_state(xs, ring + rs);
      for (long long j = 1; j < t1 - t0; ++j) {
        T* cur = ring + j * NX * B + rs;
        copy_state(ring + (j - 1) * NX * B + rs, cur);
        step_in_place(cur, t0 + j - 1);
      }
    }
    for (long long t = t1 - 1; t >= t0; --t) {
      const T* x = k > 1 ? ring + (t - t0) * NX * B + rs : xs;
      if (k > 1 && m.quadratic) {  // recompute x^t from the segment checkpoint: t - t0 steps
        T* cur = ring + rs;
        x = cur;
        copy_state(xs, cur);
        for (long long j = t0; j < t; ++j) step_in_place(cur, j);
      }
      T* gt = gtau + t * nvm * B + b;
      contact_adjoint_step<T, DT>(m, c.s, c.cv, c.warp, c.act, Col<const T>{x, B}, Col<const T>{x + nqm * B, B},
                                  tau_of(t), gq, gqd, Col<T>{gt, B}, gm, g);
      if (c.lead) {
        for (int d = nv; d < nvm; ++d) gt[d * B] = T(0);
        if (gtraj) add_seed(gtraj + t * NX * B);
      }
    }
  }
  if (!c.lead) return;
  bool ok = true;
  for (int d = 0; d < nq; ++d) ok &= finite_t(gq[d]);
  for (int d = 0; d < nv; ++d) ok &= finite_t(gqd[d]);
  for (int l = 0; l < c.s.nl; ++l) ok &= finite_t(gm[l]);
  if (!ok) m.status[b] |= 1;
}

// A work unit is a tile; the whole block walks it together.
#define ABASIM_FOR_EACH_TILE(m, ...)                                         \
  int unit = (m).persistent ? next_unit((m).counter) : (int)blockIdx.x;      \
  while ((long long)unit * LANES < (m).B) {                                  \
    __VA_ARGS__;                                                             \
    if (!(m).persistent) break;                                              \
    __syncthreads();                                                         \
    unit = next_unit((m).counter);                                           \
  }

template <class T, class DT>
__global__ void __launch_bounds__(CT_WARPS* LANES, 2)
k_rollout_contact(DevModel<T> m, const T* __restrict__ q0, const T* __restrict__ qd0, const T* __restrict__ tau,
                  long long Tn, int k, T* ckpt, T* qT, T* qdT, T* traj) {
  ABASIM_FOR_EACH_TILE(m, rollout_contact<T, DT>(m, unit, q0, qd0, tau, Tn, k, ckpt, qT, qdT, traj))
}

template <class T, class DT>
__global__ void __launch_bounds__(CT_WARPS* LANES, 2)
k_backward_contact(DevModel<T> m, const T* __restrict__ ckpt, const T* __restrict__ tau, long long Tn, int k,
                   const T* __restrict__ gqT, const T* __restrict__ gqdT, const T* __restrict__ gtraj, T* gq0, T* gqd0,
                   T* gtau, T* gm_acc, T* ring) {
  ABASIM_FOR_EACH_TILE(m, backward_contact<T, DT>(m, unit, ckpt, tau, Tn, k, gqT, gqdT, gtraj, gq0, gqd0, gtau, gm_acc,
                                                  ring))
}

}  // namespace host
}  // namespace abasim
