// One step and its forward-mode derivative on the world-aligned path (wjvp.cuh): one warp per
// 32-system tile, records in the caller's workspace staged through the warp's ring, the
// system's inputs and tangents copied to shared memory first.
#pragma once

namespace abasim {
namespace host {

// Scalars per tile in shared memory: the stack (sd > 0) and q, dq, qd, dqd, tau, dtau and the ring.
__host__ __device__ __forceinline__ long long wjvp_smem_per_tile(int nq, int nv, int sd) {
  return sd + 2LL * nq + 4LL * nv + 3 * RING_ADJ;
}
// Scalars per system of the workspace: tape, tangent record, stack.
__host__ __device__ __forceinline__ long long wjvp_work_words(int maxL, bool fr, int depth) {
  return w_tape_words(maxL, fr) + (long long)maxL * NWJ + (long long)depth * WSW;
}

template <class T, bool FR>
__global__ void __launch_bounds__(LANES)
k_wstep_jvp(DevModel<T> m, const T* __restrict__ q, const T* __restrict__ qd, const T* __restrict__ tau,
            const T* __restrict__ dq, const T* __restrict__ dqd, const T* __restrict__ dtau, T* q_out, T* qd_out,
            T* dq_out, T* dqd_out, T* work) {
  const int lane = threadIdx.x;
  const long long tile = blockIdx.x, B = m.B, L = m.maxL;
  const int slot = (int)tile * LANES + lane;
  const bool act = slot < B;
  const int b = act ? m.sys_of_slot[slot] : 0;
  const int nqm = m.nq_max, nvm = m.nv_max;
  T* ring = reinterpret_cast<T*>(g_smem);
  T* x = ring + 3 * RING_ADJ * LANES + lane;
  auto column = [&](const T* src, int n) {  // a [n][B] input (null: zeros) in shared memory
    T* c = x;
    for (int d = 0; d < n; ++d) c[d * LANES] = src ? src[d * B + b] : T(0);
    x += n * LANES;
    return Col<const T>{c, LANES};
  };
  const Col<const T> cq = column(q, nqm), cqd = column(qd, nvm), ct = column(tau, nvm);
  const Col<const T> cdq = column(dq, nqm), cdqd = column(dqd, nvm), cdt = column(dtau, nvm);
  T* tape = work + tile * wjvp_work_words(m.maxL, FR, m.wdepth) * LANES + lane;
  T* rec = tape + w_tape_words(m.maxL, FR) * LANES;
  const int nl = act ? m.nl[slot] : 0;
  const WSys<T, true> s{m.prm + tile * L * NPRM * LANES + lane, m.meta + tile * L * LANES + lane, tape, rec, nl, 1, NPRM,
                        m.sd ? x : rec + L * NWJ * LANES, tape + L * NWT * LANES, __reduce_max_sync(0xffffffffu, nl), ring,
                        true, lane};
  const V3<T> g{m.g0, m.g1, m.g2};
  wstep_forward<T, T, true, false, FR>(s, cq, cqd, ct, g, m.dt, m.integ, Col<T>{nullptr, 0}, Col<T>{nullptr, 0});
  wstep_jvp<T, T, FR>(s, cq, cqd, cdq, cdqd, cdt, g, m.dt, m.integ, Col<T>{q_out + b, B}, Col<T>{qd_out + b, B},
                      Col<T>{dq_out + b, B}, Col<T>{dqd_out + b, B});
  if (!act) return;
  // coordinates past the system's own pass through
  for (int d = m.nqv[slot] & 0xffff; d < nqm; ++d) {
    q_out[d * B + b] = cq[d];
    dq_out[d * B + b] = cdq[d];
  }
  for (int d = m.nqv[slot] >> 16; d < nvm; ++d) {
    qd_out[d * B + b] = cqd[d];
    dqd_out[d * B + b] = cdqd[d];
  }
}

}  // namespace host
}  // namespace abasim
