// The pipelined adjoint of the world-aligned step: a consumer warp and one or more
// producer warps per 32-system tile, for models without contacts or limits.  With every step's initial state checkpointed, the recompute
// of step t (Sec. 3.2, Eq. 7: Z^t = G(x^t)) depends on no adjoint, so the producers
// recompute steps ahead, in turn, into a ring of tapes while the consumer runs the
// adjoint of step after step.  Step j (counted from the last one) lives in tape j mod NT
// and is recomputed by producer j mod NP, with NT = NP (two for one producer), so that a
// tape has one producer.  The hand-off is a pair of named barriers per tape (hardware
// barriers, no spinning): FULL(b) (the producer arrives when tape b holds its step; the
// consumer waits) and EMPTY(b) (the consumer arrives when it has finished a step from tape
// b that will be reused; the producer waits before overwriting).  Both sides execute every
// barrier the same number of times whatever the systems, and neither arrives twice before
// the other's matching wait: a tape's next FULL arrival follows its EMPTY wait, which
// follows the consumer's FULL wait, and vice versa.  (A tape shared by several producers
// would need more: one could take the EMPTY arrival meant for another.)
//
// SEG, a checkpoint every k > 1 steps: a segment's states are replayed once into the
// caller's workspace by the producer of the segment's first (latest) step, with that step's
// tape as scratch, between two barriers of the producers (all have read the previous
// segment's states; all may read this one's); the consumer meanwhile finishes the steps of
// the previous segment.
//
// Why several producers: the implicit-form adjoint takes less time than the recompute
// (468 against 670 operations a link), so with one producer the consumer waits; how many
// is the launch's choice (launch_wbackward_pipe).  The tapes, the adjoint record, the
// model constants and the inputs live on chip when the block's shared memory holds them
// (ONCHIP), else in global memory (the tapes in the handle's ring), staged by each warp.
#pragma once

namespace abasim {
namespace host {

__host__ __device__ __forceinline__ int wpipe_tapes(int np) { return np > 1 ? np : 2; }

// Scalars per tile: the state adjoint and per-link mass-gradient sums; with
// ONCHIP also the tapes, the adjoint record, model constants and meta words, the
// warps' stacks of parent values (sd scalars per system each) and each producer's
// double-buffered inputs (x^t, tau^t); without ONCHIP the warps' rings of `slots`
// slots, and their stacks if the launch has room (sd > 0).
__host__ __device__ __forceinline__ long long wpipe_smem_per_tile(int maxL, int nx, int nv, bool onchip, int sd,
                                                                  bool fr, int np, int slots, bool seg) {
  const long long state = nx + maxL;
  if (!onchip) return state + (np + 1LL) * sd + (long long)slots * (RING_ADJ + np * (seg ? RING_ROLL : RING_FWD));
  return wpipe_tapes(np) * w_tape_words(maxL, fr) + (np + 1LL) * sd + (long long)maxL * (NWA + NPRM_W + 1) + state +
         2LL * np * (nx + nv);
}

__device__ __forceinline__ void pipe_sync(int id) { asm volatile("bar.sync %0, 64;\n" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pipe_arrive(int id) { asm volatile("bar.arrive %0, 64;\n" ::"r"(id) : "memory"); }

// all producers of a block
__device__ __forceinline__ void producers_sync(int nt, int np) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(1 + 2 * nt), "r"(np * LANES) : "memory");
}

// Registers: an on-chip block may have its SM alone; three global-tape blocks of one consumer
// and up to three producers share one (FP64: two).
template <class T, class DT, bool ONCHIP, bool FR, bool SEG>
__global__ void __launch_bounds__(LANES * (WPIPE_TAPES + 1),
                                  ONCHIP ? 1 : sizeof(T) == 4 ? 3 : 2)
k_wbackward_pipe(DevModel<T> m, const T* __restrict__ ckpt, const T* __restrict__ tau, long long Tn, int k,
                 const T* __restrict__ gqT, const T* __restrict__ gqdT, const T* __restrict__ gtraj, T* gq0,
                 T* gqd0, T* gtau, T* gm_acc, T* ring) {
  const int warp = threadIdx.x / LANES, lane = threadIdx.x % LANES;
  const int NP = blockDim.x / LANES - 1, NT = wpipe_tapes(NP);
  const bool consumer = warp == 0;
  const long long B = m.B;
  const int nqm = m.nq_max, nvm = m.nv_max, NX = nqm + nvm;
  const long long L = m.maxL;
  const long long TW = w_tape_words(m.maxL, FR);
  const long long units = (B + LANES - 1) / LANES;
  const V3<T> g{m.g0, m.g1, m.g2};
  constexpr int MS = (int)(sizeof(T) / sizeof(int));
  constexpr int RING_PROD = SEG ? RING_ROLL : RING_FWD;  // a replay's fused pass reads more rows
  T* base = reinterpret_cast<T*>(g_smem);
  T *s_tape = nullptr, *s_adj = nullptr, *s_prm = nullptr, *s_meta = nullptr, *s_in = nullptr;
  T* s_ring = nullptr;
  const long long sdw = ONCHIP ? (long long)m.wdepth * WSW : m.sd;  // stack scalars per system on chip
  if (ONCHIP) {
    s_tape = base;  // [NT][tape words][LANES]
    base += NT * TW * LANES;
    s_adj = base;
    base += L * NWA * LANES;
    s_prm = base;
    base += L * NPRM_W * LANES;
    s_meta = base;
    base += L * LANES;
  } else {
    s_ring = base + (long long)m.slots * LANES * (consumer ? 0 : RING_ADJ + (warp - 1) * RING_PROD);
    base += (long long)m.slots * LANES * (RING_ADJ + NP * RING_PROD);
  }
  T* s_stk = base + warp * sdw * LANES + lane;  // [NP + 1][sdw][LANES]: one per warp
  base += (NP + 1) * sdw * LANES;
  T* s_state = base;
  T* s_gm = s_state + (long long)NX * LANES;
  const int W = NX + nvm;
  if (ONCHIP && !consumer) s_in = s_gm + L * LANES + (long long)(warp - 1) * 2 * W * LANES;  // [2][NX + nvm][LANES]
  int unit = m.persistent ? next_unit(m.counter) : (int)blockIdx.x;
  while ((long long)unit * LANES < B) {
    const int slot = unit * LANES + lane;
    const bool act = slot < B;
    const int b = act ? m.sys_of_slot[slot] : 0;
    const int nl = act ? m.nl[slot] : 0;
    const int nq = act ? (m.nqv[slot] & 0xffff) : 0, nv = act ? (m.nqv[slot] >> 16) : 0;
    const int links = __reduce_max_sync(0xffffffffu, nl);
    const T* gprm = m.prm + (long long)unit * L * NPRM * LANES + lane;
    const int* gmeta = m.meta + (long long)unit * L * LANES + lane;
    int* meta_l = ONCHIP ? reinterpret_cast<int*>(s_meta + lane) : nullptr;
    if (ONCHIP && consumer && act) {
      for (int l = 0; l < nl; ++l) {
        for (int f = 0; f < NPRM_W; ++f) s_prm[(l * NPRM_W + f) * LANES + lane] = gprm[(l * NPRM + f) * LANES];
        meta_l[l * LANES * MS] = gmeta[l * LANES];
      }
    }
    __syncthreads();
    auto sys_of_buf = [&](int buf) -> WSys<T, !ONCHIP> {
      if constexpr (ONCHIP) {
        T* tape = s_tape + buf * TW * LANES + lane;
        return WSys<T>{s_prm + lane, meta_l, tape, s_adj + lane, nl, MS, NPRM_W, s_stk, tape + L * NWT * LANES};
      } else {
        T* tape = m.tape + (buf * units + unit) * TW * LANES + lane;
        return WSys<T, true>{gprm, gmeta, tape, m.adj + (long long)unit * L * NWA * LANES + lane, nl, 1, NPRM,
                             m.sd ? s_stk : w_stack(m, warp, unit, lane), tape + L * NWT * LANES, links, s_ring,
                             m.slots > 1, lane};
      }
    };
    // x^t: the checkpoint, or (SEG) the replayed state of the segment that starts at t0
    auto state_of = [&](long long t, long long t0) -> const T* {
      return SEG ? ring + (t - t0) * NX * B + (act ? slot : 0) : ckpt + t * NX * B + b;
    };
    // a producer's inputs of step t: x^t and tau^t (the system's own coordinates)
    auto fetch = [&](long long t, long long t0, int buf) {
      T* dst = s_in + buf * W * LANES + lane;
      const T* x = state_of(t, t0);
      for (int d = 0; d < nq; ++d) cp_async(dst + d * LANES, x + d * B);
      for (int d = 0; d < nv; ++d) cp_async(dst + (nqm + d) * LANES, x + (nqm + d) * B);
      for (int d = 0; d < nv; ++d) cp_async(dst + (NX + d) * LANES, tau + (t * nvm + d) * B + b);
    };
    // the segment's states x^{t0 + 1} .. x^{t1 - 1} from its checkpoint, one step each
    auto replay = [&](const WSys<T, !ONCHIP>& sp, long long seg, long long t0, long long t1) {
      if constexpr (SEG) {
        T* r = ring + (act ? slot : 0);
        const T* xs = ckpt + seg * NX * B + b;
        if (act)
          for (int d = 0; d < NX; ++d) r[d * B] = xs[d * B];
        if (ONCHIP ? act : true)
          wstep_replay<T, DT, FR>(sp, r, NX * B, B, nqm, t1 - t0 - 1,
                                  [&](long long j) { return Col<const T>{tau + (t0 + j) * nvm * B + b, B}; }, g, m.dt,
                                  m.integ);
        __threadfence_block();
        __syncwarp();
      }
    };
    if (!consumer) {  // producer `warp`: recompute steps j = warp - 1, warp - 1 + NP, ...
      long long j = warp - 1;
      int buf = (warp - 1) % NT, in = 0;
      // the whole rollout, or segment after segment
      for (long long seg = SEG ? (Tn + k - 1) / k - 1 : 0; seg >= 0; --seg) {
        const long long t0 = SEG ? seg * k : 0, t1 = SEG && t0 + k < Tn ? t0 + k : Tn;
        bool mine = false;  // SEG: this warp replays the segment (its tape is then free)
        if (SEG) {
          mine = j == Tn - t1;
          if (NP > 1) producers_sync(NT, NP);
          if (mine) {
            if (j >= NT) pipe_sync(1 + NT + buf);
            replay(sys_of_buf(buf), seg, t0, t1);
          }
          if (NP > 1) producers_sync(NT, NP);
        }
        if (ONCHIP) {
          if (act && Tn - 1 - j >= t0) fetch(Tn - 1 - j, t0, in);
          cp_commit();
        }
        for (; Tn - 1 - j >= t0; j += NP, in ^= 1) {
          const long long t = Tn - 1 - j;
          if (ONCHIP) {
            if (act && t - NP >= t0) fetch(t - NP, t0, in ^ 1);
            cp_commit();
            cp_wait_all_but_newest();
          } else if (act && t - NP >= t0 && m.slots > 1) {
            const T* xn = state_of(t - NP, t0);
            for (int d = 0; d < nq; ++d) pf_line(xn + d * B);
            for (int d = 0; d < nv; ++d) pf_line(xn + (nqm + d) * B);
            for (int d = 0; d < nv; ++d) pf_line(tau + ((t - NP) * nvm + d) * B + b);
          }
          __syncwarp();
          if (j >= NT && !mine) pipe_sync(1 + NT + buf);
          mine = false;
          if (ONCHIP ? act : true) {
            const WSys<T, !ONCHIP> sp = sys_of_buf(buf);
            const T* x = ONCHIP ? s_in + in * W * LANES + lane : state_of(t, t0);
            const T* ta = ONCHIP ? x + NX * LANES : tau + t * nvm * B + b;
            const long long st = ONCHIP ? (long long)LANES : B;
            wstep_forward<T, DT, true, false, FR>(sp, Col<const T>{x, st}, Col<const T>{x + nqm * st, st},
                                                  Col<const T>{ta, st}, g, m.dt, m.integ, Col<T>{nullptr, 0},
                                                  Col<T>{nullptr, 0});
          }
          __threadfence_block();
          __syncwarp();
          pipe_arrive(1 + buf);
          buf = (buf + NP) % NT;
        }
      }
      if (ONCHIP) cp_wait_all();
    } else {  // consumer: the adjoint of step after step
      const Col<T> gq{s_state + lane, LANES}, gqd{s_state + nqm * LANES + lane, LANES}, gm{s_gm + lane, LANES};
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
      for (int l = 0; l < nl; ++l) gm[l] = T(0);
      int buf = 0;
      for (long long j = 0; j < Tn; ++j) {
        const long long t = Tn - 1 - j;
        __syncwarp();
        pipe_sync(1 + buf);
        if (ONCHIP ? act : true) {
          const WSys<T, !ONCHIP> sc = sys_of_buf(buf);
          T* gt = gtau + t * nvm * B + b;
          wstep_adjoint<T, DT, FR>(sc, gq, gqd, Col<T>{gt, B}, gm, m.dt, m.integ, g);
          if (act)
            for (int d = nv; d < nvm; ++d) gt[d * B] = T(0);
          if (gtraj) {
            const T* gx = gtraj + t * NX * B + b;
            for (int d = 0; d < nq; ++d) gq[d] += gx[d * B];
            for (int d = 0; d < nv; ++d) gqd[d] += gx[(nqm + d) * B];
          }
        }
        __syncwarp();
        if (j + NT < Tn) pipe_arrive(1 + NT + buf);
        buf = buf + 1 == NT ? 0 : buf + 1;
      }
      if (act) {
        bool ok = true;
        for (int d = 0; d < nq; ++d) ok &= finite_t(gq[d]);
        for (int d = 0; d < nv; ++d) ok &= finite_t(gqd[d]);
        for (int l = 0; l < nl; ++l) ok &= finite_t(gm[l]);
        if (!ok) m.status[b] |= 1;
        for (int d = 0; d < nqm; ++d) gq0[d * B + b] = gq[d];
        for (int d = 0; d < nvm; ++d) gqd0[d * B + b] = gqd[d];
        for (int l = 0; l < nl; ++l) gm_acc[l * B + slot] = gm[l];
      }
    }
    __syncthreads();  // shared memory is reused by the next unit
    if (!m.persistent) break;
    unit = next_unit(m.counter);
  }
}

}  // namespace host
}  // namespace abasim
