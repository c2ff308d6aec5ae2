// cvf_wave.cuh -- what the persistent sweeps of one lattice (cvf_wave.cu, square;
// cvf3_flow.cu, cubic) share: release / acquire words, the volume engine that
// decides the moves of the coming steps, and the commit of a step.
#pragma once
#include <cstdint>

#include "cvf_device.cuh"
#include "cvf_lattice.cuh"

namespace cvf {

constexpr int kWaveEngineBar = 5;                             // the engine's two warps

__device__ __forceinline__ void st_release_u32(unsigned int* p, unsigned int v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void fence_acq_rel_gpu() {
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
}

__device__ __forceinline__ void st_relaxed_u32(unsigned int* p, unsigned int v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned int atom_add_relaxed_u32(unsigned int* p, unsigned int v) {
  unsigned int old;
  asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v)
               : "memory");
  return old;
}

__device__ __forceinline__ void engine_sync() {
  asm volatile("bar.sync %0, 64;" ::"n"(kWaveEngineBar) : "memory");
}

// Bounded wait of one thread until *flag >= target (or the launch aborts);
// false when it gave up or saw the abort word.
__device__ inline bool wave_wait_geq(const unsigned int* flag, unsigned int target, WaveHdr* H,
                              unsigned int* err) {
  unsigned int used = 0;
  for (;;) {
    if (ld_acquire(flag) >= target) return true;
    if (*(volatile unsigned int*)&H->abort) return false;
    used += 1;
    if (used > kWaitPollLimit) {
      atomicOr(err, 1u);
      atomicExch(&H->abort, 1u);
      return false;
    }
    __nanosleep(128);
  }
}

// Publishes the move of relative step r in its ring slot.
__device__ __forceinline__ void wave_publish(WaveHdr* H, long long r, const VolumeResult& m) {
  WaveMove& w = H->vring[r % kWaveRing];
  volatile WaveMove* vw = &w;
  vw->V = m.V;
  vw->u = m.u;
  vw->g = m.g;
  vw->acc = m.accepted;
  st_release_u32(&w.tag, (unsigned int)(r + 1));
}

// Commit of relative step r (one thread; the previous step is committed):
// finalize_step's bookkeeping with the counts from the step's slot and the
// step's move from the ring.
__device__ inline void wave_commit(Ctrl* ctl, const VolumeArgs& vol, cvf_obs* ring,
                                   long long ring_cap, int every, WaveHdr* H, long long step0,
                                   long long r) {
  volatile Ctrl* c = ctl;
  volatile WaveAcc* a = &H->acc[r % kWaveRing];
  volatile WaveMove* m = &H->vring[r % kWaveRing];
  const long long sweep = step0 + r;
  Ctrl s;
  const bool recorded = (every > 0) && ((sweep + 1) % every == 0);
  s.n_hb_raw = c->n_hb_raw + (long long)a->hb;
  s.n_coop = c->n_coop + (long long)a->pairs;
  s.acc_sigma = c->acc_sigma + (long long)a->moves;
  s.V_iso = m->V;
  s.u_cell = m->u;
  s.g = m->g;
  s.acc_volume = c->acc_volume + m->acc;
  s.sweep = sweep + 1;
  c->n_hb_raw = s.n_hb_raw;
  c->n_coop = s.n_coop;
  c->acc_sigma = s.acc_sigma;
  c->V_iso = s.V_iso;
  c->u_cell = s.u_cell;
  c->g = s.g;
  c->acc_volume = s.acc_volume;
  c->sweep = s.sweep;
  if (recorded) {
    const long long head = c->ring_head;
    s.error = c->error;
    for (int v = 0; v < 8; ++v) {
      s.hist[v] = (long long)a->hist[v];
      c->hist[v] = s.hist[v];
    }
    ring[head % ring_cap] = make_obs(vol, &s);
    c->ring_head = head + 1;
  }
  a->hb = 0;
  a->pairs = 0;
  a->moves = 0;
  for (int v = 0; v < 8; ++v) a->hist[v] = 0;
  a->done = 0;
  st_release_u32(&H->committed, (unsigned int)(r + 1));
}

// The volume engine (Sec. II.B step 1), run by the first two warps of one
// block: the move of every step of a call of n_steps, and of the first step of
// the next one, each from the move before it and published in the ring while
// at most kWaveRing steps are ahead of the commits.  A proposal that would
// change the gate waits for the commit of the step before and is decided with
// its bonds.  sV is a shared copy of the parameters.
__device__ inline void wave_engine(Ctrl* ctl, const VolumeArgs& sV, const RoundKeys& keys,
                                   WaveHdr* H, long long step0, long long n_steps) {
  __shared__ double s_xch;
  __shared__ VolumeResult s_res;
  __shared__ int s_go;
  unsigned int* const err = &ctl->error;
  const int role = (int)(threadIdx.x >> 5);
  volatile Ctrl* c = ctl;
  VolumeResult cur;
  cur.V = c->next_V;
  cur.u = c->next_u;
  cur.g = c->next_g;
  cur.accepted = c->next_acc;
  if (threadIdx.x == 0) wave_publish(H, 0, cur);
  bool alive = true;
  for (long long r = 1; r <= n_steps; ++r) {
    if (threadIdx.x == 0)
      s_go = (r < kWaveRing) ? 1
                             : (wave_wait_geq(&H->committed, (unsigned int)(r - kWaveRing + 1), H,
                                              err) ? 1 : 0);
    engine_sync();
    if (!s_go) {
      alive = false;
      break;
    }
    VolumeResult res;
    const bool ok = volume_decide_pair<3>(role, sV, step0 + r, cur.V, cur.u, cur.g, -1,
                                          keys, &res, &s_xch);
    if (!ok) {
      // the proposal changes the gate: decide it with the bonds after step r - 1
      if (threadIdx.x == 0) s_go = wave_wait_geq(&H->committed, (unsigned int)r, H, err) ? 1 : 0;
      engine_sync();
      if (!s_go) {
        alive = false;
        break;
      }
      const long long nhb = c->n_hb_raw;
      volume_decide_pair<3>(role, sV, step0 + r, cur.V, cur.u, cur.g, nhb, keys, &res,
                            &s_xch);
    }
    if (threadIdx.x == 0) s_res = res;  // valid in role 0's lanes
    engine_sync();
    cur = s_res;
    engine_sync();  // every thread has read s_res before the next write
    if (r < n_steps && threadIdx.x == 0) wave_publish(H, r, cur);
  }
  if (alive && threadIdx.x == 0) {
    c->next_V = cur.V;
    c->next_u = cur.u;
    c->next_g = cur.g;
    c->next_acc = cur.accepted;
    c->ahead_state = 0;
  }
}

}  // namespace cvf
