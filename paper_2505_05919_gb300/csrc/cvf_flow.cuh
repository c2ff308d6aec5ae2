// cvf_flow.cuh -- what the dataflow sweeps (cvf_flow2.cu, square lattice;
// cvf3_flow.cu, cubic) share: the loads and stores of tagged words, the bounded
// wait, the ring of steps that the warps of a block share with its clerk -- the
// warp that makes the plans, waits for the volume moves and gathers the counts
// -- and the committer beside the volume engine.
#pragma once
#include <cstdint>

#include "cvf_device.cuh"
#include "cvf_host.h"
#include "cvf_lattice.cuh"
#include "cvf_wave.cuh"

namespace cvf {

constexpr unsigned int kFlowSpinLimit = 1u << 21;  // loads of L2: about a second

// The ring of steps a block's warps share.
struct FlowSlot {
  unsigned long long plan;
  int g;
  int ready;             // relative step + 1 once plan and gate are set
  int hb, pairs, moves;  // counts of the warps that finished the step
  int done;              // their number
  uint32_t hist[8];
};

__device__ __forceinline__ uint4 ld_flow4(const uint32_t* p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_flow(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_flow4(uint32_t* p, uint4 v) {
  asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x),
               "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ void st_flow(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bit 31 set iff the word's tag, its top bits, is behind the one needed (`need`:
// the tag in the same bits, those below clear; comparison modulo).
__device__ __forceinline__ uint32_t behind(uint32_t w, uint32_t need) { return w - need; }

// After a warp's `spins` unsuccessful polls (all 32 lanes): true when it has to
// stop, since another wait gave up or this one does.
static __device__ __noinline__ bool flow_stop(unsigned int spins, WaveHdr* H, unsigned int* err) {
  const bool stop = *(volatile unsigned int*)&H->abort != 0u;
  if (__any_sync(0xFFFFFFFFu, stop)) return true;
  if (spins < kFlowSpinLimit) return false;
  if ((threadIdx.x & 31u) == 0u) {
    atomicOr(err, 1u);
    atomicExch(&H->abort, 1u);
  }
  return true;
}

// Adds a warp's counts of a step to its slot and reports the warp done with it
// (three lanes add the three counts at once).
__device__ __forceinline__ void flow_report(FlowSlot& slot, int hb, int pairs, int moves) {
  const unsigned int full = 0xFFFFFFFFu, lane = threadIdx.x & 31u;
  const int a = __reduce_add_sync(full, hb), b = __reduce_add_sync(full, pairs),
            c = __reduce_add_sync(full, moves);
  if (lane < 3u) atomicAdd(&slot.hb + lane, lane == 0u ? a : lane == 1u ? b : c);
  __threadfence_block();
  __syncwarp();
  if (lane == 0u) atomicAdd(&slot.done, 1);
}

// Bounded waiting of a warp that keeps books (the clerk, the committer): `idle`
// counts its rounds without progress; true when it has to stop.
__device__ __forceinline__ bool flow_idle(unsigned int& idle, WaveHdr* H, unsigned int* err) {
  const bool stop = *(volatile unsigned int*)&H->abort != 0u;
  if (__any_sync(0xFFFFFFFFu, stop)) return true;
  if (++idle > kFlowSpinLimit) {
    if ((threadIdx.x & 31u) == 0u) {
      atomicOr(err, 1u);
      atomicExch(&H->abort, 1u);
    }
    return true;
  }
  __nanosleep(32);
  return false;
}

// The clerk (a whole warp of every sweeping block): puts the coming steps' plans
// (make(step)) and gates into the ring, and the counts of the block's warps into
// the launch's slots.  It takes all the steps it can at once, one per lane, so
// that a round trip to L2 and a fence serve several of them.
template <typename PLAN>
__device__ __forceinline__ void flow_clerk(PLAN make, FlowSlot* ring, int warps, WaveHdr* H,
                                           unsigned int* err, long long step0, long long n_steps,
                                           int every) {
  const unsigned int full = 0xFFFFFFFFu;
  const int lane = (int)(threadIdx.x & 31u);
  long long ready = 0, flush = 0;
  unsigned int idle = 0;
  while (flush < n_steps) {
    bool moved = false;
    if (ready < n_steps && ready < flush + kWaveRing - 4) {
      const long long r = ready + lane;
      const unsigned int committed = ld_acquire(&H->committed);
      const WaveMove& m = H->vring[r % kWaveRing];
      const bool ok = lane < kWaveRing && r < n_steps && r < (long long)committed + kWaveRing &&
                      ld_acquire(&m.tag) == (unsigned int)(r + 1);
      const int n = __ffs((int)~__ballot_sync(full, ok)) - 1;
      if (lane < n) {
        FlowSlot& s = ring[r % kWaveRing];
        s.g = *(volatile const int*)&m.g;
        s.plan = make(step0 + r);
        __threadfence_block();
        *(volatile int*)&s.ready = (int)(r + 1);
      }
      ready += n;
      moved = n > 0;
    }
    const long long r = flush + lane;
    volatile FlowSlot* const s = &ring[r % kWaveRing];
    const bool ok = lane < kWaveRing && r < ready && s->done == warps;
    const int n = __ffs((int)~__ballot_sync(full, ok)) - 1;
    if (n > 0) {
      if (lane < n) {
        __threadfence_block();
        WaveAcc* const slot = &H->acc[r % kWaveRing];
        atomicAdd(&slot->hb, (unsigned long long)(long long)s->hb);
        atomicAdd(&slot->pairs, (unsigned long long)(long long)s->pairs);
        atomicAdd(&slot->moves, (unsigned long long)(long long)s->moves);
        if (step_recorded(every, step0 + r)) {
          for (int k = 0; k < 8; ++k) {
            if (s->hist[k]) atomicAdd(&slot->hist[k], (unsigned long long)s->hist[k]);
            s->hist[k] = 0;
          }
        }
        s->hb = 0;
        s->pairs = 0;
        s->moves = 0;
        s->done = 0;
        // the counts before the completion count
        fence_acq_rel_gpu();
        atomicAdd(&slot->done, 1u);
      }
      __syncwarp();
      flush += n;
      moved = true;
    }
    if (moved)
      idle = 0;
    else if (flow_idle(idle, H, err))
      return;
  }
}

// The committer (warp 2 of the engine's block): takes the steps that every
// block has reported, in step order and as many at once as there are, one per
// lane; adds their counts, writes their records, the control block and -- with
// the last step -- the tag that the next call starts from.
__device__ inline void flow_commit(Ctrl* ctl, const VolumeArgs& vol, cvf_obs* ring,
                                   long long ring_cap, int every, WaveHdr* H, int blocks,
                                   uint32_t* tag, uint32_t end_tag, long long step0,
                                   long long n_steps, unsigned int* err) {
  const unsigned int full = 0xFFFFFFFFu;
  const int lane = (int)(threadIdx.x & 31u);
  volatile Ctrl* c = ctl;
  long long n_hb_raw = c->n_hb_raw, n_coop = c->n_coop, acc_sigma = c->acc_sigma,
            acc_volume = c->acc_volume, head = c->ring_head;
  unsigned int idle = 0;
  for (long long next = 0; next < n_steps;) {
    const long long r = next + lane;
    WaveAcc* const slot = &H->acc[r % kWaveRing];
    const bool ok = lane < kWaveRing && r < n_steps &&
                    ld_acquire(&slot->done) == (unsigned int)blocks;
    const int n = __ffs((int)~__ballot_sync(full, ok)) - 1;
    if (n == 0) {
      if (flow_idle(idle, H, err)) return;
      continue;
    }
    idle = 0;
    volatile WaveAcc* const a = slot;
    volatile const WaveMove* const m = &H->vring[r % kWaveRing];
    Ctrl s;
    long long hb = 0, pairs = 0, moves = 0, volume = 0;
    if (lane < n) {
      hb = (long long)a->hb;
      pairs = (long long)a->pairs;
      moves = (long long)a->moves;
      volume = m->acc;
      s.V_iso = m->V;
      s.u_cell = m->u;
      s.g = m->g;
    }
#pragma unroll
    for (int o = 1; o < kWaveRing; o <<= 1) {  // sums over the steps up to the lane's
      const long long x = __shfl_up_sync(full, hb, o), y = __shfl_up_sync(full, pairs, o),
                      z = __shfl_up_sync(full, moves, o), v = __shfl_up_sync(full, volume, o);
      if (lane >= o) {
        hb += x;
        pairs += y;
        moves += z;
        volume += v;
      }
    }
    s.n_hb_raw = n_hb_raw + hb;
    s.n_coop = n_coop + pairs;
    s.acc_sigma = acc_sigma + moves;
    s.acc_volume = acc_volume + volume;
    s.sweep = step0 + r + 1;
    const bool rec = lane < n && step_recorded(every, step0 + r);
    const unsigned int recorded = __ballot_sync(full, rec);
    if (rec) {
      s.error = c->error;
      for (int k = 0; k < 8; ++k) {
        s.hist[k] = (long long)a->hist[k];
        a->hist[k] = 0;
        if ((recorded >> lane) == 1u) c->hist[k] = s.hist[k];  // the last record of the round
      }
      ring[(head + __popc(recorded & ((1u << lane) - 1u))) % ring_cap] = make_obs(vol, &s);
    }
    if (lane < n) {
      a->hb = 0;
      a->pairs = 0;
      a->moves = 0;
      a->done = 0;
    }
    head += __popc(recorded);
    if (lane == n - 1) {
      c->n_hb_raw = s.n_hb_raw;
      c->n_coop = s.n_coop;
      c->acc_sigma = s.acc_sigma;
      c->V_iso = s.V_iso;
      c->u_cell = s.u_cell;
      c->g = s.g;
      c->acc_volume = s.acc_volume;
      c->sweep = s.sweep;
      c->ring_head = head;
      // every block has finished the call's last step (and read the tag and
      // the step count that it started from)
      if (next + n == n_steps) *tag = end_tag;
    }
    n_hb_raw = __shfl_sync(full, s.n_hb_raw, n - 1);
    n_coop = __shfl_sync(full, s.n_coop, n - 1);
    acc_sigma = __shfl_sync(full, s.acc_sigma, n - 1);
    acc_volume = __shfl_sync(full, s.acc_volume, n - 1);
    next += n;
    __syncwarp();
    if (lane == 0) {
      fence_acq_rel_gpu();
      st_relaxed_u32(&H->committed, (unsigned int)next);
    }
  }
}

// Block 0 of a dataflow launch: the volume engine (warps 0 and 1) and the
// committer (warp 2), on an SM of their own; V is shared memory for the
// parameters.
template <typename ARGS>
__device__ __forceinline__ void flow_books(const ARGS& A, VolumeArgs& V, WaveHdr* H, int blocks,
                                           uint32_t* tag, uint32_t end_tag, long long step0,
                                           long long n_steps, int every, unsigned int* err) {
  stage_volume_args(&V, A.vol);
  __syncthreads();
  if (threadIdx.x < 64)
    wave_engine(A.ctrl, V, A.keys, H, step0, n_steps, err);
  else if (threadIdx.x < 96)
    flow_commit(A.ctrl, V, A.ring, A.ring_cap, every, H, blocks, tag, end_tag, step0, n_steps, err);
  if (threadIdx.x >= 96) return;
  // every clerk has reported the last step and looks at the header no more: it is
  // left as the next launch wants it (an abandoned launch leaves it as it is)
  asm volatile("bar.sync 6, 96;" ::: "memory");
  if (*(volatile unsigned int*)&H->abort) return;
  uint4* const words = reinterpret_cast<uint4*>(H);
  for (int i = threadIdx.x; i < (int)(sizeof(WaveHdr) / 16); i += 96)
    words[i] = make_uint4(0u, 0u, 0u, 0u);
}

// The blocks of `fn` that fit the GPU at once.
inline int flow_resident_blocks(const void* fn, int threads) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, 0) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * sm_count();
}

// The threads of a block of `fn` that sweeps `share` items (a multiple of 32),
// one a thread, of at most `most` threads with the clerk's warp: without those
// that have no item (but never fewer than the three warps of the books), where
// that lets another lattice's launch run beside it.  us per step and lattice of 8
// lattices of 130^2 on streams of their own 0.39 against 1.90 with whole blocks,
// 8 of 258^2 1.06 / 1.95, 4 cubes of 32^3 2.3 / 4.0; one alone as before (258^2
// 1.9, 32^3 4.0).
inline int flow_block(const void* fn, long long share, int most) {
  const int threads = (int)(share < 64 ? 64 : share) + 32;
  return threads < most && flow_resident_blocks(fn, threads) >= 2 * sm_count() ? threads : most;
}

}  // namespace cvf
