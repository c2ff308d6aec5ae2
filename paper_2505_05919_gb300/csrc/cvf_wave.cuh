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

// ---------------------------------------------------------------------------
// The volume engine (Sec. II.B step 1), run by the first two warps of one
// block: the move of every step of a call of n_steps, and of the first step of
// the next one, published in the ring while at most kWaveRing steps are ahead
// of the commits.  While no proposal would change the gate, a move follows from
// the volume after the move before it and the step's draws alone, so a pass
// decides kEngDepth steps at once over the tree of outcomes: node i (heap
// order, lane i) is the move of step t0 + depth(i) from the state that the
// accept / reject outcomes on its path lead to.  An FP64 instruction occupies
// the pipe for a whole warp whatever the number of active lanes, so a pass
// costs about what one decision costs (step by step 64^2 would take the 2 to 4
// us of a decision per step).  Each node runs the IEEE operations of
// volume_decide_pair in the same order, so every move equals the step-by-step
// chain's.  A proposal that would change the gate ends the walk; it waits for
// the commit of the step before and is decided with its bonds.  sV is a shared
// copy of the parameters; a wait that gives up sets *err.
// ---------------------------------------------------------------------------
constexpr int kWaveTree = 5;  // steps per pass: 31 nodes

struct WaveTree {
  double log_ratio[32];  // N log(V'/V) of the nodes, from warp 1
  double exchange;       // volume_decide_pair's
  double V, u;           // the state after the last move decided
  int g, acc;
  int flip;              // the next move would change the gate
  int settled;           // steps the pass decided
  int go;
};

// The number of shells inside the cutoff at v, from a guess: the test holds for
// a prefix of the ascending shells, so a guess is moved to the prefix's end.
__device__ __forceinline__ int lj_shells_near(const VolumeArgs& V, double v, int k) {
  const bool cubic = V.dim == 3;
  auto inside = [&](int i) {
    const double key = cubic ? (V.shell_d2[i] * v) * v : V.shell_d2[i] * v;
    return key < V.cutoff2;
  };
  while (k < V.nshell && inside(k)) ++k;
  while (k > 0 && !inside(k - 1)) --k;
  return k;
}

__device__ inline void wave_engine(Ctrl* ctl, const VolumeArgs& sV, const RoundKeys& keys,
                                   WaveHdr* H, long long step0, long long n_steps,
                                   unsigned int* err) {
  __shared__ WaveTree T;
  const unsigned int full = 0xFFFFFFFFu;
  const int role = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31u);
  const int n1 = lane + 1;       // 1-based heap index: children 2 n1 (reject), 2 n1 + 1 (accept)
  const int d = 31 - __clz(n1);  // depth (lane 31: below the tree, not used)
  const double Nd = (double)sV.N;
  volatile Ctrl* c = ctl;
  if (threadIdx.x == 0) {
    VolumeResult cur;
    cur.V = T.V = c->next_V;
    cur.u = T.u = c->next_u;
    cur.g = T.g = c->next_g;
    cur.accepted = T.acc = c->next_acc;
    T.flip = 0;
    wave_publish(H, 0, cur);
  }
  engine_sync();
  // one thread: waits until the ring has room for the move of relative step r (a
  // step more than kWaveRing behind it is committed); `seen` is what it last saw
  unsigned int seen = 0;
  auto room = [&](long long r) {
    const long long need = r - kWaveRing + 1;
    if (need <= (long long)seen) return true;
    if (!wave_wait_geq(&H->committed, (unsigned int)need, H, err)) return false;
    seen = ld_acquire(&H->committed);
    return true;
  };
  int shells = 0;  // of the last pass's root, the guess of the next
  for (long long r = 1; r <= n_steps;) {
    const double bV = T.V, bu = T.u;
    const int bg = T.g;
    const long long t0 = step0 + r;
    if (T.flip || !sV.volume_moves) {
      // the gate would change: decide the move with the bonds after step r - 1
      // (without volume moves every decision keeps the state)
      if (threadIdx.x == 0)
        T.go = (!T.flip || wave_wait_geq(&H->committed, (unsigned int)r, H, err)) ? 1 : 0;
      engine_sync();
      if (!T.go) return;
      VolumeResult res;
      volume_decide_pair<3>(role, sV, t0, bV, bu, bg, T.flip ? c->n_hb_raw : 0, keys, &res,
                            &T.exchange);
      engine_sync();  // both warps have read T
      if (threadIdx.x == 0) {  // res is valid in role 0's lanes
        T.V = res.V;
        T.u = res.u;
        T.g = res.g;
        T.acc = res.accepted;
        T.flip = 0;
        T.go = 1;
        if (r < n_steps) {  // the next call's first move stays in T
          T.go = room(r) ? 1 : 0;
          if (T.go) wave_publish(H, r, res);
        }
      }
      engine_sync();
      if (!T.go) return;
      ++r;
      continue;
    }
    const long long st = t0 + d;
    const Words4 w = philox(kCellVolume, (uint32_t)((unsigned long long)st & 0xFFFFFFFFu),
                            (uint32_t)((unsigned long long)st >> 32), kTagVolume, keys);
    const double u1 = u53(w.x, w.y), u2 = u53(w.z, w.w);
    const double dV = (2.0 * u1 - 1.0) * sV.dV_max;
    // the volume before the node's move: the accepted moves on its path, added
    // in step order (lane 2^j - 1 holds the draw of depth j)
    double Vo = bV;
#pragma unroll
    for (int j = 0; j < kWaveTree; ++j) {
      const double dVj = __shfl_sync(full, dV, (1 << j) - 1);
      if (j < d && ((n1 >> (d - 1 - j)) & 1)) Vo = Vo + dVj;
    }
    const double Vn = Vo + dV;
    if (role == 1) {
      T.log_ratio[lane] = Nd * log(Vn / Vo);
      engine_sync();  // the logs are there
      engine_sync();  // the pass is settled
    } else {
      const double vn = Vn / Nd;
      const bool hard = vn < 1.0;
      const int g_new = (vn < 2.0) ? 1 : 0;
      const int k = lj_shells_near(sV, vn, shells);
      shells = __shfl_sync(full, k, 0);
      const double un = lj_energy_at(sV, vn, k);
      // the energy before the move: that of the last accepted move on the path
      // (its lane), else the root's
      int src = -1;
#pragma unroll
      for (int j = 0; j < kWaveTree; ++j)
        if (j < d && ((n1 >> (d - 1 - j)) & 1)) src = (n1 >> (d - j)) - 1;
      const double uo_lane = __shfl_sync(full, un, src < 0 ? lane : src);
      const double uo = (src < 0) ? bu : uo_lane;
      const double J_eff = sV.J - sV.P * sV.v_HB;
      const double du = un - uo;
      const double t1 = Nd * du;
      const double t2 = sV.P * dV;
      const double t3 = ((double)(g_new - bg) * J_eff) * (double)0;
      const double dH = (t1 + t2) - t3;
      const double q = -dH / sV.kT;
      engine_sync();  // the logs are there
      const double arg = q + T.log_ratio[lane];
      const bool met = u2 < exp(arg);
      // walk the tree along the outcomes; every lane takes the same path
      const bool node = lane < 31;
      const bool flip = !hard && g_new != bg;
      const unsigned int A = __ballot_sync(full, node && !hard && !flip && met);
      const unsigned int U = __ballot_sync(full, node && flip);
      double Vc = bV, uc = bu, myV = bV, myu = bu;
      int nn = 1, j = 0, ac = 0, mya = 0;
      for (; j < kWaveTree && r + j <= n_steps; ++j) {
        const int i = nn - 1;
        if ((U >> i) & 1u) break;
        ac = (int)((A >> i) & 1u);
        const double Vi = __shfl_sync(full, Vn, i), ui = __shfl_sync(full, un, i);
        if (ac) {
          Vc = Vi;
          uc = ui;
        }
        if (lane == j) {  // lane j publishes the move of relative step r + j
          myV = Vc;
          myu = uc;
          mya = ac;
        }
        nn = 2 * nn + ac;
      }
      // the pass's moves behind one fence (a release for each, and a look at the
      // commits before each, held every small lattice at 1.5 us per step)
      const int n = (int)min((long long)j, n_steps - r);
      bool go = true;
      if (lane == 0 && n > 0) go = room(r + n - 1);
      go = __shfl_sync(full, go ? 1 : 0, 0) != 0;
      WaveMove& m = H->vring[(r + lane) % kWaveRing];
      if (go && lane < n) {
        volatile WaveMove* vm = &m;
        vm->V = myV;
        vm->u = myu;
        vm->g = bg;
        vm->acc = mya;
      }
      __syncwarp();
      fence_acq_rel_gpu();
      if (go && lane < n) st_relaxed_u32(&m.tag, (unsigned int)(r + lane + 1));
      if (lane == 0) {
        T.V = Vc;
        T.u = uc;
        if (j > 0) T.acc = ac;
        T.flip = (j < kWaveTree && r + j <= n_steps && ((U >> (nn - 1)) & 1u)) ? 1 : 0;
        T.settled = j;
        T.go = go ? 1 : 0;
      }
      engine_sync();  // the pass is settled
    }
    if (!T.go) return;
    r += T.settled;
  }
  engine_sync();
  if (threadIdx.x == 0) {
    c->next_V = T.V;
    c->next_u = T.u;
    c->next_g = T.g;
    c->next_acc = T.acc;
    c->ahead_state = 0;
  }
}

}  // namespace cvf
