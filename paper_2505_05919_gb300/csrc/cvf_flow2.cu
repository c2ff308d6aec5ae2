// cvf_flow2.cu -- the MC steps of one square lattice as a single persistent,
// cooperative launch per call in which every word carries its own progress
// (dataflow; cvf3_flow.cu is the cubic one and says why it is sound).
//
// Checkerboard (k_flow2).  A thread owns V vertically adjacent words (two cells
// each, one of either colour) of a strip of V rows, in registers for the whole
// call, and writes them to a copy of the lattice after every colour.  The spare
// bits 3 and 7 of a cell there hold the number of steps it has finished, modulo
// 4.  A colour-0 cell of step r needs its four neighbours after r steps, a
// colour-1 cell after r + 1, and since the neighbours wait for it in turn, they
// have never done more: a thread loads the words its colour reads until the
// two bits say so.  Nothing it overwrites is still needed, for the same reason.
// A call first writes the lattice into the copy with the next number after the
// one the last call ended with (word 0 of the copy), so no cell of it can be
// taken for a later one; the words after the last step go to the lattice.
//
// Layered schedule (k_flow2_layer).  As the cubic sweep: a segment of the arm
// order at a time (layer_plan), one 32-bit word per cell in the copy with a
// 16-bit count of finished parts above the cell, four cells of a row per thread
// and group.
//
// What bounds them: the chain of a part -- store, the neighbour's load of it
// (0.27 to 0.5 us between SMs), the four arm updates -- up to about 512^2, the
// instructions of the cells beyond (the launches and waits that it replaces
// took 2.7 us per step at 64^2, 8.2 at 258^2, 7.3 at 512^2 and 11.9 at 1024^2;
// now 1.3, 1.9, 2.7 and 7.4).  The draws of a part are made before its first
// load.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstring>

#include "cvf_fastdiv.cuh"
#include "cvf_flow.cuh"
#include "cvf_flow2.cuh"
#include "cvf_host.h"
#include "cvf_lattice.cuh"
#include "cvf_tile.cuh"

namespace cvf {
namespace {

// Up to this many rows a thread the draws of a part are made before its first load
// (they are the work there is while the neighbours' words come: 900^2 6.0 us per
// step, 6.3 without; 1024^2 7.5 and 7.7); the draws of eight rows do not fit the
// registers.  Nor do two words per update for four rows (152 bytes of spill stores
// with 736 threads, 388 with 992): there 900^2 takes 8.3 us per step and 1024^2
// 10.6, and 7.8 and 9.6 with the draws made after the loads.
constexpr int kAheadRows = 4;
// From this many rows on a warp rests between two looks at its neighbours' words:
// the looks take instructions from the warps that sweep (ns; 1536^2 18.3 us per
// step without, 17.7 with 100, 17.0 with 300; 1024^2 7.39 and 7.33).
constexpr int kRestRows = 4;
constexpr unsigned int kRestNs = 300;
constexpr int kFlow2Head = 32;  // words before the copy's cells (word 0: the tag)

// Tables of both gates and the ring of steps.
struct Flow2Smem {
  Tables2 Tb[2];
  FlowSlot ring[kWaveRing];
};
// A block's shared memory: a sweeping block's, or the books' copy of the
// parameters.
union Flow2Block {
  Flow2Smem sweep;
  VolumeArgs vol;
};

template <typename SMEM>
__device__ __forceinline__ void flow2_setup(SMEM& S, const LatticeArgs& A, int threads) {
  for (int g = 0; g < 2; ++g) {
    fill_rows2(S.Tb[g], A.table24, g, threads);
    fill_prop2(S.Tb[g], A.q);
  }
  uint32_t* ring = reinterpret_cast<uint32_t*>(S.ring);
  for (int i = threadIdx.x; i < (int)(sizeof(S.ring) / 4); i += threads) ring[i] = 0u;
}

// Waits (a whole warp) until the clerk has step rel ready; false to stop.
__device__ __forceinline__ bool flow_ready(const FlowSlot& slot, long long rel, WaveHdr* H,
                                           unsigned int* err) {
  unsigned int spins = 0;
  while (!__all_sync(0xFFFFFFFFu, *(const volatile int*)&slot.ready == (int)(rel + 1))) {
    if ((++spins & 1023u) == 0u && flow_stop(spins >> 6, H, err)) return false;
  }
  __threadfence_block();
  return true;
}

// A warp's counts of a step (and N_q' in the 16-bit lanes v, v + 4 of h[v])
// into its slot.  MANY: the warp may have counted more than the 65535 arms of one
// state that the lanes of its sum hold, so the two are summed apart.
template <bool MANY = false>
__device__ __forceinline__ void flow_report2(FlowSlot& slot, const TileCounts& cnt, bool rec,
                                             const uint32_t h[4]) {
  if (rec) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      uint32_t low, high;
      if (MANY) {
        low = __reduce_add_sync(0xFFFFFFFFu, h[v] & 0xFFFFu);
        high = __reduce_add_sync(0xFFFFFFFFu, h[v] >> 16);
      } else {
        const uint32_t lanes = __reduce_add_sync(0xFFFFFFFFu, h[v]);
        low = lanes & 0xFFFFu;
        high = lanes >> 16;
      }
      if ((threadIdx.x & 31u) == 0u) {
        if (low) atomicAdd(&slot.hist[v], low);
        if (high) atomicAdd(&slot.hist[v + 4], high);
      }
    }
  }
  flow_report(slot, cnt.dhb(), cnt.dc(), (int)cnt.nacc);
}

// The two spare bits of both cells of a word for t finished steps (of the low
// cell, the high cell).
__device__ __forceinline__ uint32_t tag_bits(uint32_t t_low, uint32_t t_high) {
  return ((t_low & 1u) << 3) | ((t_low & 2u) << 6) | ((t_high & 1u) << 19) | ((t_high & 2u) << 22);
}

// The Philox words of a cell's draws, before they are split.
template <int RNG_WORDS>
struct CellWords {
  Words4 u, p;  // p: two words per update only
};
template <int RNG_WORDS>
__device__ __forceinline__ CellWords<RNG_WORDS> cell_words(uint32_t c, const StepDraw& sd,
                                                           const RoundKeys& K) {
  CellWords<RNG_WORDS> w;
  w.u = philox_cell(c, sd.acc, K);
  w.p = (RNG_WORDS == 2) ? philox_cell(c, sd.prop, K) : w.u;
  return w;
}

// A block of a lattice's launch: the books (b < 0) or block b of `blocks` that
// sweep.
template <int RNG_WORDS, bool CMP64, int V>
__device__ __forceinline__ void flow2_strips(Flow2Block& U, const LatticeArgs& A,
                                             const Flow2Geom& G, WaveHdr* H, uint32_t* copy,
                                             long long n_steps, int every, int b, int blocks,
                                             unsigned int* err) {
  constexpr bool kAhead = V <= kAheadRows;  // the draws of a part are made before its loads
  const int sweepers = (int)blockDim.x - 32;  // threads; the last warp is the clerk
  Ctrl* const ctl = A.ctrl;
  // the committed step count and the copy's tag: neither changes before every
  // block has taken part in the first (last) step
  const long long step0 = *(volatile long long*)&ctl->sweep;
  const uint32_t tag0 = *(volatile uint32_t*)copy + 1u;
  if (b < 0) {
    flow_books(A, U.vol, H, blocks, copy,
               tag0 + (uint32_t)((unsigned long long)n_steps & 0xFFFFFFu), step0, n_steps, every,
               err);
    return;
  }
  Flow2Smem& S = U.sweep;
  uint32_t* const F = copy + kFlow2Head;
  const uint32_t t_lo = (uint32_t)b * G.per_block, t_hi = min(t_lo + G.per_block, G.items);
  const int warps = (int)((t_hi - t_lo + 31u) / 32u);
  flow2_setup(S, A, (int)blockDim.x);
  __syncthreads();
  if ((int)threadIdx.x >= sweepers) {
    flow_clerk([](long long) { return 0ull; }, S.ring, warps, H, err, step0, n_steps, every);
    return;
  }
  if ((int)(threadIdx.x >> 5) >= warps) return;
  const unsigned int full = 0xFFFFFFFFu;
  const bool mine = t_lo + threadIdx.x < t_hi;
  const uint32_t item = min(t_lo + threadIdx.x, t_hi - 1u);  // (a lane without one reads along)
  const uint32_t L = (uint32_t)A.L, Lh = L >> 1, q = A.q;
  const uint32_t strip = fdiv(item, G.div_row), p = item - strip * Lh, y0 = strip * (uint32_t)V;
  const uint32_t h = min((uint32_t)V, L - y0);  // rows (even, but for V = 1)
  const uint32_t up = ((y0 == 0u) ? L - 1u : y0 - 1u) * Lh + p;
  const uint32_t down = ((y0 + h == L) ? 0u : y0 + h) * Lh + p;
  const uint32_t left = (p == 0u) ? Lh - 1u : p - 1u, right = (p + 1u == Lh) ? 0u : p + 1u;
  const uint32_t odd0 = y0 & 1u;  // 0 unless V = 1

  uint32_t w[V];
  {
    const long long N = (long long)L * L;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(A.state + (size_t)(step0 & 1) * N);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      w[k] = 0u;
      if ((uint32_t)k < h && dcheck((y0 + k) * Lh + p < L * Lh, err, kSiteStage)) {
        w[k] = __ldcg(src + (y0 + k) * Lh + p);
        if (mine) st_flow(F + (y0 + k) * Lh + p, w[k] | tag_bits(tag0, tag0));
      }
    }
  }

  for (long long rel = 0; rel < n_steps; ++rel) {
    const long long step = step0 + rel;
    FlowSlot& slot = S.ring[rel % kWaveRing];
    const uint32_t tag = tag0 + (uint32_t)((unsigned long long)rel & 0xFFFFFFu);
    const StepDraw sd = step_draw((uint32_t)((unsigned long long)step & 0xFFFFFFFFu),
                                  (uint32_t)((unsigned long long)step >> 32), A.keys);
    uint32_t pk = 0;
    int g = 0;
#pragma unroll
    for (int colour = 0; colour < 2; ++colour) {
      auto words_of = [&](int k) {
        const uint32_t hi = (odd0 + (uint32_t)(k ^ colour)) & 1u;
        return cell_words<RNG_WORDS>((y0 + k) * L + 2u * p + hi, sd, A.keys);
      };
      CellWords<RNG_WORDS> draw[kAhead ? V : 1];
      if (kAhead) {
#pragma unroll
        for (int k = 0; k < V; ++k) draw[kAhead ? k : 0] = words_of(k);
      }
      if (colour == 0) {
        if (!flow_ready(slot, rel, H, err)) return;
        g = slot.g;
      }
      // what the neighbours' cells (of the other colour) have to show
      const uint32_t need = tag_bits(tag + (uint32_t)colour, tag + (uint32_t)colour);
      // The words beside and above and below the thread's column.  Of two
      // rows one needs the word to the right, whose low cell is the right
      // neighbour of its high cell, the other the word to the left, whose high
      // cell is the left neighbour of its low one; of the words above and below
      // (rows come in twos) one half each: two halves in a register.
      constexpr int kPairs = V / 2;
      uint32_t side[V == 1 ? 1 : kPairs], top = 0u, bottom = 0u;
      for (unsigned int spins = 0;;) {
        uint32_t late = 0u;
        if (V == 1) {
          const uint32_t hi = (odd0 + (uint32_t)colour) & 1u;
          side[0] = ld_flow(F + y0 * Lh + (hi ? right : left));
          late = (side[0] ^ need) & (hi ? 0x88u : 0x880000u);
          top = ld_flow(F + up);
          bottom = ld_flow(F + down);
          late |= ((top ^ need) | (bottom ^ need)) & (hi ? 0x880000u : 0x88u);
        } else {
#pragma unroll
          for (int m = 0; m < kPairs; ++m) {
            side[m] = 0u;
            if ((uint32_t)(2 * m) < h) {
              const uint32_t xr = ld_flow(F + (y0 + 2 * m + 1 - colour) * Lh + right);
              const uint32_t xl = ld_flow(F + (y0 + 2 * m + colour) * Lh + left);
              side[m] = __byte_perm(xr, xl, 0x7610u);
              late |= (side[m] ^ need) & 0x00880088u;
            }
          }
          const uint32_t above = ld_flow(F + up), below = ld_flow(F + down);
          top = colour ? __byte_perm(below, above, 0x7610u) : __byte_perm(above, below, 0x7610u);
          bottom = top;
          late |= (top ^ need) & 0x00880088u;
        }
        if (__all_sync(full, late == 0u)) break;
        if ((++spins & 255u) == 0u && flow_stop(spins, H, err)) return;
        if (V >= kRestRows) __nanosleep(kRestNs);
      }
      if (mine) {
        const Tables2& Tb = S.Tb[g];
#pragma unroll
        for (int k = 0; k < V; ++k) {
          if ((uint32_t)k < h) {
            uint32_t acc[4], kk[4];
            if (!kAhead) draw[0] = words_of(k);
            const CellWords<RNG_WORDS>& d = draw[kAhead ? k : 0];
            split_draws<RNG_WORDS>(d.u, d.p, q, acc, kk);
            const uint32_t sw = side[k / 2];
            const uint32_t ym = (k == 0) ? top : w[(k > 0) ? k - 1 : 0];
            const uint32_t yp = ((uint32_t)k + 1u == h) ? bottom : w[(k + 1 < V) ? k + 1 : 0];
            const int hi = (V == 1) ? (int)((odd0 + (uint32_t)colour) & 1u) : ((k ^ colour) & 1);
            const uint32_t cell =
                (V == 1) ? update_cell<CMP64>(w[k], sw, sw, ym, yp, hi, acc, kk, q, Tb, pk)
                : hi ? update_cell<CMP64, 1>(w[k], sw, sw, ym, yp, 1, acc, kk, q, Tb, pk)
                     : update_cell<CMP64, 0>(w[k], sw, sw, ym, yp, 0, acc, kk, q, Tb, pk);
            w[k] = put_cell(w[k], cell, hi != 0);
            const uint32_t other = tag + (uint32_t)colour;  // steps the word's other cell has done
            st_flow(F + (y0 + k) * Lh + p,
                    w[k] | (hi ? tag_bits(other, tag + 1u) : tag_bits(tag + 1u, other)));
          }
        }
      }
    }
    TileCounts cnt{0, 0, 0};
    cnt.add(pk);
    const bool rec = step_recorded(every, step);
    uint32_t hist[4] = {0u, 0u, 0u, 0u};
    if (rec && mine) {
#pragma unroll
      for (int k = 0; k < V; ++k) {
        if ((uint32_t)k < h) {
          const uint32_t n = count_word4(w[k] & 0xFFFFu) + count_word4(w[k] >> 16);  // nibbles <= 8
#pragma unroll
          for (int v = 0; v < 4; ++v) hist[v] += (n >> (4 * v)) & 0x000F000Fu;
        }
      }
    }
    flow_report2(slot, cnt, rec, hist);
  }
  if (mine) {
    const long long N = (long long)L * L;
    uint32_t* dst = reinterpret_cast<uint32_t*>(A.state + (size_t)((step0 + n_steps) & 1) * N);
#pragma unroll
    for (int k = 0; k < V; ++k)
      if ((uint32_t)k < h && dcheck((y0 + k) * Lh + p < L * Lh, err, kSiteTileWrite))
        dst[(y0 + k) * Lh + p] = w[k];
  }
}

template <int RNG_WORDS, bool CMP64, int V, int NT>
__global__ void __launch_bounds__(NT + 32, 1)
    k_flow2(const __grid_constant__ LatticeArgs A, const __grid_constant__ Flow2Geom G, WaveHdr* H,
            uint32_t* copy, long long n_steps, int every) {
  __shared__ Flow2Block U;
  flow2_strips<RNG_WORDS, CMP64, V>(U, A, G, H, copy, n_steps, every, (int)blockIdx.x - 1,
                                    (int)gridDim.x - 1, &A.ctrl->error);
}

// Many lattices, each with blocks of its own and its own number of steps: the
// books of all of them first (on SMs apart while there are as many), then the
// blocks that sweep.
template <int RNG_WORDS, bool CMP64, int V, int NT>
__global__ void __launch_bounds__(NT + 32, 1024 / (NT + 32))
    k_flow2_batch(const __grid_constant__ Flow2Batch B) {
  __shared__ Flow2Block U;
  const Flow2Replica& R = B.item[B.of_block[blockIdx.x]];
  flow2_strips<RNG_WORDS, CMP64, V>(
      U, R.args, R.geom, R.hdr, R.copy, R.n_steps, 0,
      blockIdx.x < (unsigned int)B.n ? -1 : (int)(blockIdx.x - R.first_block), (int)R.blocks,
      B.err);
}

// ---------------------------------------------------------------------------
// Small lattices: the same with one word per thread in the shared memory of a
// thread-block cluster.  A CTA holds a run of words and, on either side, copies
// of the Lh words next to it (a word's neighbours are at most Lh away), which
// their owners write as well: every thread reads its own CTA's memory only, so
// a part costs a store to the next SM and not a load's round trip to it (64^2:
// 1.27 us per step against 1.41 with remote loads and 1.77 through L2).  The
// last CTA of the cluster runs the volume engine and the committer on an SM of
// its own (FP64 instructions hold back the integer multiplies beside them).  The
// words live in shared memory for one call only, so their tags start at 0.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
}
// The address of shared-memory word p in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const uint32_t* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(a)
      : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
  asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

constexpr int kClusterThreads = 576;  // sweeping threads of a CTA
constexpr int kClusterHalo = 64;      // words of a row at most

template <int RNG_WORDS, bool CMP64>
__global__ void __launch_bounds__(kClusterThreads + 32, 1)
    k_flow2_cluster(const __grid_constant__ LatticeArgs A, const __grid_constant__ Flow2Geom G,
                    WaveHdr* H, long long n_steps, int every) {
  __shared__ Flow2Block U;
  __shared__ uint32_t s_word[kClusterThreads + 2 * kClusterHalo];
  __shared__ uint32_t s_no_tag;
  Ctrl* const ctl = A.ctrl;
  unsigned int* const err = &ctl->error;
  const long long step0 = *(volatile long long*)&ctl->sweep;  // (as in k_flow2)
  const uint32_t L = (uint32_t)A.L, Lh = L >> 1, q = A.q;
  const long long N = (long long)L * L;
  const bool books = blockIdx.x == gridDim.x - 1u;
  Flow2Smem& S = U.sweep;
  const uint32_t t_lo = blockIdx.x * G.per_block, t_hi = min(t_lo + G.per_block, G.items);
  const int warps = books ? 0 : (int)((t_hi - t_lo + 31u) / 32u);
  const bool sweeps = threadIdx.x < kClusterThreads && (int)(threadIdx.x >> 5) < warps;
  const bool mine = sweeps && t_lo + threadIdx.x < t_hi;
  const uint32_t item = sweeps ? min(t_lo + threadIdx.x, t_hi - 1u) : 0u;
  const uint32_t y = fdiv(item, G.div_row), p = item - y * Lh;
  // the CTA's words lie at s_word[Lh], those before and after them around
  const int cnt = (int)(t_hi - t_lo), W = (int)G.items;
  auto word_of = [&](uint32_t i) -> volatile uint32_t* {
    int d = (int)i - (int)t_lo;
    if (d < 0 || d >= cnt) {
      const int before = (d < 0) ? d : d - W;
      d = (before >= -(int)Lh) ? before : (d < 0) ? d + W : d;
    }
    if (!dcheck(d >= -(int)Lh && d < cnt + (int)Lh, err, kSiteResident2)) d = 0;
    return s_word + (int)Lh + d;
  };
  volatile uint32_t *own = s_word, *up = s_word, *down = s_word, *left = s_word, *right = s_word;
  uint32_t to_prev = 0u, to_next = 0u;  // the word's copies in the CTAs beside this one
  if (sweeps) {
    own = word_of(item);
    up = word_of(((y == 0u) ? L - 1u : y - 1u) * Lh + p);
    down = word_of(((y + 1u == L) ? 0u : y + 1u) * Lh + p);
    left = word_of(y * Lh + ((p == 0u) ? Lh - 1u : p - 1u));
    right = word_of(y * Lh + ((p + 1u == Lh) ? 0u : p + 1u));
    const uint32_t n = gridDim.x - 1u;  // CTAs with words
    if (n > 1u && mine) {
      const uint32_t prev = (blockIdx.x == 0u) ? n - 1u : blockIdx.x - 1u;
      const uint32_t next = (blockIdx.x + 1u == n) ? 0u : blockIdx.x + 1u;
      const uint32_t prev_cnt = min(G.per_block, G.items - prev * G.per_block);
      if (item - t_lo < Lh) to_prev = cluster_addr(s_word + Lh + prev_cnt + (item - t_lo), prev);
      if (t_hi - item <= Lh) to_next = cluster_addr(s_word + Lh - (t_hi - item), next);
    }
  }
  auto put = [&](uint32_t v) {
    *own = v;
    if (to_prev) st_cluster(to_prev, v);
    if (to_next) st_cluster(to_next, v);
  };
  uint32_t w = 0u;
  if (sweeps && dcheck(item < L * Lh, err, kSiteResident2))
    w = __ldcg(reinterpret_cast<const uint32_t*>(A.state + (size_t)(step0 & 1) * N) + item);
  if (!books) flow2_setup(S, A, kClusterThreads + 32);
  cluster_sync_all();  // every CTA runs
  if (mine) put(w);
  __syncthreads();
  cluster_sync_all();  // and every word is in place

  auto sweep = [&]() {
    const unsigned int full = 0xFFFFFFFFu;
    for (long long rel = 0; rel < n_steps; ++rel) {
      const long long step = step0 + rel;
      FlowSlot& slot = S.ring[rel % kWaveRing];
      const uint32_t tag = (uint32_t)((unsigned long long)rel & 0xFFFFFFu);
      const StepDraw sd = step_draw((uint32_t)((unsigned long long)step & 0xFFFFFFFFu),
                                    (uint32_t)((unsigned long long)step >> 32), A.keys);
      uint32_t pk = 0;
      int g = 0;
#pragma unroll
      for (int colour = 0; colour < 2; ++colour) {
        const uint32_t hi = (y + (uint32_t)colour) & 1u;
        const CellWords<RNG_WORDS> draw = cell_words<RNG_WORDS>(y * L + 2u * p + hi, sd, A.keys);
        uint32_t acc[4], kk[4];
        split_draws<RNG_WORDS>(draw.u, draw.p, q, acc, kk);
        if (colour == 0) {
          if (!flow_ready(slot, rel, H, err)) return;
          g = slot.g;
        }
        const uint32_t need = tag_bits(tag + (uint32_t)colour, tag + (uint32_t)colour);
        const uint32_t vertical = hi ? 0x880000u : 0x88u, across = hi ? 0x88u : 0x880000u;
        uint32_t side, top, bottom;
        for (unsigned int spins = 0;;) {
          side = *(hi ? right : left);
          top = *up;
          bottom = *down;
          const uint32_t late =
              ((side ^ need) & across) | (((top ^ need) | (bottom ^ need)) & vertical);
          if (__all_sync(full, late == 0u)) break;
          if ((++spins & 1023u) == 0u && flow_stop(spins >> 2, H, err)) return;
        }
        if (mine) {
          const uint32_t cell = update_cell<CMP64>(w, side, side, top, bottom, (int)hi, acc, kk, q,
                                                   S.Tb[g], pk);
          w = put_cell(w, cell, hi != 0u);
          const uint32_t other = tag + (uint32_t)colour;
          put(w | (hi ? tag_bits(other, tag + 1u) : tag_bits(tag + 1u, other)));
        }
      }
      TileCounts cnt{0, 0, 0};
      cnt.add(pk);
      const bool rec = step_recorded(every, step);
      uint32_t hist[4] = {0u, 0u, 0u, 0u};
      if (rec && mine) {
        const uint32_t n = count_word4(w & 0xFFFFu) + count_word4(w >> 16);
#pragma unroll
        for (int v = 0; v < 4; ++v) hist[v] = (n >> (4 * v)) & 0x000F000Fu;
      }
      flow_report2(slot, cnt, rec, hist);
    }
    if (mine && dcheck(item < L * Lh, err, kSiteResident2))
      reinterpret_cast<uint32_t*>(A.state + (size_t)((step0 + n_steps) & 1) * N)[item] = w;
  };
  if (books)
    flow_books(A, U.vol, H, (int)gridDim.x - 1, &s_no_tag, 0u, step0, n_steps, every, err);
  else if (sweeps)
    sweep();
  else if (threadIdx.x >= kClusterThreads)
    flow_clerk([](long long) { return 0ull; }, S.ring, warps, H, err, step0, n_steps, every);
  __syncwarp();
  cluster_sync_all();  // no CTA leaves while another may still read its words
}

// ---------------------------------------------------------------------------
// Layered schedule: the arms of a segment (at most two, no opposite pair) of
// every cell, four cells of a row per group; the tag of a part in the top 16
// bits of a cell's word, a step advancing it by 4.  ONE: one group per thread,
// its words and the step's draws in registers; otherwise the draws are made
// again for every segment.
// ---------------------------------------------------------------------------
template <int RNG_WORDS, bool CMP64, bool ONE, int NT>
__global__ void __launch_bounds__(NT + 32, 1)
    k_flow2_layer(const __grid_constant__ LatticeArgs A, const __grid_constant__ Flow2Geom G,
                  WaveHdr* H, uint32_t* copy, long long n_steps, int every) {
  __shared__ Flow2Block U;
  Ctrl* const ctl = A.ctrl;
  unsigned int* const err = &ctl->error;
  const long long step0 = *(volatile long long*)&ctl->sweep;
  const uint32_t tag0 = *(volatile uint32_t*)copy + 4u;
  if (blockIdx.x == 0) {
    flow_books(A, U.vol, H, (int)gridDim.x - 1, copy,
               tag0 + 4u * (uint32_t)((unsigned long long)n_steps & 0xFFFFFFu), step0, n_steps,
               every, err);
    return;
  }
  Flow2Smem& S = U.sweep;
  uint32_t* const F = copy + kFlow2Head;
  const uint32_t t_lo = (blockIdx.x - 1u) * G.per_block, t_hi = min(t_lo + G.per_block, G.items);
  // as many groups for every warp, as in the cubic sweep
  // sweeping threads; the warp after them is the clerk
  const uint32_t sweepers = ONE ? blockDim.x - 32u : (uint32_t)NT;
  const uint32_t rounds = (G.per_block + sweepers - 1u) / sweepers;
  const uint32_t stride = ONE ? (uint32_t)NT : (G.per_block / 32u + rounds - 1u) / rounds * 32u;
  const int warps = (int)min((t_hi - t_lo + 31u) / 32u, stride / 32u);
  flow2_setup(S, A, (int)sweepers + 32);
  __syncthreads();
  if (threadIdx.x >= sweepers) {
    flow_clerk([&](long long s) { return (unsigned long long)layer_plan(s, A.keys); }, S.ring,
               warps, H, err, step0, n_steps, every);
    return;
  }
  if ((int)(threadIdx.x >> 5) >= warps) return;
  const unsigned int full = 0xFFFFFFFFu;
  const uint32_t L = (uint32_t)A.L, q = A.q;
  const uint32_t Gx = G.groups_x, pitch = 4u * Gx;  // groups per row; the copy's row pitch
  const long long N = (long long)L * L;
  const uint32_t first = t_lo + (threadIdx.x & ~31u), lane = threadIdx.x & 31u;

  // a group: its row, its x group and its number of cells (2 in a row's last
  // group when L % 4 == 2)
  struct Group {
    uint32_t y, x, n;
  };
  auto locate = [&](uint32_t i) {
    Group gr;
    gr.y = fdiv(i, G.div_row);
    gr.x = i - gr.y * Gx;
    gr.n = min(4u, L - 4u * gr.x);
    return gr;
  };
  uint32_t w[4] = {0u, 0u, 0u, 0u};  // the group's cells
  CellWords<RNG_WORDS> draw[4];
  {
    const uint16_t* src = A.state + (size_t)(step0 & 1) * N;
    for (uint32_t i0 = first; i0 < t_hi; i0 += stride) {
      const uint32_t i = min(i0 + lane, t_hi - 1u);
      const Group gr = locate(i);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        w[c] = ((uint32_t)c < gr.n) ? __ldcg(src + (size_t)gr.y * L + 4u * gr.x + c) : 0u;
      if (i0 + lane < t_hi)
        st_flow4(F + (size_t)gr.y * pitch + 4u * gr.x,
                 make_uint4(w[0] | (tag0 << 16), w[1] | (tag0 << 16), w[2] | (tag0 << 16),
                            w[3] | (tag0 << 16)));
    }
  }
  uint16_t* const dst = A.state + (size_t)((step0 + n_steps) & 1) * N;

  for (long long rel = 0; rel < n_steps; ++rel) {
    const long long step = step0 + rel;
    FlowSlot& slot = S.ring[rel % kWaveRing];
    const uint32_t tag = tag0 + 4u * (uint32_t)((unsigned long long)rel & 0xFFFFFFu);
    const StepDraw sd = step_draw((uint32_t)((unsigned long long)step & 0xFFFFFFFFu),
                                  (uint32_t)((unsigned long long)step >> 32), A.keys);
    auto draw_group = [&](const Group& gr) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        draw[c] = cell_words<RNG_WORDS>(gr.y * L + 4u * gr.x + (uint32_t)c, sd, A.keys);
    };
    if (ONE) draw_group(locate(min(first + lane, t_hi - 1u)));
    if (!flow_ready(slot, rel, H, err)) return;
    const uint32_t plan = (uint32_t)slot.plan;
    const Tables2& Tb = S.Tb[slot.g];
    const bool rec = step_recorded(every, step);
    const int nseg = 1 + __popc(plan >> 9);
    TileCounts cnt{0, 0, 0};
    // a group adds up to 16 arms of one state to a thread's 16-bit lane, which holds
    // kFlow2LayerGroups of them (449 at kFlowLayerMaxSide on 152 SMs)
    uint32_t hist[4] = {0u, 0u, 0u, 0u};
    for (int j = 0; j < nseg; ++j) {
      const uint32_t arms = layer_segment(plan, j);
      const int na = (int)(arms & 3u);
      const bool last = j == nseg - 1;
      const uint32_t need = (tag + (uint32_t)j) << 16;
      const uint32_t out = (last ? tag + 4u : tag + 1u + (uint32_t)j) << 16;
      for (uint32_t i0 = first; i0 < t_hi; i0 += stride) {
        const bool mine = i0 + lane < t_hi;
        const Group gr = locate(min(i0 + lane, t_hi - 1u));
        uint32_t* const own = F + (size_t)gr.y * pitch + 4u * gr.x;
        if (!ONE) {
          const uint4 v = __ldcg(reinterpret_cast<const uint4*>(own));
          w[0] = v.x & 0xFFFFu;
          w[1] = v.y & 0xFFFFu;
          w[2] = v.z & 0xFFFFu;
          w[3] = v.w & 0xFFFFu;
          draw_group(gr);
        }
        uint32_t nb[2][4];
        for (unsigned int spins = 0;;) {
          uint32_t late = 0u;
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            if (s >= na) continue;
            const uint32_t a = (arms >> (2 + 2 * s)) & 3u;
            if (a >= 2u) {
              const uint32_t yn = (a == 2u) ? (gr.y + 1u == L ? 0u : gr.y + 1u)
                                            : (gr.y == 0u ? L - 1u : gr.y - 1u);
              const uint4 v = ld_flow4(F + (size_t)yn * pitch + 4u * gr.x);
              nb[s][0] = v.x;
              nb[s][1] = v.y;
              nb[s][2] = v.z;
              nb[s][3] = v.w;
              late |= behind(v.x, need) | behind(v.y, need);
              if (gr.n == 4u) late |= behind(v.z, need) | behind(v.w, need);
            } else {
              // the group's own cells serve but for the one at its end: arm a^1
              // does not change in the segment
              const uint32_t x = (a == 0u) ? (4u * gr.x + gr.n == L ? 0u : 4u * gr.x + 4u)
                                           : (gr.x == 0u ? L - 1u : 4u * gr.x - 1u);
              const uint32_t e = ld_flow(F + (size_t)gr.y * pitch + x);
              late |= behind(e, need);
              const bool plus = a == 0u;
              nb[s][0] = plus ? w[1] : e;
              nb[s][1] = plus ? (gr.n == 2u ? e : w[2]) : w[0];
              nb[s][2] = plus ? w[3] : w[1];
              nb[s][3] = plus ? e : w[2];
            }
          }
          if (__all_sync(full, (int32_t)late >= 0)) break;
          if ((++spins & 255u) == 0u && flow_stop(spins, H, err)) return;
        }
        if (mine) {
          uint32_t pk = 0;
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            if (s >= na) continue;
            const uint32_t a = (arms >> (2 + 2 * s)) & 3u;
            auto pass = [&](auto arm_c) {
              constexpr int ARM = decltype(arm_c)::value;
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                if ((uint32_t)c >= gr.n) continue;
                uint32_t acc[4], kk[4];
                split_draws<RNG_WORDS>(draw[c].u, draw[c].p, q, acc, kk);
                const uint32_t n2 = twice(nb[s][c], false);
                const uint32_t p2 = (ARM & 1) ? n2 << 4 : n2 >> 4;  // nibble a^1 to nibble a
                w[c] = update_arm2<CMP64, ARM>(twice(w[c], false), p2, acc[ARM], kk[ARM], q, Tb,
                                               pk) & 0xFFFFu;
              }
            };
            if (a == 0u)
              pass(std::integral_constant<int, 0>{});
            else if (a == 1u)
              pass(std::integral_constant<int, 1>{});
            else if (a == 2u)
              pass(std::integral_constant<int, 2>{});
            else
              pass(std::integral_constant<int, 3>{});
          }
          cnt.add(pk);
          st_flow4(own, make_uint4(w[0] | out, w[1] | out, w[2] | out, w[3] | out));
          if (last && rec) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint32_t n = ((uint32_t)c < gr.n) ? count_word4(w[c]) : 0u;
#pragma unroll
              for (int v = 0; v < 4; ++v) hist[v] += (n >> (4 * v)) & 0x000F000Fu;
            }
          }
          if (last && rel == n_steps - 1) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if ((uint32_t)c < gr.n &&
                  dcheck((long long)gr.y * L + 4u * gr.x + c < N, err, kSiteLayer))
                dst[(size_t)gr.y * L + 4u * gr.x + c] = (uint16_t)w[c];
          }
        }
        __syncwarp();
      }
    }
    flow_report2<!ONE>(slot, cnt, rec, hist);
  }
}

template <int V, int NT>
const void* flow2_kernel(int rng_words, bool cmp64) {
  if (rng_words == 1)
    return cmp64 ? (const void*)k_flow2<1, true, V, NT> : (const void*)k_flow2<1, false, V, NT>;
  return cmp64 ? (const void*)k_flow2<2, true, V, NT> : (const void*)k_flow2<2, false, V, NT>;
}

template <bool ONE, int NT>
const void* flow2_layer_kernel(int rng_words, bool cmp64) {
  if (rng_words == 1)
    return cmp64 ? (const void*)k_flow2_layer<1, true, ONE, NT>
                 : (const void*)k_flow2_layer<1, false, ONE, NT>;
  return cmp64 ? (const void*)k_flow2_layer<2, true, ONE, NT>
               : (const void*)k_flow2_layer<2, false, ONE, NT>;
}

// Adopts the kernel of `form` for `items` spread over the SMs, one item per
// thread (one) or any number, if they fit.
struct Flow2Form {
  int v, threads;
  const void* (*kernel)(int rng_words, bool cmp64);
};
bool adopt(Flow2Plan* P, const Flow2Form& form, int rng_words, bool cmp64, long long items,
           bool one) {
  if (one && items > (long long)(sm_count() - 1) * form.threads) return false;
  const void* const kernel = form.kernel(rng_words, cmp64);
  const long long room =
      std::min(sm_count(), flow_resident_blocks(kernel, form.threads + 32)) - 1;
  if (room < 1 || (one && items > room * form.threads)) return false;
  const long long share = ((items + room - 1) / room + 31) / 32 * 32;
  P->kernel = kernel;
  P->threads = one ? flow_block(kernel, share, form.threads + 32) : form.threads + 32;
  P->geom.items = (uint32_t)items;
  P->geom.per_block = (uint32_t)share;
  P->blocks = (int)((items + share - 1) / share);
  return true;
}

// The strips of the checkerboard sweep, the first that fits: the fewest rows a
// thread, then the fewest threads (the most registers) a block.  us per MC step
// on GB300, with the sides where each ends (151 blocks): one row and 480
// threads (380), 992 (547): 512^2 2.74 against 2.82 with two rows and 480; two
// rows, 736 (667): 640^2 3.38 against 3.61 with 992; 992 (774): 768^2 4.49
// against 5.08 with four and 736; four rows, 736 (943): 896^2 6.0 against 6.35;
// 992 (1094): 1024^2 7.4 against 11.9 with eight rows and 480, which hides too
// little latency.  Eight rows and 736 threads (1332) where the wavefront's tiles
// do not divide the side: 1096^2 10.3 against 12.9 with the wavefront, 1200^2 11.0
// / 14.6, 1300^2 14.0 / 21.5, but 1152^2 12.4 / 12.3 and 1280^2 14.1 / 13.5; with
// two-word draws where rows are not 16-byte aligned, too: 1300^2 19.9 / 25.2, but
// 1120^2 16.6 / 15.4.
const Flow2Form kStrips[] = {{1, 480, flow2_kernel<1, 480>}, {1, 992, flow2_kernel<1, 992>},
                             {2, 736, flow2_kernel<2, 736>}, {2, 992, flow2_kernel<2, 992>},
                             {4, 736, flow2_kernel<4, 736>}, {4, 992, flow2_kernel<4, 992>},
                             {8, 736, flow2_kernel<8, 736>}};
// The layered sweep: one group a thread (512^2 4.3 us per step), or several with
// as many warps as fit (1024^2 14.0 us with 992 threads, 16.4 with 736, 17.3
// with 480; 4096^2 195, 201, 240).
const Flow2Form kLayerOne = {0, 480, flow2_layer_kernel<true, 480>};
const Flow2Form kLayerMany = {0, 992, flow2_layer_kernel<false, 992>};
// Groups of a thread at most: their arms of one state fit its 16-bit counters.
constexpr uint32_t kFlow2LayerGroups = 65535u / 16u;
// The cluster form: at most fifteen CTAs with words (128^2) and one with the
// books; a CTA for every so many words (64^2 1.27 us per step with 64 or 128,
// 1.30 with 256, 1.56 with 544).
constexpr int kClusterCtas = 15, kClusterShare = 128;

const void* cluster_kernel(int rng_words, bool cmp64) {
  if (rng_words == 1)
    return cmp64 ? (const void*)k_flow2_cluster<1, true> : (const void*)k_flow2_cluster<1, false>;
  return cmp64 ? (const void*)k_flow2_cluster<2, true> : (const void*)k_flow2_cluster<2, false>;
}

cudaLaunchConfig_t cluster_config(int ctas, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kClusterThreads + 32);
  cfg.stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = ctas;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Adopts the cluster form if the lattice's words fit one cluster and the GPU can
// place it.
bool adopt_cluster(Flow2Plan* P, int rng_words, bool cmp64, long long words, long long row) {
  if (row > kClusterHalo || words > (long long)kClusterCtas * kClusterThreads) return false;
  // (the last CTA holds a row of words at least: a word then has copies in the
  // CTAs beside its own only)
  long long ctas = std::min<long long>(kClusterCtas, (words + kClusterShare - 1) / kClusterShare);
  long long share = 0;
  for (;; --ctas) {
    share = ((words + ctas - 1) / ctas + 31) / 32 * 32;
    ctas = (words + share - 1) / share;
    if (ctas == 1 || words - (ctas - 1) * share >= row) break;
  }
  if (share > kClusterThreads) return false;
  const void* const kernel = cluster_kernel(rng_words, cmp64);
  const int n = (int)ctas + 1;  // + the books'
  int clusters = 0;
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = cluster_config(n, &attr, nullptr);
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess || clusters < 1) {
    cudaGetLastError();
    return false;
  }
  P->kernel = kernel;
  P->threads = kClusterThreads + 32;
  P->blocks = n - 1;
  P->cluster = true;
  P->geom.items = (uint32_t)words;
  P->geom.per_block = (uint32_t)share;
  P->copy_words = 0;
  return true;
}

}  // namespace

namespace {
template <int V, int NT>
const void* batch_kernel(int rng_words, bool cmp64) {
  if (rng_words == 1)
    return cmp64 ? (const void*)k_flow2_batch<1, true, V, NT>
                 : (const void*)k_flow2_batch<1, false, V, NT>;
  return cmp64 ? (const void*)k_flow2_batch<2, true, V, NT>
               : (const void*)k_flow2_batch<2, false, V, NT>;
}
// Four small blocks per SM for lattices that would leave much of a large one
// empty, or one large one.  (Eight rows would take batches of up to twice the
// cells, but are no faster than the tiled sweep there: 5 of 512^2 18.1 us per step
// against 15.3, 24 of 256^2 16.4 / 16.8, 8 of 512^2 17.7 / 20.3.)
const Flow2Form kBatchForms[kFlow2BatchForms] = {
    {1, 224, batch_kernel<1, 224>}, {1, 992, batch_kernel<1, 992>},
    {2, 224, batch_kernel<2, 224>}, {2, 992, batch_kernel<2, 992>},
    {4, 224, batch_kernel<4, 224>}, {4, 992, batch_kernel<4, 992>}};
long long batch_words(int L) {  // of a copy, in whole 128 bytes
  return ((long long)kFlow2Head + (long long)L * L / 2 + 31) / 32 * 32;
}
// The blocks that sweep a lattice, and the items of each.
void batch_blocks(const Flow2Form& form, int L, Flow2Geom* G, int* blocks) {
  const long long Lh = L / 2, items = Lh * ((L + form.v - 1) / form.v);
  const long long n = (items + form.threads - 1) / form.threads;
  *G = Flow2Geom{};
  G->items = (uint32_t)items;
  G->per_block = (uint32_t)(((items + n - 1) / n + 31) / 32 * 32);
  G->div_row = make_fastdiv((uint32_t)Lh);
  *blocks = (int)((items + G->per_block - 1) / G->per_block);
}
}  // namespace

size_t flow2_batch_scratch() {
  return (size_t)kFlow2BatchMax * sizeof(WaveHdr) + sizeof(uint32_t) * (size_t)kFlow2BatchWords;
}

bool flow2_batch_plan(Flow2Batch* B, const int* sides, int n, int rng_words, bool cmp64,
                      int* slots, int* form) {
  if (n > kFlow2BatchMax) return false;
  long long words = 0;
  for (int i = 0; i < n; ++i) words += batch_words(sides[i]);
  if (words > kFlow2BatchWords) return false;
  Flow2Geom G;
  int own = 0;
  // The form with the least cost, about its step in 0.01 us beyond 1.2 us: the
  // chain of a thread's rows, and what the warps of the SM with the most blocks do
  // (a quarter more where blocks share SMs, and so some of them an SM with a
  // volume engine, whose FP64 instructions hold back the integer multiplies
  // beside them).  us per step on 152 SMs, small blocks / large: 64^2 1.8 / 2.3,
  // 24 of 64^2 2.3 / 2.5, 100 of 64^2 4.8 / do not fit, 24 of 128^2 5.0 / 4.0, 4
  // of 256^2 3.3 (one row a thread), 4.5 (four) / 3.0, 8 of 256^2 5.3 / 4.4, 12 of
  // 256^2 7.3 / 8.7, 4 of 512^2 10.2 / 8.5.
  long long best = LLONG_MAX;
  for (int f = 0; f < kFlow2BatchForms; ++f) {
    const Flow2Form& F = kBatchForms[f];
    if (slots[f] == 0)
      slots[f] = std::min(kFlow2BatchBlocks,
                          flow_resident_blocks(F.kernel(rng_words, cmp64), F.threads + 32));
    long long blocks = n, warps = 0;
    for (int i = 0; i < n && blocks <= slots[f]; ++i) {
      batch_blocks(F, sides[i], &G, &own);
      blocks += own;
      warps = std::max<long long>(warps, G.per_block / 32);
    }
    if (blocks > slots[f]) continue;
    const long long per_sm = (blocks + sm_count() - 1) / sm_count();
    const long long cost = 45 * F.v + per_sm * warps * F.v * (per_sm > 1 ? 5 : 4);
    if (cost < best) {
      best = cost;
      *form = f;
    }
  }
  if (best == LLONG_MAX) return false;
  B->n = n;
  int next = n;
  for (int i = 0; i < n; ++i) {
    batch_blocks(kBatchForms[*form], sides[i], &B->item[i].geom, &own);
    B->item[i].first_block = (uint32_t)next;
    B->item[i].blocks = (uint32_t)own;
    B->of_block[i] = (uint8_t)i;
    std::memset(B->of_block + next, i, (size_t)own);
    next += own;
  }
  return true;
}

cudaError_t launch_flow2_batch(Flow2Batch* B, void* scratch, int rng_words, bool cmp64, int form,
                               cudaStream_t s) {
  WaveHdr* hdr = reinterpret_cast<WaveHdr*>(scratch);
  uint32_t* copy = reinterpret_cast<uint32_t*>(hdr + B->n);
  int blocks = B->n;
  for (int i = 0; i < B->n; ++i) {
    B->item[i].hdr = hdr + i;
    B->item[i].copy = copy;
    copy += batch_words(B->item[i].args.L);
    blocks += (int)B->item[i].blocks;
  }
  const size_t bytes = (size_t)(reinterpret_cast<char*>(copy) - reinterpret_cast<char*>(scratch));
  const cudaError_t e = cudaMemsetAsync(scratch, 0, bytes, s);
  if (e != cudaSuccess) return e;
  void* args[1] = {B};
  const Flow2Form& F = kBatchForms[form];
  return cudaLaunchCooperativeKernel(F.kernel(rng_words, cmp64), dim3(blocks), dim3(F.threads + 32),
                                     args, 0, s);
}

Flow2Plan flow2_plan(int L, int schedule, int rng_words, bool cmp64) {
  Flow2Plan P{};
  if (schedule == CVF_SCHED_LAYERED) {
    const long long gx = (L + 3) / 4, groups = gx * L;
    P.geom.groups_x = (uint32_t)gx;
    P.geom.div_row = make_fastdiv((uint32_t)gx);
    P.copy_words = (size_t)kFlow2Head + 4 * (size_t)groups;
    if (!adopt(&P, kLayerOne, rng_words, cmp64, groups, true) &&
        adopt(&P, kLayerMany, rng_words, cmp64, groups, false) &&
        P.geom.per_block > (uint32_t)kLayerMany.threads * kFlow2LayerGroups)
      P.blocks = 0;  // (a GPU of few SMs)
    return P;
  }
  const long long Lh = L / 2;
  P.geom.div_row = make_fastdiv((uint32_t)Lh);
  if (adopt_cluster(&P, rng_words, cmp64, Lh * L, Lh)) return P;
  P.copy_words = (size_t)kFlow2Head + (size_t)(Lh * L);
  for (const Flow2Form& form : kStrips)
    if ((form.v < 8 || L % (rng_words == 1 ? 128 : 8) != 0) &&
        adopt(&P, form, rng_words, cmp64, Lh * ((L + form.v - 1) / form.v), true)) break;
  return P;
}

cudaError_t launch_flow2(const LatticeArgs& A, const Flow2Plan& P, WaveHdr* H, long long n_steps,
                         int every, cudaStream_t s) {
  if (P.cluster) {
    void* args[5] = {const_cast<LatticeArgs*>(&A), const_cast<Flow2Geom*>(&P.geom), &H, &n_steps,
                     &every};
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(P.blocks + 1, &attr, s);
    return cudaLaunchKernelExC(&cfg, P.kernel, args);
  }
  uint32_t* copy = reinterpret_cast<uint32_t*>(H + 1);
  void* args[6] = {const_cast<LatticeArgs*>(&A), const_cast<Flow2Geom*>(&P.geom), &H, &copy,
                   &n_steps, &every};
  return cudaLaunchCooperativeKernel(P.kernel, dim3(P.blocks + 1), dim3(P.threads), args, 0, s);
}

}  // namespace cvf
