// cvf3_flow.cu -- the MC steps of one cubic lattice as a single persistent,
// cooperative launch per call in which every word carries its own progress.
//
// A step is a row of parts: the eta moves of the checkerboard cubes (App. A,
// with eta moves), then the two to four segments of arm passes (make_plan).
// Between two parts a cell needs nothing but the words of its neighbours (and
// of its two cubes, a cube those of its eight corners), so no barrier and no
// fence separates them: the sweep works on a copy of the cube in which bits
// 24..31 of every word (spare in the lattice's layout) hold a tag that counts
// the parts the cell has finished, value and tag in one 32-bit access.  A
// thread loads the words that its part reads until their tags say that the
// part before is done in them, computes, and stores its own words with the
// next tag.
//   - What is read is there: the tag says so.  A neighbour that is further on
//     is just as good: arm a^1 of the neighbour in direction a changes only in
//     the pass over a^1, which reads the cell's own word and so waits for it.
//   - What is overwritten has been read, for the same reason: the passes over a
//     and a^1, a cube and its corners wait for each other's words.
// So neighbours are at most about a step apart, and a comparison of the 8-bit
// tags modulo 256 is exact.  Steps advance the tag by 8, the parts inside by
// 1 (the last one completes the eight).  A call starts from the tag that the
// last one left (word 0 of the copy) and first writes every word of the
// lattice into the copy with the next tag, so no barrier is needed there
// either; the words of its last part go to the lattice as well.
//
// The threads of a block share the step's plan, its gate and its counts
// through a ring of kWaveRing steps in shared memory, kept by one more warp
// (the clerk): it makes the plans, waits for the volume moves that block 0
// decides ahead (wave_engine) and gathers the counts of the block's warps; a
// warp of block 0 commits the steps (flow_commit).  So no warp that sweeps
// waits for anything but the words it reads.
//
// All blocks are co-resident (a cooperative launch) and a part waits only for
// earlier parts, so the earliest unfinished part can always run.  Every wait is
// bounded; one that gives up sets the lattice's error bit and the abort word,
// and every warp then stops.
//
// What bounds it: up to about 64^3 the chain of a step, a part's store, the
// reader's load of it (together 0.27 us between SMs of one die, 0.5 us between
// the dies) and one to three arm updates, three to five times; beyond it the
// arm updates.  Where a thread has one group (ONE) its words stay in registers
// and the numbers of a part are drawn before its first load.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "cvf3.cuh"
#include "cvf_flow.cuh"
#include "cvf_host.h"

namespace cvf {
namespace {

// Sweeping threads of a block (one more warp is the clerk), one block per SM:
// with one group per thread as many registers as the three passes of a segment
// like (51^3: 5.6 us per step; 6.5 with 480 threads at 128 registers, 7.3 with
// the proposals made before the wait, which spills), with several groups 480
// threads at 128 (100^3: 22.7 us; 24.1 with 512 at 96 and spills, 24.8 with two
// blocks of 224, 28.6 with 736).
constexpr int kFlowThreadsOne = 224, kFlowThreadsMany = 480;
inline int flow_threads(bool one) { return one ? kFlowThreadsOne : kFlowThreadsMany; }
// A warp with several groups rests between two looks at its neighbours' words,
// which take instructions from the warps that sweep (ns; 100^3 22.8 us per step
// without, 22.1 so; 120^3 35.2 and 34.4; not where rows are no whole groups: 97^3
// 25.7 and 27.0).
constexpr unsigned int kRestNs = 300;
constexpr int kFlowHead = 32;                    // words before the copy's cells (word 0: the tag)
struct FlowSmem {
  Tables3 Tb[2];  // per gate (the proposals in the first)
  unsigned long long eta_thr[2][9];
  uint32_t eta_mask[9];
  uint32_t forbid[8][9];  // eta copies that are 0 at corner j in configuration c
  FlowSlot ring[kWaveRing];
};

// ALIGNED: L % 4 == 0, a group (four consecutive cells) lies in one row and
// its words and its y and z neighbours' are 16-byte vectors; otherwise every
// cell has its own coordinates.  ONE: no thread has more than one group (and
// one cube), whose words stay in its registers.
template <bool ALIGNED, bool CMP64, bool ONE>
__global__ void __launch_bounds__((ONE ? kFlowThreadsOne : kFlowThreadsMany) + 32, 1)
    k_flow3(const __grid_constant__ Args3 A, uint32_t groups_per_block, WaveHdr* H,
            uint32_t* copy, long long n_steps, int every) {
  __shared__ union {
    FlowSmem sweep;
    VolumeArgs vol;  // the engine block's copy of the parameters
  } U;
  Ctrl* const ctl = A.ctrl;
  unsigned int* const err = &ctl->error;
  // the committed step count and the copy's tag: neither changes before every
  // block has taken part in the first (last) step
  const long long step0 = *(volatile long long*)&ctl->sweep;
  const uint32_t tag0 = *(volatile uint32_t*)copy + 8u;
  const uint32_t end_tag = tag0 + 8u * (uint32_t)((unsigned long long)n_steps & 0xFFFFFFu);
  if (blockIdx.x == 0) {
    flow_books(A, U.vol, H, (int)gridDim.x - 1, copy, end_tag, step0, n_steps, every, err);
    return;
  }
  // sweeping threads; the warp after them is the clerk
  const uint32_t sweepers = ONE ? blockDim.x - 32u : (uint32_t)kFlowThreadsMany;
  const int threads = (int)sweepers + 32;
  FlowSmem& S = U.sweep;
  const uint32_t b = blockIdx.x - 1u;
  uint32_t* const F = copy + kFlowHead;             // the cells' words
  uint32_t* const C = F + 4u * (size_t)A.groups;    // the cubes' words
  const uint32_t g_lo = b * groups_per_block, g_hi = min(g_lo + groups_per_block, A.groups);
  const uint32_t g_first = g_lo + threadIdx.x;
  const bool eta_on = A.eta != nullptr;
  // Every warp sweeps as many groups (but for the last ones): a warp with one
  // less would spend that time on loads that wait for the others, which slows
  // them (70^3 without eta moves 22.3 us per step, so 14.0; 97^3 38.1 / 26.2).
  // From four rounds of aligned groups on the idle warps cost more (100^3 19.5
  // us with all of them, 21.9 so).
  const uint32_t rounds = (groups_per_block + sweepers - 1u) / sweepers;
  const uint32_t stride = ONE ? (uint32_t)kFlowThreadsOne  // (no second round)
                          : (ALIGNED && rounds > 3u)
                              ? sweepers
                              : (groups_per_block / 32u + rounds - 1u) / rounds * 32u;
  const int warps = (int)min((g_hi - g_lo + 31u) / 32u, stride / 32u);  // that have a group
  const uint32_t q = A.q;
  for (int g = 0; g < 2; ++g) fill_rows3(S.Tb[g], A.table + g * kRows3, threads);
  fill_prop3(S.Tb[0], q, threads);
  fill_prop3(S.Tb[1], q, threads);
  if (eta_on && threadIdx.x < 18) S.eta_thr[threadIdx.x / 9][threadIdx.x % 9] = A.eta_table[threadIdx.x];
  if (eta_on && threadIdx.x < 9) {
    const uint32_t m = A.masks[threadIdx.x];
    S.eta_mask[threadIdx.x] = pack_edge_mask(m);
    for (int j = 0; j < 8; ++j) {
      uint32_t f = 0u;
      for (int e = 0; e < 12; ++e) {
        const int d = e >> 2, lo = edge_lo(e);
        if (((m >> e) & 1u) && (j == lo || j == (lo | (1 << d))))
          f |= 8u << (4 * (2 * d + (j == lo ? 0 : 1)));
      }
      S.forbid[j][threadIdx.x] = f;
    }
  }
  {
    uint32_t* ring = reinterpret_cast<uint32_t*>(S.ring);
    for (int i = threadIdx.x; i < (int)(sizeof(S.ring) / 4); i += threads) ring[i] = 0u;
  }
  __syncthreads();
  if (threadIdx.x >= sweepers) {
    flow_clerk([&](long long s) { return make_plan(s, A.keys); }, S.ring, warps, H, err, step0,
               n_steps, every);
    return;
  }
  if ((int)(threadIdx.x >> 5) >= warps) return;
  const unsigned int full = 0xFFFFFFFFu;

  // coordinates of a group (ALIGNED: x group, y, z; else x, y, z of each of
  // its cells), ten bits each
  auto coords = [&](uint32_t gi, uint32_t out[4]) {
    if (ALIGNED) {
      const uint32_t row = fdiv(gi, A.div_G);  // y + L z
      const uint32_t z = fdiv(row, A.div_L);
      out[0] = (gi - row * A.G) | ((row - z * A.L) << 10) | (z << 20);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t c = min(4u * gi + (uint32_t)i, A.N - 1u);
        const uint32_t z = fdiv(c, A.div_L2), rem = c - z * A.L2, y = fdiv(rem, A.div_L);
        out[i] = (rem - y * A.L) | (y << 10) | (z << 20);
      }
    }
  };
  auto load_own = [&](uint32_t gi, const uint32_t* from, uint32_t w[4]) {
    if (ALIGNED) {
      const uint4 v = dcheck(4u * gi + 3u < A.N, err, kSitePass3)
                          ? __ldcg(reinterpret_cast<const uint4*>(from + 4u * gi))
                          : make_uint4(0u, 0u, 0u, 0u);
      w[0] = v.x & 0xFFFFFFu;
      w[1] = v.y & 0xFFFFFFu;
      w[2] = v.z & 0xFFFFFFu;
      w[3] = v.w & 0xFFFFFFu;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        w[i] = (4u * gi + (uint32_t)i < A.N) ? __ldcg(from + 4u * gi + i) & 0xFFFFFFu : 0u;
    }
  };
  // a group's words with a tag into the copy (every group has four words there)
  auto store_own = [&](uint32_t gi, const uint32_t w[4], uint32_t tag) {
    if (dcheck(gi < A.groups, err, kSitePass3))
      st_flow4(F + 4u * gi, make_uint4(w[0] | tag, w[1] | tag, w[2] | tag, w[3] | tag));
  };
  auto store_state = [&](uint32_t gi, const uint32_t w[4]) {
    if (ALIGNED) {
      if (dcheck(4u * gi + 3u < A.N, err, kSitePass3))
        *reinterpret_cast<uint4*>(A.state + 4u * gi) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (4u * gi + (uint32_t)i < A.N) A.state[4u * gi + i] = w[i];
    }
  };

  uint32_t xyz[4] = {0u, 0u, 0u, 0u}, w[4] = {0u, 0u, 0u, 0u}, cfg = 0u;
  for (uint32_t gi = g_first; gi < g_hi; gi += stride) {
    load_own(gi, A.state, w);
    store_own(gi, w, tag0 << 24);
    if (eta_on) {  // as many cubes as groups
      cfg = A.eta[gi];
      st_flow(C + gi, cfg | (tag0 << 24));
    }
  }
  // (a lane without a group reads along with the last one)
  if (ONE) coords(min(g_first, g_hi - 1u), xyz);

  for (long long rel = 0; rel < n_steps; ++rel) {
    const long long step = step0 + rel;
    const uint32_t s_lo = (uint32_t)((unsigned long long)step & 0xFFFFFFFFu);
    const uint32_t s_hi = (uint32_t)((unsigned long long)step >> 32);
    const uint32_t tag = tag0 + 8u * (uint32_t)((unsigned long long)rel & 0xFFFFFFu);
    FlowSlot& slot = S.ring[rel % kWaveRing];
    {
      unsigned int spins = 0;
      while (!__all_sync(full, *(volatile int*)&slot.ready == (int)(rel + 1))) {
        if ((++spins & 1023u) == 0u && flow_stop(spins >> 6, H, err)) return;
      }
      __threadfence_block();
    }
    const unsigned long long plan = slot.plan;
    const int g = slot.g;
    const Tables3& Tb = S.Tb[g];
    const int nseg = plan_segments(plan);
    const bool rec = step_recorded(every, step);
    const bool last_step = rel == n_steps - 1;
    // accepted moves and the biased sums of their dN_HB + 1 and dN_sigma + 5
    uint32_t nacc = 0, hb_b = 0, dc_b = 0, pk = 0;
    uint32_t eta_dhb = 0;

    if (eta_on) {
      // Step 2 of the MC step: one Metropolis move of every cube with the
      // sigma fixed -- configuration (c + 1 + k) mod 9, k = floor(r0 8 / 2^32),
      // accepted iff r1 < T[g][dN_HB + 4], r = Philox((cube, step, 5)).  The
      // edges leaving the matching become allowed and those entering it
      // forbidden, so dN_HB = |bonded & old| - |bonded & new|.
      const uint32_t need = tag << 24;
      for (uint32_t cube0 = g_lo + (threadIdx.x & ~31u); cube0 < g_hi; cube0 += stride) {
        const uint32_t cube = cube0 + (threadIdx.x & 31u);
        const bool mine = cube < g_hi;
        const Words4 r = philox(cube, s_lo, s_hi, kTagEta, A.keys);
        uint32_t cell[8], v[8];
        cube_corners(A, min(cube, g_hi - 1u), cell);
        if (!ONE && mine) cfg = __ldcg(C + cube) & 15u;
        for (unsigned int spins = 0;;) {
          uint32_t late = 0u;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            v[j] = dcheck(cell[j] < A.N, err, kSiteEta3) ? ld_flow(F + cell[j]) : need;
            late |= behind(v[j], need);
          }
          if (__all_sync(full, (int32_t)late >= 0)) break;
          if ((++spins & 255u) == 0u && flow_stop(spins, H, err)) return;
          if (ALIGNED && !ONE) __nanosleep(kRestNs);
        }
        if (mine && dcheck(cfg < 9u, err, kSiteEta3)) {
          const uint32_t bonds = cube_bonds_packed(v);
          uint32_t nw = cfg + 1u + __umulhi(r.x, 8u);
          if (nw >= 9u) nw -= 9u;
          const uint32_t zo = S.eta_mask[cfg], zn = S.eta_mask[nw];
          const int dhb = __popc(bonds & zo) - __popc(bonds & zn);
          if ((unsigned long long)r.y < S.eta_thr[g][dhb + 4]) {
            cfg = nw;
            eta_dhb += (uint32_t)dhb;
          }
          st_flow(C + cube, cfg | ((tag + 1u) << 24));
          if (last_step) A.eta[cube] = (uint8_t)cfg;
        }
      }
    }

    for (int j = 0; j < nseg; ++j) {
      const uint32_t seg = plan_segment(plan, j);
      const bool last = j == nseg - 1;
      const uint32_t need = (j == 0 ? tag : tag + 1u + (uint32_t)j) << 24;
      const uint32_t out = (last ? tag + 8u : tag + 2u + (uint32_t)j) << 24;
      // Pass p's neighbour of a cell is at c + dlt - (coordinate == edge ? wrp
      // : 0) with the coordinate (x, y or z; ALIGNED: the group's x), the edge
      // value, the offset and the periodic wrap fixed for the segment.
      auto body = [&](auto na_c) -> bool {
        constexpr int NA = decltype(na_c)::value;
        Pass3 P[NA];
        uint32_t tagp[NA], axis[NA], edge[NA], dlt[NA], wrp[NA];
#pragma unroll
        for (int p = 0; p < NA; ++p) {
          const int a = segment_arm(seg, p);
          P[p] = make_pass3(a);
          tagp[p] = kTagArm0 + (uint32_t)a;
          const bool plus = (a & 1) == 0;
          axis[p] = 10u * (uint32_t)(a >> 1);
          if (a < 2) {
            edge[p] = plus ? (ALIGNED ? A.G : A.L) - 1u : 0u;
            dlt[p] = plus ? (ALIGNED ? 4u : 1u) : 0u - 1u;
            wrp[p] = plus ? A.L : 0u - A.L;
          } else if (a < 4) {
            edge[p] = plus ? A.L - 1u : 0u;
            dlt[p] = plus ? A.L : 0u - A.L;
            wrp[p] = plus ? A.L2 : 0u - A.L2;
          } else {
            edge[p] = plus ? A.L - 1u : 0u;
            dlt[p] = plus ? A.L2 : 0u - A.L2;
            wrp[p] = plus ? A.N : 0u - A.N;
          }
        }
        for (uint32_t gi0 = g_lo + (threadIdx.x & ~31u); gi0 < g_hi; gi0 += stride) {
          const uint32_t gi = gi0 + (threadIdx.x & 31u);
          const bool mine = gi < g_hi;
          const uint32_t c0 = 4u * min(gi, g_hi - 1u);
          Words4 draw[NA];
          if (ONE) {
#pragma unroll
            for (int p = 0; p < NA; ++p) draw[p] = philox(gi, s_lo, s_hi, tagp[p], A.keys);
          } else {
            coords(c0 >> 2, xyz);
            load_own(c0 >> 2, F, w);
          }
          // where the neighbours' words are (ALIGNED: one vector or, along x,
          // one word; else a word per cell)
          constexpr int NO = ALIGNED ? 1 : 4;
          uint32_t at[NA][NO], nb[NA][4];
#pragma unroll
          for (int p = 0; p < NA; ++p) {
#pragma unroll
            for (int i = 0; i < NO; ++i) {
              const uint32_t c = ALIGNED ? c0 : min(c0 + (uint32_t)i, A.N - 1u);
              const uint32_t coord = (xyz[i] >> axis[p]) & 1023u;
              at[p][i] = c + dlt[p] - ((coord == edge[p]) ? wrp[p] : 0u);
              if (!dcheck(at[p][i] + ((ALIGNED && axis[p] != 0u) ? 3u : 0u) < A.N, err, kSitePass3))
                at[p][i] = 0u;
            }
          }
          uint32_t cb[8];  // the cubes' words of the cells (colour 0, colour 1)
          const bool read_eta = eta_on && j == 0;
          for (unsigned int spins = 0;;) {
            uint32_t late = 0u;
#pragma unroll
            for (int p = 0; p < NA; ++p) {
              if (ALIGNED && axis[p] != 0u) {
                const uint4 v = ld_flow4(F + at[p][0]);
                nb[p][0] = v.x;
                nb[p][1] = v.y;
                nb[p][2] = v.z;
                nb[p][3] = v.w;
                late |= behind(v.x, need) | behind(v.y, need) | behind(v.z, need) |
                        behind(v.w, need);
              } else if (ALIGNED) {
                // the group's own words serve for the x neighbours: arm a^1
                // does not change in the segment
                const uint32_t xw = ld_flow(F + at[p][0]);
                late |= behind(xw, need);
                const bool plus = P[p].sh == 0u;
                nb[p][0] = plus ? w[1] : xw;
                nb[p][1] = plus ? w[2] : w[0];
                nb[p][2] = plus ? w[3] : w[1];
                nb[p][3] = plus ? xw : w[2];
              } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  nb[p][i] = ld_flow(F + at[p][i % NO]);
                  late |= behind(nb[p][i], need);
                }
              }
            }
            if (read_eta) {
              // the cubes of cell (x, y, z): colour c's has its corner of
              // smallest coordinates at the coordinates of parity c, the cell's
              // own or one less (periodic)
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const uint32_t x = ALIGNED ? 4u * (xyz[0] & 1023u) + (uint32_t)i : xyz[i] & 1023u;
                const uint32_t y = (xyz[ALIGNED ? 0 : i] >> 10) & 1023u, z = xyz[ALIGNED ? 0 : i] >> 20;
                const uint32_t H1 = A.H - 1u;
                const uint32_t k0 = ((z >> 1) * A.H + (y >> 1)) * A.H + (x >> 1);
                const uint32_t X = (x == 0u) ? H1 : (x - 1u) >> 1, Y = (y == 0u) ? H1 : (y - 1u) >> 1,
                               Z = (z == 0u) ? H1 : (z - 1u) >> 1;
                const uint32_t k1 = A.ncube / 2u + (Z * A.H + Y) * A.H + X;
                const bool in = dcheck(k0 < A.ncube && k1 < A.ncube, err, kSiteEta3);
                cb[i] = in ? ld_flow(C + k0) : need + (1u << 24);
                cb[4 + i] = in ? ld_flow(C + k1) : need + (1u << 24);
                late |= behind(cb[i], need + (1u << 24)) | behind(cb[4 + i], need + (1u << 24));
              }
            }
            if (__all_sync(full, (int32_t)late >= 0)) break;
            if ((++spins & 255u) == 0u && flow_stop(spins, H, err)) return false;
            if (ALIGNED && !ONE) __nanosleep(kRestNs);
          }
          if (mine) {
            if (read_eta) {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const uint32_t x = ALIGNED ? (uint32_t)i : xyz[i];  // parities
                const uint32_t y = xyz[ALIGNED ? 0 : i] >> 10, z = xyz[ALIGNED ? 0 : i] >> 20;
                const uint32_t j0 = (x & 1u) | ((y & 1u) << 1) | ((z & 1u) << 2);
                const uint32_t f0 = cb[i] & 15u, f1 = cb[4 + i] & 15u;
                const bool in = dcheck(f0 < 9u && f1 < 9u, err, kSiteEta3);
                const uint32_t f = in ? S.forbid[j0][f0] | S.forbid[j0 ^ 7u][f1] : 0u;
                w[i] = (w[i] & kArmBits) | (~f & kEtaBits);
              }
            }
            const uint32_t n = min(4u, A.N - c0);  // cells of the group (ALIGNED: 4)
#pragma unroll
            for (int p = 0; p < NA; ++p) {
              const Words4 r = ONE ? draw[p] : philox(gi, s_lo, s_hi, tagp[p], A.keys);
              const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (ALIGNED || (uint32_t)i < n)
                  w[i] = update_arm3<CMP64>(w[i], nb[p][i], rw[i], P[p], q, Tb, pk);
            }
            unpack_counts(pk, nacc, hb_b, dc_b);
            store_own(gi, w, out);
            if (last && last_step) store_state(gi, w);
            if (last && rec) {
              hist_group(w[0], w[1], w[2], w[3], slot.hist);
              // the words past the end (zero) count six arms in state 0 each
              if (!ALIGNED && n < 4u) atomicSub(&slot.hist[0], 6u * (4u - n));
            }
          }
          __syncwarp();
        }
        return true;
      };
      const int n = segment_passes(seg);
      const bool alive = (n == 1)   ? body(std::integral_constant<int, 1>{})
                         : (n == 2) ? body(std::integral_constant<int, 2>{})
                                    : body(std::integral_constant<int, 3>{});
      if (!alive) return;
    }

    flow_report(slot, (int)(hb_b - nacc + eta_dhb), (int)(dc_b - 5u * nacc), (int)nacc);
  }
}

template <bool ONE>
const void* flow3_kernel(bool aligned, bool cmp64) {
  if (aligned)
    return cmp64 ? (const void*)k_flow3<true, true, ONE> : (const void*)k_flow3<true, false, ONE>;
  return cmp64 ? (const void*)k_flow3<false, true, ONE> : (const void*)k_flow3<false, false, ONE>;
}

}  // namespace

// The launch of a cube: one group per thread and one block per SM (beside the
// engine's) where its groups allow it, else every resident block with several
// groups per thread.
Flow3Plan flow3_plan(const Args3& A, bool cmp64) {
  Flow3Plan P{};
  const bool aligned = (A.L % 4u) == 0u;
  const long long groups = A.groups;
  for (int one = 1; one >= 0 && P.blocks == 0; --one) {
    P.kernel = one ? flow3_kernel<true>(aligned, cmp64) : flow3_kernel<false>(aligned, cmp64);
    P.threads = flow_threads(one) + 32;
    const long long room =
        std::min(one ? sm_count() : INT_MAX, flow_resident_blocks(P.kernel, P.threads)) - 1;
    if (room < 1 || (one && groups > room * flow_threads(true))) continue;
    const long long share = (groups + room - 1) / room;
    P.groups_per_block = (uint32_t)((share + 31) / 32 * 32);
    if (one) P.threads = flow_block(P.kernel, P.groups_per_block, P.threads);
    P.blocks = (int)((groups + P.groups_per_block - 1) / P.groups_per_block);
  }
  P.copy_words = (size_t)kFlowHead + 4 * (size_t)groups + A.ncube;
  return P;
}

cudaError_t launch_flow3(const Args3& A, const Flow3Plan& P, WaveHdr* H, long long n_steps,
                         int every, cudaStream_t s) {
  if (P.blocks < 1) return cudaErrorCooperativeLaunchTooLarge;
  uint32_t gpb = P.groups_per_block;
  uint32_t* copy = reinterpret_cast<uint32_t*>(H + 1);
  void* args[6] = {const_cast<Args3*>(&A), &gpb, &H, &copy, &n_steps, &every};
  return cudaLaunchCooperativeKernel(P.kernel, dim3(P.blocks + 1), dim3(P.threads), args, 0, s);
}

}  // namespace cvf
