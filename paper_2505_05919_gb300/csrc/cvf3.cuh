// cvf3.cuh -- device building blocks of the cubic lattice (cvf3.cu,
// cvf3_flow.cu): the launch arguments, the arm order of a step, the Metropolis
// update of one arm (Sec. II.C with Eq. H) and the geometry of the
// checkerboard cubes of the eta update (App. A).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "cvf_device.cuh"
#include "cvf_fastdiv.cuh"
#include "cvf_lattice.cuh"

namespace cvf {

constexpr int kThreads3 = 256;
constexpr uint32_t kTagArm0 = 8u;       // draws of arm a: Philox tag 8 + a
constexpr uint32_t kTagInit0 = 16u;     // random init of arm a: tag 16 + a
constexpr uint32_t kR6 = 0x111111u;       // 1 in the six arm nibbles
constexpr uint32_t kArmBits = 0x777777u;  // the sigma bits of the six arm nibbles
constexpr uint32_t kEtaBits = 0x888888u;  // bit 3 of the six arm nibbles: the edges' eta
constexpr uint32_t kTagEta = 5u;          // cube moves: Philox tag 5
constexpr uint32_t kTagEtaInit = 6u;      // random initial cube configurations: tag 6

struct Args3 {
  uint32_t* state;                  // L^3 words, updated in place
  Ctrl* ctrl;
  const unsigned long long* table;  // [g][(dN_HB+1)*11 + dN_sigma+5]
  const VolumeArgs* vol;
  cvf_obs* ring;
  long long ring_cap;
  RoundKeys keys;
  uint32_t L, L2, N;
  uint32_t groups;                  // ceil(N / 4): four consecutive cells each
  uint32_t G;                       // L / 4 (groups per row when L % 4 == 0)
  uint32_t q;
  FastDiv div_G, div_L, div_L2;
  // eta (App. A): cube configurations (L^3/4 bytes; null without eta moves),
  // the 12-bit edge masks of the nine configurations, the move thresholds
  // [g][dN_HB + 4], L / 2 and the number of cubes
  uint8_t* eta;
  const unsigned long long* eta_table;
  uint16_t masks[9];
  uint32_t H, ncube;
  FastDiv div_H;
};

// The dataflow sweep of a cube (cvf3_flow.cu): its kernel, the blocks that own
// cells and the groups of each, and the words of its tagged copy of the cube
// (zero before the first call).
struct Flow3Plan {
  const void* kernel;
  int threads;
  int blocks;  // 0: the kernel has no room on this GPU
  uint32_t groups_per_block;
  size_t copy_words;
};
Flow3Plan flow3_plan(const Args3& A, bool cmp64);
// Enqueues the call's steps in one cooperative launch; H is its scratch, and the
// copy lies behind it.
cudaError_t launch_flow3(const Args3& A, const Flow3Plan& P, WaveHdr* H, long long n_steps,
                         int every, cudaStream_t s);

// ---------------------------------------------------------------------------
// Arm order and segments of a step.  The order is permutation number
// floor(w 720 / 2^32) of the six arms (lexicographic), w word 0 of
// Philox((2^32-2, step, 4)).  A pass over arm a reads, besides the cell's own
// word, only arm a^1 of the neighbour in direction a, which only the pass over
// a^1 changes; so consecutive passes without an opposite pair form a segment
// that every cell goes through in registers: every partner it reads is
// constant during the segment, whichever version of the neighbour's word it
// sees, and the result is the one of the passes run one after the other.  The
// order is cut before the first arm whose opposite is already in the current
// segment: 2 to 4 segments (2.67 on average over the 720 orders) of at most
// three passes.
//
// Plan: bits 0..2 the number of segments; segment j in the eleven bits from
// 3 + 11 j on: two bits for its passes, then three bits for each pass's arm.
// ---------------------------------------------------------------------------
__device__ inline unsigned long long make_plan(long long step, const RoundKeys& K) {
  const Words4 r = philox(kCellLayers, (uint32_t)((unsigned long long)step & 0xFFFFFFFFu),
                          (uint32_t)((unsigned long long)step >> 32), kTagLayers, K);
  uint32_t idx = __umulhi(r.x, 720u);
  const uint32_t fact[6] = {120u, 24u, 6u, 2u, 1u, 1u};
  uint32_t avail = 0x543210u;  // the arms left, one per nibble
  unsigned long long plan = 0;
  uint32_t segments = 0, n = 0, arms = 0, seen = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const uint32_t j = idx / fact[i];
    idx -= j * fact[i];
    const uint32_t a = (avail >> (4u * j)) & 7u;
    const uint32_t low = (1u << (4u * j)) - 1u;
    avail = (avail & low) | ((avail >> 4) & ~low);
    if (seen & (1u << (a ^ 1u))) {
      plan |= (unsigned long long)(n | (arms << 2)) << (3u + 11u * segments);
      ++segments;
      n = arms = seen = 0u;
    }
    seen |= 1u << a;
    arms |= a << (3u * n);
    ++n;
  }
  plan |= (unsigned long long)(n | (arms << 2)) << (3u + 11u * segments);
  return plan | (segments + 1u);
}

__device__ __forceinline__ int plan_segments(unsigned long long plan) { return (int)(plan & 7u); }

// Segment j of a plan: the number of its passes, and their arms (three bits
// each, from bit 2 on).
__device__ __forceinline__ uint32_t plan_segment(unsigned long long plan, int j) {
  return (uint32_t)(plan >> (3 + 11 * j)) & 0x7FFu;
}
__device__ __forceinline__ int segment_passes(uint32_t seg) { return (int)(seg & 3u); }
__device__ __forceinline__ int segment_arm(uint32_t seg, int p) {
  return (int)((seg >> (2 + 3 * p)) & 7u);
}

// Shared tables of one (cube, gate): the proposals for the current q and the
// threshold rows.
//   prop[q k + sigma]  7 ^ sigma' (sigma' = (sigma + 1 + k) mod q) in every arm
//                      nibble, k <= q - 2 <= 6 (q = 6: 30 entries in 30 banks)
//   thr[i], change[i]  for i = 11 (dN_HB + 1) + dN_sigma + 5: T - 1 and the
//                      packed count change of an accepted move ((1 << 24) +
//                      ((dN_HB + 1) << 16) + dN_sigma + 5); both 0 where T = 0
//                      (no draw is below it; the kernels of a table that holds
//                      a T = 0 also ask for a nonzero change: CMP64)
constexpr int kRows3 = 33;
struct Tables3 {
  uint32_t thr[kRows3 + 3];
  uint32_t change[kRows3 + 3];
  uint32_t prop[64];
};

// Both fills are called by the block's first `threads` threads.
__device__ __forceinline__ void fill_prop3(Tables3& Tb, uint32_t q, int threads) {
  for (int e = threadIdx.x; e < 64; e += threads) {
    const uint32_t k = (uint32_t)e / q, s = (uint32_t)e - k * q;
    uint32_t sp = s + 1u + k;  // entries with k > q - 2 are never read
    while (sp >= q) sp -= q;
    Tb.prop[e] = (sp ^ 7u) * kR6;
  }
}

__device__ __forceinline__ void fill_rows3(Tables3& Tb, const unsigned long long* table33,
                                           int threads) {
  for (int i = threadIdx.x; i < kRows3; i += threads) {
    const unsigned long long t = table33[i];
    Tb.thr[i] = t ? (uint32_t)(t - 1ull) : 0u;
    Tb.change[i] = t ? (1u << 24) + ((uint32_t)(i / 11) << 16) + (uint32_t)(i % 11) : 0u;
  }
}

// One pass of a segment: its arm a and what follows from it.
struct Pass3 {
  uint32_t sh;     // 4a
  uint32_t nrot;   // right rotation that moves nibble a^1 to nibble a
  uint32_t arm;    // 7 << 4a
  uint32_t edge;   // 8 << 4a: the edge's eta copy
  uint32_t crot;   // right rotation that moves the nibble-a sums to bit 0
};

__device__ __forceinline__ Pass3 make_pass3(int a) {
  Pass3 p;
  p.sh = 4u * (uint32_t)a;
  p.nrot = (a & 1) ? 28u : 4u;
  p.arm = 7u << p.sh;
  p.edge = 8u << p.sh;
  p.crot = p.sh + 3u;
  return p;
}

// ---------------------------------------------------------------------------
// Metropolis update of the arm of pass P of one cell (Sec. II.C with Eq. H).
//   w     the cell word (sigma_b in the low three bits of nibble b, the eta
//         copy of the arm's edge in bit 3), nw the neighbour's word in the
//         arm's direction (its nibble a^1 is the partner), r the cell's draw
// Proposal: r (q-1) = k 2^32 + u, sigma' from the shared table.  x holds the
// partner in the arm's own nibble; a nibble y of x ^ sigma gives y + 7, whose
// bit 3 is set iff it differs, a nibble 7 ^ y of x ^ (7 ^ sigma') gives
// (7 ^ y) + 1, whose bit 3 is set iff it is equal to sigma' (no carry leaves
// a nibble).  Over the five other arms the bits of both words count
// dN_sigma + 5; the two of the arm's own nibble add up to c = dN_HB + 1 -- or to
// 1 on an edge with eta = 0, where the first is forced on and the second
// off.  So popc of both words is D + c with D = dN_sigma + 5, and the row is
// D + 11 c: 33 thresholds in 33 words, read without bank conflicts.
// ---------------------------------------------------------------------------
template <bool CMP64>
__device__ __forceinline__ uint32_t update_arm3(uint32_t w, uint32_t nw, uint32_t r,
                                                const Pass3& P, uint32_t q, const Tables3& Tb,
                                                uint32_t& pk) {
  uint32_t u, k;
  asm("{\n\t.reg .b64 t;\n\tmul.wide.u32 t, %2, %3;\n\tmov.b64 {%0, %1}, t;\n\t}"
      : "=r"(u), "=r"(k)
      : "r"(r), "r"(q - 1u));
  const uint32_t s = (w >> P.sh) & 7u;
  const uint32_t nR = Tb.prop[k * q + s];
  const uint32_t x = ((w & ~P.arm) | (__funnelshift_r(nw, nw, P.nrot) & P.arm)) & kArmBits;
  const uint32_t off = ~w & P.edge;  // the edge is not allowed
  const uint32_t fs = (((x ^ (s * kR6)) + 0x777777u) | off) & kEtaBits;
  const uint32_t fp = ((x ^ nR) + kR6) & ~off & kEtaBits;
  const uint32_t c = ((fs + fp) >> P.crot) & 3u;
  const uint32_t i = (uint32_t)(__popc(fs) + __popc(fp)) + 10u * c;
  const uint32_t thr = Tb.thr[i], change = Tb.change[i];
  bool accept = u <= thr;
  if (CMP64) accept = accept && change != 0u;
  if (accept) {
    w = (w & ~P.arm) | (~nR & P.arm);
    pk += change;
  }
  return w;
}

// Adds a group's packed count changes to the thread's totals.
__device__ __forceinline__ void unpack_counts(uint32_t& pk, uint32_t& nacc, uint32_t& hb_b,
                                              uint32_t& dc_b) {
  nacc += pk >> 24;
  hb_b += (pk >> 16) & 0xFFu;
  dc_b += pk & 0xFFFFu;
  pk = 0;
}

// N_q' of the four final cell words of a group, added to the block's eight
// shared counters: per word a count word (nibble v = arms in state v), two
// words summed (nibbles <= 12), nibbles v and v+4 moved to the 16-bit lanes
// of word v (<= 24 per lane), reduced over the converged lanes of the warp
// (<= 768 per lane) and added by the lowest of them.
__device__ __forceinline__ uint32_t count_word(uint32_t w) {
  uint32_t c = 0;
#pragma unroll
  for (int b = 0; b < 6; ++b) c += 1u << (4u * ((w >> (4 * b)) & 7u));
  return c;
}

__device__ __forceinline__ void hist_group(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                                           uint32_t* s_hist) {
  const uint32_t h01 = count_word(w0) + count_word(w1);
  const uint32_t h23 = count_word(w2) + count_word(w3);
  const unsigned mask = __activemask();
  const int leader = __ffs(mask) - 1;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    uint32_t lanes = ((h01 >> (4 * v)) & 0x000F000Fu) + ((h23 >> (4 * v)) & 0x000F000Fu);
    lanes = __reduce_add_sync(mask, lanes);
    if ((int)(threadIdx.x & 31) == leader) {
      if (lanes & 0xFFFFu) atomicAdd(&s_hist[v], lanes & 0xFFFFu);
      if (lanes >> 16) atomicAdd(&s_hist[v + 4], lanes >> 16);
    }
  }
}

// ---------------------------------------------------------------------------
// eta (App. A).  Cube (colour, X, Y, Z) has its corner of smallest
// coordinates at (2X + colour, 2Y + colour, 2Z + colour); corner j sits at
// offset (j & 1, (j >> 1) & 1, (j >> 2) & 1); edge e runs along axis d = e / 4
// from corner lo(e) -- the (e % 4)-th corner with bit d clear -- to lo(e) |
// (1 << d).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int edge_lo(int e) {
  const int d = e >> 2, k = e & 3;
  // corners with bit d clear, in increasing order: d = 0: 0 2 4 6; d = 1:
  // 0 1 4 5; d = 2: 0 1 2 3
  return (d == 0) ? 2 * k : (d == 1) ? ((k & 1) | ((k >> 1) << 2)) : k;
}

// The eight corner cells of a cube: the corner of smallest coordinates and
// the steps +x, +y, +z from it (periodic).
__device__ __forceinline__ void cube_corners(const Args3& A, uint32_t cube, uint32_t cell[8]) {
  const uint32_t H = A.H, H2 = H * H;
  const uint32_t colour = (cube >= H2 * H) ? 1u : 0u;
  const uint32_t rest = cube - colour * H2 * H;
  const uint32_t Zc = fdiv(rest, A.div_H);  // Z H + Y
  const uint32_t X = rest - Zc * H;
  const uint32_t Z = fdiv(Zc, A.div_H);
  const uint32_t Y = Zc - Z * H;
  const uint32_t L = A.L, L2 = A.L2;
  const uint32_t x0 = 2u * X + colour, y0 = 2u * Y + colour, z0 = 2u * Z + colour;
  const uint32_t base = z0 * L2 + y0 * L + x0;
  const uint32_t dx = (x0 + 1u == L) ? 1u - L : 1u;
  const uint32_t dy = (y0 + 1u == L) ? L - L2 : L;
  const uint32_t dz = (z0 + 1u == L) ? L2 - A.N : L2;  // unsigned wrap-around
  cell[0] = base;
  cell[1] = base + dx;
  cell[2] = base + dy;
  cell[3] = cell[1] + dy;
  cell[4] = base + dz;
  cell[5] = cell[1] + dz;
  cell[6] = cell[2] + dz;
  cell[7] = cell[3] + dz;
}

// The bonded edges of a cube (sigma only; eta is not read) in the packed
// layout of the edge masks: edge e = 4 d + k (axis d, k-th lower corner)
// at bit 8 k + 7 - d.  For axis d, byte d of a corner word holds its +d arm
// (low nibble) and -d arm (high nibble); the bytes of the four lower and of
// the four upper corners are gathered into one word each, and one nibble
// comparison per byte tests the four edges at once.
__device__ __forceinline__ uint32_t cube_bonds_packed(const uint32_t w[8]) {
  uint32_t bonds = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    // corners with bit d clear, in increasing order, and their +d partners
    const int l0 = (d == 0) ? 0 : 0, l1 = (d == 0) ? 2 : 1, l2 = (d == 0) ? 4 : (d == 1) ? 4 : 2,
              l3 = (d == 0) ? 6 : (d == 1) ? 5 : 3;
    const int u = 1 << d;
    const uint32_t sel = (uint32_t)d | ((uint32_t)(4 + d) << 4);
    const uint32_t lo = __byte_perm(__byte_perm(w[l0], w[l1], sel), __byte_perm(w[l2], w[l3], sel),
                                    0x5410u);
    const uint32_t hi = __byte_perm(__byte_perm(w[l0 | u], w[l1 | u], sel),
                                    __byte_perm(w[l2 | u], w[l3 | u], sel), 0x5410u);
    // byte k: the +d arm of lower corner k against the -d arm of its partner
    const uint32_t m = (lo ^ (hi >> 4)) & 0x07070707u;
    const uint32_t differ = (m | 0x80808080u) - 0x01010101u;  // bit 7 set where m != 0
    bonds |= (~differ & 0x80808080u) >> d;
  }
  return bonds;
}

// An edge mask (bit e = edge e) in the packed layout of cube_bonds_packed.
__device__ __forceinline__ uint32_t pack_edge_mask(uint32_t m12) {
  uint32_t p = 0;
#pragma unroll
  for (int e = 0; e < 12; ++e) p |= ((m12 >> e) & 1u) << (8 * (e & 3) + 7 - (e >> 2));
  return p;
}

// The eta-copy flips of the corner words for the edges set in a packed flip
// mask: the +d arm (bit 8 d + 3) of the lower corner and the -d arm (bit
// 8 d + 7) of the upper corner of each edge.
__device__ __forceinline__ void cube_flip_bits(uint32_t flip, uint32_t x[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = 0u;
#pragma unroll
  for (int e = 0; e < 12; ++e) {
    const int d = e >> 2, lo = edge_lo(e), hi = lo | (1 << d);
    const uint32_t f = (flip >> (8 * (e & 3) + 7 - d)) & 1u;
    x[lo] ^= f << (8 * d + 3);
    x[hi] ^= f << (8 * d + 7);
  }
}

}  // namespace cvf
