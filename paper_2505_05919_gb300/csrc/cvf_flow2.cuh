// cvf_flow2.cuh -- the dataflow sweep of the square lattice (cvf_flow2.cu) and
// the layered schedule's arm order.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "cvf_device.cuh"
#include "cvf_fastdiv.cuh"
#include "cvf_lattice.cuh"

namespace cvf {

// Items of a launch: strips' words (checkerboard) or groups (layered).
struct Flow2Geom {
  uint32_t items, per_block;
  uint32_t groups_x;  // layered: groups per row
  FastDiv div_row;    // by the items of a row
};

// The launch of a lattice and the words of its tagged copy (zero before the
// first call).
struct Flow2Plan {
  const void* kernel;
  int threads, blocks;  // blocks 0: the lattice is too large for it
  bool cluster;         // one cluster holds the words: no copy
  Flow2Geom geom;
  size_t copy_words;
};

Flow2Plan flow2_plan(int L, int schedule, int rng_words, bool cmp64);
// Enqueues the call's steps in one cooperative launch; H is its scratch, and the
// copy lies behind it.
cudaError_t launch_flow2(const LatticeArgs& A, const Flow2Plan& P, WaveHdr* H, long long n_steps,
                         int every, cudaStream_t s);

// Many lattices in one launch (k_flow2_batch): what the kernel takes by value.
constexpr int kFlow2BatchBlocks = 640;          // blocks of a launch at most
constexpr int kFlow2BatchMax = 128;             // lattices of a launch at most
constexpr long long kFlow2BatchWords = 5 << 17;  // words of its copies at most
constexpr int kFlow2BatchForms = 6;             // kernels to choose from
struct Flow2Replica {
  LatticeArgs args;
  Flow2Geom geom;
  WaveHdr* hdr;
  uint32_t* copy;
  long long n_steps;             // at most 2^30
  uint32_t first_block, blocks;  // that sweep
};
struct Flow2Batch {
  int n;
  unsigned int* err;  // set when a wait gives up or an index check fails
  uint8_t of_block[kFlow2BatchBlocks];  // the lattice of a block (the first n: the books)
  Flow2Replica item[kFlow2BatchMax];
};
static_assert(sizeof(Flow2Batch) <= 32764, "fits a kernel's parameters");

// Bytes of scratch that any launch fits.
size_t flow2_batch_scratch();
// Chooses the form of a launch for n lattices of these sides and its blocks; false
// if they are not resident at once in any form.  slots[f]: the resident blocks of
// form f, 0 until asked for.
bool flow2_batch_plan(Flow2Batch* B, const int* sides, int n, int rng_words, bool cmp64,
                      int slots[kFlow2BatchForms], int* form);
// Clears the scratch and launches; args, n_steps and err are the caller's.
cudaError_t launch_flow2_batch(Flow2Batch* B, void* scratch, int rng_words, bool cmp64, int form,
                               cudaStream_t s);

// Order of the layered schedule's arms in a step: the Fisher-Yates order drawn
// from Philox((2^32-2, step, tag 4)), cut before the first arm whose opposite is
// already in the segment (two or three segments).  Plan word: bits 2i..2i+1 the
// arm of pass i, bit 8 + i set when pass i opens a new segment (i = 1..3).
__device__ inline uint32_t layer_plan(long long step, const RoundKeys& K) {
  const Words4 r = philox(kCellLayers, (uint32_t)((unsigned long long)step & 0xFFFFFFFFu),
                          (uint32_t)((unsigned long long)step >> 32), kTagLayers, K);
  const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
  uint32_t order = 0xE4u;  // arms 0, 1, 2, 3 in two bits each
#pragma unroll
  for (int i = 3; i >= 1; --i) {
    const uint32_t j = __umulhi(rw[3 - i], (uint32_t)(i + 1));
    const uint32_t x = ((order >> (2 * i)) ^ (order >> (2u * j))) & 3u;  // swap i and j
    order ^= (x << (2 * i)) | (x << (2u * j));
  }
  uint32_t plan = 0, in_segment = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t a = (order >> (2 * i)) & 3u;
    if (in_segment & (1u << (a ^ 1u))) {
      plan |= 1u << (8 + i);
      in_segment = 0;
    }
    in_segment |= 1u << a;
    plan |= a << (2 * i);
  }
  return plan;
}

// Segment j of a plan: bits 0..1 the number of its arms (0: no such segment),
// then two bits for each.
__device__ __forceinline__ uint32_t layer_segment(uint32_t plan, int j) {
  uint32_t segment = 0, n = 0, arms = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (i > 0 && ((plan >> (8 + i)) & 1u)) ++segment;
    if (segment == (uint32_t)j && n < 2u) {
      arms |= ((plan >> (2 * i)) & 3u) << (2u + 2u * n);
      ++n;
    }
  }
  return arms | n;
}

}  // namespace cvf
