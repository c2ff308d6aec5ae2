// cvf_observe.cu -- the observables' kernel (cvf_observe.cuh).
//
// What bounds it: at small lattices the launch, at large ones the bytes (2 or 4
// a cell).  Each thread counts the arms of its cells in nibbles, two cells at a
// time, and adds them to 16-bit lanes; the warp sums them by redux, the block in
// shared memory, and the last block of a lattice writes its record -- to pinned
// host memory where the host waits for it -- and clears the counters, so a read
// is one launch and no memset or copy (a memset, a count with nine contended
// 64-bit shared atomics per thread, a second launch and a copy took 38 us at
// 32^2, 113 us at 1024^2).
#include <cuda_runtime.h>

#include "cvf_host.h"
#include "cvf_observe.cuh"

namespace cvf {
namespace {

// Nibble v: the arms in state v among the cells of a word (ARMS nibbles).
template <int ARMS>
__device__ __forceinline__ uint32_t count_arms(uint32_t w) {
  uint32_t n = 0;
#pragma unroll
  for (int b = 0; b < ARMS; ++b) n += 1u << (4u * ((w >> (4 * b)) & 7u));
  return n;
}

// Equal pairs inside the two cells of a word: every arm against the next one of
// its cell (four pairs), and arms 0 and 1 against those two further on.
__device__ __forceinline__ uint32_t word_pairs(uint32_t w) {
  const uint32_t next = ((w >> 4) & 0x0FFF0FFFu) | ((w << 12) & 0xF000F000u);
  const uint32_t far = __byte_perm(w, 0u, 0x2301u);
  // a nibble of w ^ x is 0 where the arms are equal: then adding 7 leaves bit 3 clear
  const uint32_t e1 = ~((w ^ next) + 0x77777777u) & 0x88888888u;
  const uint32_t e2 = ~((w ^ far) + 0x77777777u) & 0x00880088u;
  return (uint32_t)(__popc(e1) + __popc(e2));
}

template <bool CUBIC>
__global__ void __launch_bounds__(kObserveThreads)
    k_observe(const __grid_constant__ ObserveArgs A) {
  const ObserveItem& I = A.item[blockIdx.y];
  __shared__ unsigned long long s_cnt[9];
  __shared__ int s_last;
  const long long N = I.N;
  // blocks with work (every lattice has at least two cells)
  constexpr long long kCells = 4;
  const long long loads = (N + kCells - 1) / kCells;
  const int blocks = (int)min((long long)gridDim.x, (loads + kObserveThreads - 1) / kObserveThreads);
  if ((int)blockIdx.x >= blocks) return;
  if (threadIdx.x < 9) s_cnt[threadIdx.x] = 0ull;
  __syncthreads();
  uint32_t h[4] = {0u, 0u, 0u, 0u}, pairs = 0u;
  auto add = [&](uint32_t n) {  // n: nibbles of at most two cells
#pragma unroll
    for (int v = 0; v < 4; ++v) h[v] += (n >> (4 * v)) & 0x000F000Fu;
  };
  for (long long i = (long long)blockIdx.x * kObserveThreads + threadIdx.x; i < loads;
       i += (long long)blocks * kObserveThreads) {
    if (CUBIC) {
      const uint32_t* c = reinterpret_cast<const uint32_t*>(I.state) + 4 * i;
      if (4 * i + 4 <= N) {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(c));
        add(count_arms<6>(w.x) + count_arms<6>(w.y));
        add(count_arms<6>(w.z) + count_arms<6>(w.w));
      } else {
        for (long long k = 4 * i; k < N; ++k) add(count_arms<6>(c[k - 4 * i]));
      }
    } else {  // N is a multiple of 4 and so is the start of either half of the pair
      const uint2 w = __ldg(reinterpret_cast<const uint2*>(I.state) + i);
      add(count_arms<8>(w.x));
      add(count_arms<8>(w.y));
      pairs += word_pairs(w.x) + word_pairs(w.y);
    }
  }
#pragma unroll
  for (int v = 0; v < 9; ++v) {
    const uint32_t x = (v == 8) ? pairs : (h[v & 3] >> ((v & 4) ? 16 : 0)) & 0xFFFFu;
    const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, x);
    if ((threadIdx.x & 31u) == 0u && sum) atomicAdd(&s_cnt[v], (unsigned long long)sum);
  }
  __syncthreads();
  if (threadIdx.x < 9 && s_cnt[threadIdx.x]) atomicAdd(&I.counts[threadIdx.x], s_cnt[threadIdx.x]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0)
    s_last = (atomicAdd(&I.counts[9], 1ull) == (unsigned long long)(blocks - 1)) ? 1 : 0;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (threadIdx.x < 9) {
    s_cnt[threadIdx.x] = __ldcg(&I.counts[threadIdx.x]);
    I.counts[threadIdx.x] = 0ull;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    I.counts[9] = 0ull;
    Ctrl c = *I.ctl;
    if (!CUBIC) c.n_coop = (long long)s_cnt[8];
    cvf_obs o = make_obs(*I.vol, &c);
    for (int v = 0; v < 8; ++v) o.n_state[v] = (long long)s_cnt[v];
    *I.out = o;
    if (A.error_out && blockIdx.y == 0) *A.error_out = A.error ? *A.error : 0u;
  }
}

}  // namespace

cudaError_t launch_observe(const ObserveArgs& A, int items, long long most, bool cubic,
                           cudaStream_t s) {
  const dim3 grid((unsigned)observe_blocks(most, sm_count(), cubic ? 6 : 4), (unsigned)items);
  if (cubic)
    k_observe<true><<<grid, kObserveThreads, 0, s>>>(A);
  else
    k_observe<false><<<grid, kObserveThreads, 0, s>>>(A);
  return cudaGetLastError();
}

}  // namespace cvf
