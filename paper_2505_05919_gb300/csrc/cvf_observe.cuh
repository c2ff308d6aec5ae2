// cvf_observe.cuh -- the observables of a lattice at a point of its stream
// (Eq. V, Eq. H, Eq. correlation): N_q' and, on the square lattice, N_sigma
// counted from the cell words, and the record written where the caller reads it,
// in one launch.
#pragma once
#include <cstdint>

#include "cvf_device.cuh"

namespace cvf {

// One lattice to observe.  counts: ten 64-bit words, zero before the launch and
// left zero (N_q'[8], N_sigma, finished blocks); out: device or pinned host
// memory.
struct ObserveItem {
  const void* state;  // uint16 cells (square) or uint32 cells (cubic)
  long long N;
  const VolumeArgs* vol;
  const Ctrl* ctl;
  unsigned long long* counts;
  cvf_obs* out;
};

// The items of a launch travel as a kernel parameter.
constexpr int kObserveItems = 64;
struct ObserveArgs {
  ObserveItem item[kObserveItems];
  const unsigned int* error;  // a word to copy beside the records (or null)
  unsigned int* error_out;
};

constexpr int kObserveThreads = 256;
// Blocks per lattice of N cells of `arms` arms: two loads of four cells a thread
// for small ones, eight blocks an SM for large ones, but as many as it takes for
// a thread's arms of one state to fit its 16-bit lanes.
inline int observe_blocks(long long N, int sms, int arms) {
  const long long want = (N + 8 * kObserveThreads - 1) / (8 * kObserveThreads);
  const long long most = 8ll * sms;
  const long long loads = 65535 / (4 * arms);  // of a thread at most
  const long long least = (N + 4 * kObserveThreads * loads - 1) / (4 * kObserveThreads * loads);
  const long long blocks = want > most ? most : want;
  return (int)(blocks > least ? blocks : least);
}

// Enqueues the observation of items (at most kObserveItems) of lattices of up
// to `most` cells; cubic: six arms in a uint32 per cell, else four in a uint16.
cudaError_t launch_observe(const ObserveArgs& A, int items, long long most, bool cubic,
                           cudaStream_t s);

}  // namespace cvf
