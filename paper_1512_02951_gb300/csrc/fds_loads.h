// The copies a warp has under way into its shared-memory buffers, one mbarrier for each buffer: which
// phase of a barrier comes next, and whether a copy has been announced on it that has not arrived.  A
// warp that gives up on a copy waits once more, with a limit, for exactly those before it leaves: the
// one it gave up on among them (its bytes may still be written to shared memory), and none that was
// never issued (that wait could only run out).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FDS_LOADS_FN __host__ __device__ __forceinline__
#else
#define FDS_LOADS_FN inline
#endif

namespace fds {

constexpr int kMaxLoads = 8;

// bit i: the parity to wait for on barrier i; bit kMaxLoads + i: a copy is pending there
struct Loads {
  uint32_t st = 0;

  // a copy has been announced on barrier i (one at a time)
  FDS_LOADS_FN void issued(int i) { st ^= (1u << kMaxLoads) << i; }
  // the copy pending on barrier i has arrived
  FDS_LOADS_FN void arrived(int i) { st ^= ((1u << kMaxLoads) | 1u) << i; }
  FDS_LOADS_FN uint32_t parity(int i) const { return (st >> i) & 1u; }
  FDS_LOADS_FN bool pending(int i) const { return (st >> (kMaxLoads + i)) & 1u; }
  // wait(i, parity) for every pending copy of the first n barriers
  template <typename Wait>
  FDS_LOADS_FN void drain(int n, Wait wait) const {
    for (int i = 0; i < n; ++i)
      if (pending(i)) wait(i, parity(i));
  }
};

}  // namespace fds
