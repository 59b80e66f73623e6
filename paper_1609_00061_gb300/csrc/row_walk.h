// The walk of the row-OR kernel's warps over the rows of a contraction: batches of
// consecutive rows, dealt out cyclically over every warp.  Plain C++, so that its
// limits can be checked on the host.
#ifndef PA_ROW_WALK_H_
#define PA_ROW_WALK_H_

#include <stdint.h>

#ifdef __CUDACC__
#define PA_HD __host__ __device__ __forceinline__
#else
#define PA_HD inline
#endif

namespace pa {

// A warp's batches start at rows warp * batch, + step, + 2 step, ..  The kernel
// fetches three batches ahead, so it forms rows up to M + 4 step: 32 unsigned bits
// hold them for every M below 2^31, a step being at most 32 rows of some 1e4 warps.
struct RowWalk {
  uint32_t M;      // rows
  uint32_t batch;  // rows of a batch: 32 / lanes, fewer when that leaves warps idle
  uint32_t step;
  PA_HD RowWalk(int64_t rows, int warps, int lanes_per_row) : M((uint32_t)rows) {
    const uint32_t most = 32u / (uint32_t)lanes_per_row;
    const uint32_t share = (M + (uint32_t)warps - 1u) / (uint32_t)warps;
    batch = share < most ? share : most;
    step = (uint32_t)warps * batch;
  }
};

}  // namespace pa

#endif  // PA_ROW_WALK_H_
