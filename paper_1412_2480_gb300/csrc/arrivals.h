// The arrival counters of the grid-wide waits, for host and device code.
#pragma once

#ifdef __CUDACC__
#define PIC_HD __host__ __device__ __forceinline__
#else
#define PIC_HD inline
#endif

namespace pic {

// Whether a counter that every block raises by one at each of its waits says that all
// `nblocks` have reached wait number `epoch`. The counter is 32 bits wide and may wrap: a
// block is at most one wait ahead of another, so the distance to the target, taken modulo
// 2^32, is small and its sign tells.
PIC_HD bool all_arrived(unsigned int seen, unsigned int epoch, unsigned int nblocks) {
    return static_cast<int>(seen - epoch * nblocks) >= 0;
}

}  // namespace pic
