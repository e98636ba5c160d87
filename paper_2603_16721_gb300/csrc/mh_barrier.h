// The rules by which the blocks of a team agree, at a grid barrier, to stop for a batch's
// yield request.  Arrivals count up over the barriers of a launch, so barrier k (from 0) of
// n blocks ends with the (k + 1) n-th.  A block may find the request set before its arrival
// at barrier k while others, that came earlier, did not; and a fast block may be through
// barrier k, and find the request on its way to barrier k + 1, before a slow one has looked
// for a request of barrier k.  So the flag names the barrier: it is written before the
// arrival, hence seen by all after the barrier, and a flag of a later barrier does not
// count yet.  (A block that finds the request writes it once at most: all stop there.)
#pragma once

#ifdef __CUDACC__
#define MH_BOTH __host__ __device__ __forceinline__
#else
#define MH_BOTH static inline
#endif

namespace mh {

// The flag of a block that has not arrived yet and reads `arrived` arrivals.
MH_BOTH unsigned yield_flag(unsigned arrived, unsigned nblocks) { return arrived / nblocks + 1u; }

// Whether the blocks stop at the barrier that a block came to as the (old + 1)-th arrival.
MH_BOTH bool yield_stops(unsigned flag, unsigned old, unsigned nblocks) { return flag != 0u && flag <= old / nblocks + 1u; }

}  // namespace mh
