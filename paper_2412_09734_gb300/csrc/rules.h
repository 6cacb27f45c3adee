// Predicates that kernels decide by, also as plain C++ so that they can be checked on any
// machine.
#pragma once

#ifdef __CUDACC__
#define MPAX_RULE __host__ __device__ __forceinline__
#else
#define MPAX_RULE inline
#endif

namespace mpax {

// Whether launch t of a power iteration whose state says `done` (the launch that ended it, 0
// while it runs) has nothing to do.  Launch t itself may write done = t while other blocks
// of it still read the word, so both values must decide alike: warps of one block that
// disagreed would leave the others alone at the block's barriers.
MPAX_RULE bool power_round_over(int done, int t) { return done != 0 && done != t; }

}  // namespace mpax
