// walk_ordered1q.cu -- instances of the ordered walk with up to 1 i-particle per
// lane, nodes with quadrupoles (separate translation unit so the instances compile
// in parallel).
#include "walk_ordered.cuh"

namespace nb {
template cudaError_t launch_ordered_ipl<1, true>(cudaStream_t, const WalkArgs &, const WalkShape &, int);
}  // namespace nb
