// walk_ordered1.cu -- instances of the ordered walk with up to 1 i-particle per
// lane, monopole nodes (separate translation unit so the instances compile
// in parallel).
#include "walk_ordered.cuh"

namespace nb {
template cudaError_t launch_ordered_ipl<1, false>(cudaStream_t, const WalkArgs &, const WalkShape &, int);
}  // namespace nb
