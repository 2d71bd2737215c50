// walk_ordered2q.cu -- instances of the ordered walk with up to 2 i-particles per
// lane, nodes with quadrupoles (separate translation unit so the instances compile
// in parallel).
#include "walk_ordered.cuh"

namespace nb {
template cudaError_t launch_ordered_ipl<2, true>(cudaStream_t, const WalkArgs &, const WalkShape &, int);
}  // namespace nb
