// walk_coop3q.cu -- instances of the cooperative tree walk with up to 3
// i-particles per lane, nodes with quadrupoles (separate translation unit so
// the instances compile in parallel).
#include "walk_coop.cuh"

namespace nb {
template cudaError_t launch_coop_ipl<3, true>(cudaStream_t, const WalkArgs &, const WalkShape &, int);
}  // namespace nb
