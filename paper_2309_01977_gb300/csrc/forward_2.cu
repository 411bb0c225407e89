// Forward projector kernel: 1 j-blur strip(s) per thread, radii up to kMaxR.
#include "forward.cuh"

namespace spect {
template cudaError_t forward_launch_ipt<1, true>(const ForwardArgs&, cudaStream_t);
template int forward_occupancy_ipt<1, true>(int, size_t);
}  // namespace spect
