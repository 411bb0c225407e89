// Forward projector kernel: 1 j-blur strip(s) per thread, radii up to kLowR.
#include "forward.cuh"

namespace spect {
template cudaError_t forward_launch_ipt<1, false>(const ForwardArgs&, cudaStream_t);
template int forward_occupancy_ipt<1, false>(int, size_t);
}  // namespace spect
