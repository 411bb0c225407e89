// Back blur kernels: attenuation planes read from global memory, radii up to kLowR.
#include "blur_back.cuh"

namespace spect {
template cudaError_t launch_blur_back_v<false, false>(const BlurBackArgs&, cudaStream_t);
template int blur_back_blocks_v<false, false>(const BackTiling&);
}  // namespace spect
