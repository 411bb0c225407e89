// Back blur kernels: attenuation planes staged in shared memory, radii up to kLowR.
#include "blur_back.cuh"

namespace spect {
template cudaError_t launch_blur_back_v<true, false>(const BlurBackArgs&, cudaStream_t);
template int blur_back_blocks_v<true, false>(const BackTiling&);
}  // namespace spect
