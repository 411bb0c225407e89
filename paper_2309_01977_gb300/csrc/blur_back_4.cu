// Back blur kernels: attenuation planes staged in shared memory, radii up to kMaxR.
#include "blur_back.cuh"

namespace spect {
template cudaError_t launch_blur_back_v<true, true>(const BlurBackArgs&, cudaStream_t);
template int blur_back_blocks_v<true, true>(const BackTiling&);
}  // namespace spect
