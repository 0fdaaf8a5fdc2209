// The one-launch frames compiled for one vertex form.
#include "cbt_frame.cuh"

namespace cbtgpu {

template cudaError_t launch_frame_form<kFormFixed>(const BatchDev&, int, cudaStream_t);
template int frame_blocks_form<kFormFixed>();
template cudaError_t launch_frame1_form<kFormFixed>(const BatchDev&, int, uint32_t, cudaStream_t);
template int frame1_blocks_form<kFormFixed>();

}  // namespace cbtgpu
