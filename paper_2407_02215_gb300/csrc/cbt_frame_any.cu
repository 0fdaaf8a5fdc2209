// The one-launch frames compiled for one vertex form.
#include <algorithm>

#include "cbt_frame.cuh"

namespace cbtgpu {

// compiled in their own files
extern template cudaError_t launch_frame_form<kFormF32>(const BatchDev&, int, cudaStream_t);
extern template int frame_blocks_form<kFormF32>();
extern template cudaError_t launch_frame1_form<kFormF32>(const BatchDev&, int, uint32_t, cudaStream_t);
extern template int frame1_blocks_form<kFormF32>();
extern template cudaError_t launch_frame_form<kFormF32Disp>(const BatchDev&, int, cudaStream_t);
extern template int frame_blocks_form<kFormF32Disp>();
extern template cudaError_t launch_frame1_form<kFormF32Disp>(const BatchDev&, int, uint32_t, cudaStream_t);
extern template int frame1_blocks_form<kFormF32Disp>();
extern template cudaError_t launch_frame_form<kFormFixed>(const BatchDev&, int, cudaStream_t);
extern template int frame_blocks_form<kFormFixed>();
extern template cudaError_t launch_frame1_form<kFormFixed>(const BatchDev&, int, uint32_t, cudaStream_t);
extern template int frame1_blocks_form<kFormFixed>();
extern template cudaError_t launch_frame_form<kFormF64>(const BatchDev&, int, cudaStream_t);
extern template int frame_blocks_form<kFormF64>();
extern template cudaError_t launch_frame1_form<kFormF64>(const BatchDev&, int, uint32_t, cudaStream_t);
extern template int frame1_blocks_form<kFormF64>();
extern template cudaError_t launch_frame_form<kFormSphere>(const BatchDev&, int, cudaStream_t);
extern template int frame_blocks_form<kFormSphere>();
extern template cudaError_t launch_frame1_form<kFormSphere>(const BatchDev&, int, uint32_t, cudaStream_t);
extern template int frame1_blocks_form<kFormSphere>();

template cudaError_t launch_frame_form<kFormAny>(const BatchDev&, int, cudaStream_t);
template int frame_blocks_form<kFormAny>();

cudaError_t launch_wait_selftest(BatchGlobals* bg, int blocks, int limit, cudaStream_t s) {
    return launch_coop<BatchGlobals*, int>(k_wait_selftest, blocks, s, bg, limit);
}

// The grid of a launch has to be resident whichever form it runs as.
int frame_blocks_per_sm() {
    return std::min({frame_blocks_form<kFormAny>(), frame_blocks_form<kFormF32>(), frame_blocks_form<kFormF32Disp>(),
                     frame_blocks_form<kFormFixed>(), frame_blocks_form<kFormF64>(), frame_blocks_form<kFormSphere>()});
}

int frame1_blocks_per_sm() {
    return std::min({frame1_blocks_form<kFormF32>(), frame1_blocks_form<kFormF32Disp>(),
                     frame1_blocks_form<kFormFixed>(), frame1_blocks_form<kFormF64>(),
                     frame1_blocks_form<kFormSphere>()});
}

cudaError_t launch_frame(const BatchDev& bt, int form, int grid, cudaStream_t s) {
    switch (form) {
        case kFormF32: return launch_frame_form<kFormF32>(bt, grid, s);
        case kFormF32Disp: return launch_frame_form<kFormF32Disp>(bt, grid, s);
        case kFormFixed: return launch_frame_form<kFormFixed>(bt, grid, s);
        case kFormF64: return launch_frame_form<kFormF64>(bt, grid, s);
        case kFormSphere: return launch_frame_form<kFormSphere>(bt, grid, s);
        default: return launch_frame_form<kFormAny>(bt, grid, s);
    }
}

cudaError_t launch_frame1(const BatchDev& bt, int form, int grid, uint32_t tbits, cudaStream_t s) {
    switch (form) {
        case kFormF32Disp: return launch_frame1_form<kFormF32Disp>(bt, grid, tbits, s);
        case kFormFixed: return launch_frame1_form<kFormFixed>(bt, grid, tbits, s);
        case kFormF64: return launch_frame1_form<kFormF64>(bt, grid, tbits, s);
        case kFormSphere: return launch_frame1_form<kFormSphere>(bt, grid, tbits, s);
        default: return launch_frame1_form<kFormF32>(bt, grid, tbits, s);
    }
}

}  // namespace cbtgpu
