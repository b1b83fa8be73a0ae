// kernels_block_f32_small.cu -- FP32 instantiation of the block-team kernel for blocks of up to 512 threads.
#include "kernels.cuh"

namespace sscs {
template const void* kblock_build<float, BLOCK_SMALL>();
}  // namespace sscs
