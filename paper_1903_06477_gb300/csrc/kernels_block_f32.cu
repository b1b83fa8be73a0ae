// kernels_block_f32.cu -- FP32 instantiation of the block-team kernel for blocks of up to 1024 threads.
#include "kernels.cuh"

namespace sscs {
template const void* kblock_build<float, BLOCK_LARGE>();
}  // namespace sscs
