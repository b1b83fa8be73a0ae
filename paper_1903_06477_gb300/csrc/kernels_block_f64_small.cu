// kernels_block_f64_small.cu -- FP64 instantiation of the block-team kernel for blocks of up to 512 threads.
#include "kernels.cuh"

namespace sscs {
template const void* kblock_build<double, BLOCK_SMALL>();
}  // namespace sscs
