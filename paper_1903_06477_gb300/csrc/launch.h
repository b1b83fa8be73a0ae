// launch.h -- host-visible handles of the solver kernels, defined in the
// per-precision translation units.
#pragma once

#include <cuda_runtime.h>

#include "solver.cuh"

namespace sscs {

template <typename T>
const void* kgrid_ptr();
template <typename T, int MAXT>
const void* kblock_build();  // one translation unit per precision and block-size bound
template <typename T>
cudaError_t launch_block(const void* kernel, int grid, int threads, size_t dyn, cudaStream_t st, const Args<T>* insts,
                         int B, int* queue, const DevSettings& S, int mode)
{
    void* args[] = {(void*)&insts, (void*)&B, (void*)&queue, (void*)&S, (void*)&mode};
    return cudaLaunchKernel(kernel, dim3(grid), dim3(threads), args, dyn, st);
}
cudaError_t launch_f2d(const float* in, double* out, long long n, cudaStream_t st);
cudaError_t launch_batch_handoff(const Args<float>* a32, const Args<double>* a64, int B, int mem, int resume,
                                 cudaStream_t st);
cudaError_t launch_batch_pack(const Args<double>* a64, int B, const long long* off, double* packed, cudaStream_t st);

}  // namespace sscs
