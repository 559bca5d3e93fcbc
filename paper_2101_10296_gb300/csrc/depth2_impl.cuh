// Instantiations of the depth-2 kernel for one register width.
#pragma once

#include "depth2_kernel.cuh"

namespace qaoa {

int occupancy_grid(const void *fn, int block, size_t smem);

template <int R, bool GRAD>
const void *depth2_fn_r(int cmax1) {
    return depth2_narrow(cmax1) ? (const void *)depth2_kernel<R, GRAD, true>
                                : (const void *)depth2_kernel<R, GRAD, false>;
}

template <int R, bool GRAD>
cudaError_t depth2_prepare_r() {
    cudaError_t e = cudaFuncSetAttribute((const void *)depth2_kernel<R, GRAD, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kRegMaxSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)depth2_kernel<R, GRAD, false>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kRegMaxSmem);
    return e;
}

template <int R, bool GRAD>
cudaError_t launch_depth2_r(const RegLaunch &a, int grid, cudaStream_t s) {
    const size_t sm = depth2_smem_bytes(a.jpt, a.cmax1, GRAD);
    if (depth2_narrow(a.cmax1))
        depth2_kernel<R, GRAD, true><<<grid, kRegBlock, sm, s>>>(a);
    else
        depth2_kernel<R, GRAD, false><<<grid, kRegBlock, sm, s>>>(a);
    return cudaGetLastError();
}

}  // namespace qaoa
