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
    RegLaunch arg = a;
    void *args[] = {&arg};
    return launch_after(depth2_fn_r<R, GRAD>(a.cmax1), grid, kRegBlock, args, sm, s);
}

}  // namespace qaoa
