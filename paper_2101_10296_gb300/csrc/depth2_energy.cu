// Energy instantiations of the depth-2 kernel, the dispatch over its variants,
// and the records of its work lists.
#include <algorithm>

#include "depth2_impl.cuh"

namespace qaoa {

namespace {

// The records of a depth-2 work list (see RegWork): slot s of cone c at offset
// t = s - start[c] holds inner qubits R..n_in-1 in the low bits of t and block
// group t >> max(n_in - R, 0); register bits [2, nr), nr = min(n_in, R), are
// inner qubits and bits [nr, R) pick one of 2^(R - nr) blocks of the group.
__global__ void depth2_records_kernel(const DevCone *__restrict__ cones, const uint64_t *__restrict__ shell,
                                      const int32_t *__restrict__ slot_cone, const int64_t *__restrict__ start,
                                      int64_t slots, int R, int scale, uint32_t *__restrict__ cnt,
                                      float *__restrict__ wk) {
    const int S = 1 << (R - 2);
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < slots * S;
         e += int64_t(gridDim.x) * blockDim.x) {
        const int64_t sl = e % slots;
        const int k = int(e / slots);
        const int32_t sc = slot_cone[sl];
        const int ci = sc & 0x7fffffff;
        const DevCone *__restrict__ C = cones + ci;
        const int64_t t = sc >= 0 ? sl - start[ci] : 0;  // padding: the cone's first slot, weight 0
        const int nr = min(C->n_in, R), gb = max(C->n_in - R, 0), inner = nr - 2;
        const int64_t beta = ((t >> gb) << (R - nr)) + (k >> inner);
        float mult = 0.f;
        uint64_t h = 0;
        if (beta < C->n_blocks) h = shell_block(C, shell, uint32_t(beta), mult);
        for (int q = R; q < C->n_in; ++q)
            if ((t >> (q - R)) & 1) h ^= C->col[q];
        for (int b = 0; b < inner; ++b)
            if ((k >> b) & 1) h ^= C->col[2 + b];
        const uint64_t c0 = C->col[0], c1 = C->col[1];
        const uint64_t lo[4] = {0ull, c0, c1, c0 ^ c1};
        uint32_t w = 0, f = 0;  // without flips; after the first layer's
        for (int a = 0; a < 4; ++a) {
            w |= uint32_t(__popcll(lo[a] ^ h) * scale) << (8 * a);
            f |= uint32_t(__popcll(lo[a] ^ h ^ C->pw[0]) * scale) << (8 * a);
        }
        cnt[e] = w;
        cnt[slots * S + e] = f;
        wk[e] = sc >= 0 ? mult : 0.f;
    }
}

}  // namespace

cudaError_t build_depth2_records(const DevCone *cones, const uint64_t *shell, const int32_t *slot_cone,
                                 const int64_t *start, int64_t slots, int R, int cmax1, uint32_t *cnt, float *wk) {
    const int64_t n = slots << (R - 2);
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 65535);
    int scale = depth2_narrow(cmax1) ? 4 : 2;
    void *args[] = {&cones, &shell, &slot_cone, &start, &slots, &R, &scale, &cnt, &wk};
    return launch((const void *)depth2_records_kernel, int(blocks), 256, args, nullptr);
}

template cudaError_t depth2_prepare_r<kRegBitsEnergy, false>();
template const void *depth2_fn_r<kRegBitsEnergy, false>(int);
template cudaError_t launch_depth2_r<kRegBitsEnergy, false>(const RegLaunch &, int, cudaStream_t);

// instantiated in depth2_grad4.cu and depth2_grad5.cu
extern template cudaError_t depth2_prepare_r<4, true>();
extern template const void *depth2_fn_r<4, true>(int);
extern template cudaError_t launch_depth2_r<4, true>(const RegLaunch &, int, cudaStream_t);
extern template cudaError_t depth2_prepare_r<5, true>();
extern template const void *depth2_fn_r<5, true>(int);
extern template cudaError_t launch_depth2_r<5, true>(const RegLaunch &, int, cudaStream_t);

cudaError_t depth2_prepare() {
    cudaError_t e = depth2_prepare_r<kRegBitsEnergy, false>();
    if (e == cudaSuccess) e = depth2_prepare_r<4, true>();
    if (e == cudaSuccess) e = depth2_prepare_r<5, true>();
    return e;
}

int depth2_grid(bool grad, int rg, int cmax1, size_t smem) {
    const void *fn = !grad ? depth2_fn_r<kRegBitsEnergy, false>(cmax1)
                     : rg == 5 ? depth2_fn_r<5, true>(cmax1)
                               : depth2_fn_r<4, true>(cmax1);
    return occupancy_grid(fn, kRegBlock, smem);
}

cudaError_t launch_depth2(const RegLaunch &a, bool grad, int rg, int grid, cudaStream_t s) {
    if (!grad) return launch_depth2_r<kRegBitsEnergy, false>(a, grid, s);
    return rg == 5 ? launch_depth2_r<5, true>(a, grid, s) : launch_depth2_r<4, true>(a, grid, s);
}

}  // namespace qaoa
