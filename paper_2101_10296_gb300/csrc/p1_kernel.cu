// Depth-1 register kernel: energy, or energy and adjoint gradient, at p = 1.
//
// At p = 1 the mixer of the only layer acts, after gate pruning (Sec. 2.3),
// on the qubits within distance p - 1 = 0 of the edge: qubits 0 and 1 (u, v)
// alone.  Every other cone qubit stays classical, so a cone's state is a sum
// of independent 4-amplitude blocks, one per shell assignment (merged into
// shell blocks with multiplicities, see DevCone), and the amplitudes of one
// block never meet those of another.  The kernel therefore works on a flat
// list of blocks per graph (the blocks of all of the graph's representative
// cones, back to back): a thread takes kP1Blocks consecutive blocks and, for
// each parameter point, evolves them one after the other.  Only one block's
// amplitudes are live at a time, which leaves registers for more resident
// warps, and the per-point costs (table pointers, the output stash and the
// warp reductions) are shared by 16 blocks.
//
// Per block, with amplitude a = z_u + 2 z_v and c_a its cut value, and the
// record's weight W = (block multiplicity) x (orbit size) x 2^-n, all fixed
// at upload, in the stored form psi = kappa^2 2^-n/2 x of the general kernel:
//   s_a = exp(-i gamma c_a) from the phase table (|+> up to 2^-n/2),
//   x = (I - i tau X_v)(I - i tau X_u) s,
//   orbit-weighted <Z_u Z_v> = kappa^4 W (|x_0|^2 + |x_3|^2 - |x_1|^2 - |x_2|^2)  (Sec. 2.4),
// and E gets -1/2 of it.  Adjoint (co-state lambda = -1/2 Z_u Z_v psi, r =
// Z_u Z_v x):
//   dE/dbeta = 2 Im<lambda|X_u + X_v|psi>.  With r = Z_u Z_v x the two pair
//     terms of a qubit coincide, Im(conj r_i x_j) = Im(conj r_j x_i), so
//     Im<r|X_u + X_v|x> = 2 [Im(x_0* x_1) - Im(x_2* x_3) + Im(x_0* x_2) - Im(x_1* x_3)]
//     (half the products of the general form);
//   dE/dgamma = 2 Im<lambda|C|s> with the mixer undone on r.  Im<r|s> is
//     zero within every block (it equals <x|Z_u Z_v|x>, which is real), so C
//     may be shifted by any per-block constant: the block's first cut value
//     c_0, which drops one of the four terms.  The upload orders each block's
//     amplitudes so that c_0 is the one of its four cut values nearest their
//     middle (relabelling by X_u, X_v or both, which leave |+> and the mixers
//     unchanged and turn Z_u Z_v into -Z_u Z_v, +Z_u Z_v: the weight W takes
//     the sign).  That keeps the weights c_a - c_0 within about half the
//     block's spread, which limits how much of the FP32 state's rounding the
//     cancelling sum keeps.
// The block terms are accumulated per thread in four partial sums (blocks
// mod 4) and the lanes' shares of each point are summed with compensation
// (reg_flush).
//
// Two blocks at a time sit in packed FP32x2 registers (packed.cuh): every
// operation on a block is the same for both, one instruction for two, and the
// four partial sums are two pairs.  The phase table of a point keeps real and
// imaginary parts in rows of their own, and a block's record holds each cut value
// as its byte offset in a row, so that one byte permute makes an address and two
// 4-byte loads, free of bank conflicts, fill one half of the packed registers.
//
// Bound: the FP32 pipe's operand reads.  A block takes 62 FP32 lane operations
// with the adjoint; a packed instruction with three fresh operand pairs issues
// every 2.8 cycles (85 lane operations per clock and SM measured, 120 where one
// operand repeats, as tau does in the butterflies), and the kernel runs at 83.
// The 48-graph mix, 256 points: adjoint 736 -> 691 us, energy 392 -> 347 us
// against one block at a time with 8-byte loads; random n = 10,000, mean degree
// 4, every edge, 101 points: 87 -> 70 us.
#include "packed.cuh"
#include "reg_common.cuh"

namespace qaoa {

int occupancy_grid(const void *fn, int block, size_t smem);

namespace {

// Table row layouts: SMALL up to 32 entries (256 bytes: real parts, imaginary
// parts from byte 128), MID up to 64 (512 bytes, from byte 256), both with the
// count bytes scaled by 4 and the row at a multiple of 256, so that the byte
// replaces the lowest byte of the row's address; LARGE 65 entries, bytes unscaled.
template <int ROW>
struct P1Row {
    static constexpr bool kPerm = ROW != kP1RowLarge;
    static constexpr float kScale = kPerm ? 4.f : 1.f;
    static constexpr uint32_t kIm = ROW / 2;
    static __device__ __forceinline__ uint32_t addr(uint32_t w, int a, uint32_t row) {
        return kPerm ? __byte_perm(w, row, 0x7650u | uint32_t(a)) : row + (__byte_perm(w, 0u, 0x4440u | uint32_t(a)) << 2);
    }
    // entries of count byte a of two blocks
    static __device__ __forceinline__ C2 entry(uint32_t wa, uint32_t wb, int a, uint32_t row) {
        const uint32_t p = addr(wa, a, row), q = addr(wb, a, row);
        return C2{p2(lds1(p), lds1(q)), p2(lds1(p + kIm), lds1(q + kIm))};
    }
    // count byte a of two blocks as FP32 2^23 + kScale c (differences are exact)
    static __device__ __forceinline__ P2 count(uint32_t wa, uint32_t wb, int a) {
        return p2(__uint_as_float(__byte_perm(wa, 0x4B000000u, 0x7540u | uint32_t(a))),
                  __uint_as_float(__byte_perm(wb, 0x4B000000u, 0x7540u | uint32_t(a))));
    }
};

template <bool GRAD, int ROW>
__global__ void __launch_bounds__(kRegBlock, GRAD ? kP1GradMinBlocks : kP1EnergyMinBlocks)
    reg_p1_kernel(const RegLaunch L) {
    wait_before();
    using T = P1Row<ROW>;
    extern __shared__ __align__(256) unsigned char s_raw[];
    constexpr int kWarps = kRegBlock / 32, kPairs = kP1Blocks / 2;
    constexpr int NOUT = reg_outputs(1, GRAD);
    constexpr int G = reg_p1_group(GRAD);
    const int lane = threadIdx.x & 31;
    const int warp = warp_index();
    const RegWork &W = L.work;
    const int cm1 = L.cmax1;
    // per warp: the phase tables of the task's points, the slots' records, the
    // reduction buffer, and (tau, kappa^4) per point
    unsigned char *my_tab = s_raw + size_t(warp) * (L.jpt * ROW);
    uint4 *my_rec = reinterpret_cast<uint4 *>(s_raw + size_t(kWarps) * (L.jpt * ROW)) + warp * (kPairs * 32);
    float *red = reinterpret_cast<float *>(s_raw + size_t(kWarps) * (L.jpt * ROW + kPairs * 32 * sizeof(uint4))) +
                 warp * (NOUT * G * 32);
    float2 *my_mix = reinterpret_cast<float2 *>(s_raw + size_t(kWarps) * (L.jpt * ROW + kPairs * 32 * sizeof(uint4) +
                                                                          NOUT * G * 32 * sizeof(float))) +
                     warp * L.jpt;
    const uint32_t tab0 = static_cast<uint32_t>(__cvta_generic_to_shared(my_tab));
    const int64_t gw = int64_t(blockIdx.x) * kWarps + warp;
    const int64_t nw = int64_t(gridDim.x) * kWarps;
    const int64_t nblk = (L.n_points + L.jpt - 1) / L.jpt;
    const int64_t ntask = W.warps * nblk;
    for (int64_t task = gw; task < ntask; task += nw) {
        const int64_t jb = task / W.warps;
        const int64_t w = task - jb * W.warps;
        const int64_t j0 = jb * L.jpt;
        const int jn = int(L.n_points - j0 < L.jpt ? L.n_points - j0 : L.jpt);
        const int64_t slot = w * 32 + lane;  // < W.slots: the slot count is a multiple of 32
        const int gwarp = __ldg(W.warp_graph + w);
        const int64_t row0 = int64_t(gwarp) * L.n_points + j0;
        __syncwarp();  // the previous task's reads of the staged data are done
        {
            const float *__restrict__ src = reinterpret_cast<const float *>(L.lut + row0 * cm1);
            for (int j = 0; j < jn; ++j)
                for (int e = lane; e < cm1; e += 32) {
                    cp_async4(my_tab + j * ROW + 4 * e, src + 2 * (j * cm1 + e));
                    cp_async4(my_tab + j * ROW + T::kIm + 4 * e, src + 2 * (j * cm1 + e) + 1);
                }
            for (int e = lane; e < jn; e += 32) {
                cp_async4(&my_mix[e].x, &L.mix[row0 + e].x);
                cp_async4(&my_mix[e].y, L.kpow + (row0 + e) * kKpow + 2);  // kappa^(2 k), k = 2
            }
#pragma unroll
            for (int k = 0; k < kPairs; ++k) cp_async16(my_rec + k * 32 + lane, W.rec_cw + k * W.slots + slot);
        }
        cp_async_wait_all();
        __syncwarp();  // the staged data are complete and visible to the warp
        for (int jj = 0; jj < jn; ++jj) {
            const uint32_t row = tab0 + uint32_t(jj * ROW);
            const float2 tk = my_mix[jj];
            const float tau = tk.x;
            // sums of the blocks b mod 4: pairs (0, 1) and (2, 3)
            P2 e4[2] = {splat(0.f), splat(0.f)}, b4[2] = {splat(0.f), splat(0.f)}, g4[2] = {splat(0.f), splat(0.f)};
#pragma unroll
            for (int b = 0; b < kPairs; ++b) {
                const uint4 rc = my_rec[b * 32 + lane];
                const P2 wb = p2(__uint_as_float(rc.z), __uint_as_float(rc.w));
                C2 s[4], x[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    s[a] = T::entry(rc.x, rc.y, a, row);
                    x[a] = s[a];
                }
                mix01(x, tau);
                const P2 pos = fma2(x[0].r, x[0].r, fma2(x[0].i, x[0].i, fma2(x[3].r, x[3].r, mul2(x[3].i, x[3].i))));
                const P2 ngv = fma2(x[1].r, x[1].r, fma2(x[1].i, x[1].i, fma2(x[2].r, x[2].r, mul2(x[2].i, x[2].i))));
                e4[b & 1] = fma2(wb, add2(pos, neg(ngv)), e4[b & 1]);
                if constexpr (GRAD) {
                    // half of Im<r|X_u + X_v|x> (each pair term once)
                    P2 d = splat(0.f);
                    acc_imconj(d, x[0], x[1]);
                    acc_imconj(d, x[0], x[2]);
                    d = fma2(neg(x[2].r), x[3].i, d);
                    d = fma2(x[2].i, x[3].r, d);
                    d = fma2(neg(x[1].r), x[3].i, d);
                    d = fma2(x[1].i, x[3].r, d);
                    b4[b & 1] = fma2(wb, d, b4[b & 1]);
                    // r = Z_u Z_v x with the mixer undone: (I + i tau X) Z = Z (I - i tau X), so r is
                    // Z_u Z_v times a second forward mixing of x
                    mix01(x, tau);
                    P2 dg = splat(0.f);
#pragma unroll
                    for (int a = 1; a < 4; ++a) {
                        const C2 ra = a == 3 ? x[a] : neg(x[a]);
                        dg = fma2(add2(T::count(rc.x, rc.y, a), neg(T::count(rc.x, rc.y, 0))), imconj(ra, s[a]), dg);
                    }
                    g4[b & 1] = fma2(wb, dg, g4[b & 1]);
                }
            }
            const float k4 = tk.y;
            const int col = (lane + jj) & 31;
            auto sum4 = [](const P2(&v)[2]) { return (lo(v[0]) + hi(v[0])) + (lo(v[1]) + hi(v[1])); };
            red[(jj & (G - 1)) * 32 + col] = -0.5f * k4 * sum4(e4);
            if constexpr (GRAD) {
                // gamma_1, then beta_1 (the pair terms were counted once above)
                red[(1 * G + (jj & (G - 1))) * 32 + col] = -k4 * ((1.f / T::kScale) * sum4(g4));
                red[(2 * G + (jj & (G - 1))) * 32 + col] = -2.f * k4 * sum4(b4);
            }
            if ((jj & (G - 1)) == G - 1 || jj == jn - 1) {
                __syncwarp();
                reg_flush<NOUT>(red, NOUT, G, jj, lane, row0, 2, L.energy, L.grad);
                __syncwarp();
            }
        }
    }
}

template <bool GRAD>
const void *p1_fn(int cmax1) {
    switch (p1_row_bytes(cmax1)) {
        case kP1RowSmall: return (const void *)reg_p1_kernel<GRAD, kP1RowSmall>;
        case kP1RowMid: return (const void *)reg_p1_kernel<GRAD, kP1RowMid>;
        default: return (const void *)reg_p1_kernel<GRAD, kP1RowLarge>;
    }
}
const void *p1_fn(bool grad, int cmax1) { return grad ? p1_fn<true>(cmax1) : p1_fn<false>(cmax1); }

}  // namespace

int reg_p1_grid(bool grad, int cmax1, size_t smem) { return occupancy_grid(p1_fn(grad, cmax1), kRegBlock, smem); }

cudaError_t reg_p1_prepare() {
    cudaError_t e = cudaSuccess;
    for (int grad = 0; grad < 2; ++grad)
        for (int cmax1 : {32, 64, 65})
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(p1_fn(grad != 0, cmax1), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kRegMaxSmem);
    return e;
}

cudaError_t launch_reg_p1(const RegLaunch &a, bool grad, int grid, cudaStream_t s) {
    RegLaunch arg = a;
    void *args[] = {&arg};
    return launch_after(p1_fn(grad, a.cmax1), grid, kRegBlock, args, reg_p1_smem_bytes(a.jpt, a.cmax1, grad), s);
}

}  // namespace qaoa
