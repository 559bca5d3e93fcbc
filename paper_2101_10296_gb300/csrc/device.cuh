// Device-side data layout shared by the kernels and the C-ABI launch code.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/qaoa.h"

namespace qaoa {

// One simulated cone (representative edge), as the kernels read it.
//
// Local qubits: 0 = u, 1 = v, then by (distance, vertex id).  `col[q]` has
// bit e set when cone edge e touches qubit q, so for a basis index z the
// word M(z) = XOR over set bits q of z of col[q] has bit e set exactly when
// edge e is cut, and the cut value is C(z) = popcount(M(z)).  M is linear
// over GF(2): M(hi | lo) = M(hi) ^ M(lo), which the kernels use to split z
// into a per-thread part and a per-register part.
struct alignas(16) DevCone {
    int32_t graph;   // graph index g
    int32_t n;       // qubits
    int32_t n_in;    // inner qubits: the only ones any mixer touches
    int32_t m;       // cut-word bits: cone edges, an edge of weight w counting |w|
    int32_t k[QAOA_MAX_P];  // layer l mixes qubits [0, k[l])
    double weight;   // orbit size
    int64_t rep;     // row of this cone in terms[]
    int64_t n_blocks;  // shell blocks: prod over shell classes of (size + 1)
    int32_t n_cls;     // shell classes
    int32_t cls_off;   // this cone's entries in the shell table
    uint64_t col[QAOA_MAX_CONE_QUBITS];
    uint64_t pw[QAOA_MAX_P];  // M of the qubits layer l mixes, [0, k[l])
    uint64_t neg;             // bits of negative-weight edges (already in the shell table's words)
};

// Shell table, per cone from cls_off.  n_cls < 0: an explicit list of
// n_blocks (shell word, multiplicity as float bits) pairs -- the blocks left
// after merging those related by the cone's symmetries.  Otherwise per
// class c of size s: word 0 = s,
// words 1..s+1 = XOR of col[] over the class's first 0..s qubits, words
// s+2..2s+2 = binomial(s, 0..s) as float bits.  Block beta of a cone is the
// mixed-radix number (n_0, n_1, ...) with 0 <= n_c <= s_c, least significant
// class first: its shell word is the XOR of the classes' prefix words for
// n_c and its multiplicity the product of binomial(s_c, n_c).
__device__ __forceinline__ uint64_t shell_block(const DevCone *__restrict__ C, const uint64_t *__restrict__ tab,
                                                uint32_t beta, float &mult) {
    if (C->n_cls < 0) {  // explicit list: (word, multiplicity bits) per block
        if (int64_t(beta) >= C->n_blocks) {
            mult = 0.f;
            return 0;
        }
        const uint64_t *e = tab + C->cls_off + 2 * size_t(beta);
        mult = __uint_as_float(uint32_t(e[1]));
        return e[0];
    }
    const uint64_t *t = tab + C->cls_off;
    uint64_t m = 0;
    float w = 1.f;
    for (int c = 0; c < C->n_cls; ++c) {
        const uint32_t sz = uint32_t(t[0]);
        const uint32_t q = beta / (sz + 1);
        const uint32_t nc = beta - q * (sz + 1);
        beta = q;
        m ^= t[1 + nc];
        w *= __uint_as_float(uint32_t(t[2 + sz + nc]));
        t += 2 * sz + 3;
    }
    mult = w;
    return m;
}

// Work list of the register-resident kernels.  An inner block of 2^n_in
// amplitudes takes G = 2^max(n_in - R, 0) threads (R register qubits per
// thread); when n_in < R a thread holds S = 2^(R - n_in) blocks.  A (cone,
// point) needs T_c = ceil(B / S) * G threads for its B shell blocks.  Cones
// are sorted by (G descending, graph) and packed back to back, T_c slots
// each; a graph change is padded to the next multiple of 32 slots, so every
// cone's first slot is aligned to min(G, 32) lanes and no warp spans two
// graphs.  A warp task covers 32 consecutive slots for `jpt` consecutive
// parameter points of that graph.
//
// Slot records: everything a thread derives from its slot before the first
// point does not depend on the parameters, so it is computed once at upload.
// For register index i = 4k + r of slot s's thread (r = bits 0-1: qubits u,
// v), rec_hi[k * slots + s] is the part of the cut word M(z_i) that does not
// involve qubits 0 and 1 -- the thread's inner qubits, its shell block's word
// and register bits 2.. -- and rec_wk[k * slots + s] the multiplicity of the
// block index i belongs to (0 past the cone's blocks and in padding slots).
// Words are uint32 when every cone has at most 32 cut bits, else uint64.
//
// The lists of the depth-2 kernel hold rec_cnt instead of rec_hi: the cut values
// themselves, of amplitudes 4k .. 4k + 3 in rec_cnt[k * slots + s], one byte
// each, scaled by 4 when every cone has at most 31 cut bits, else by 2; then
// the same after the first layer's flips (from row S = 2^(R-2) on).
struct RegWork {
    const DevCone *cones = nullptr;       // plan order
    const int32_t *slot_cone = nullptr;   // plan index of each slot's cone; bit 31: padding slot
    const int32_t *warp_graph = nullptr;  // the graph of each warp's slots
    const void *rec_hi = nullptr;         // slot records (above)
    const uint32_t *rec_cnt = nullptr;
    const float *rec_wk = nullptr;
    const uint4 *rec_cw = nullptr;        // depth-1 work lists: cut values and weights of two blocks
    int32_t n_cones = 0;
    int64_t slots = 0;                    // slots per point (with padding; a multiple of 32)
    int64_t warps = 0;                    // warps per point
};

// Per-point mixer data.  exp(-i beta X) = kappa (I - i tau X) with
// tau = tan(beta), kappa = cos(beta) when |tan(beta)| <= 1; otherwise the
// kernel applies exp(-i (beta - pi/2) X) (tau = -cot(beta), kappa = sin(beta))
// followed by exp(-i pi/2 X) = -i X, whose bit flip it tracks instead of
// applying (flip = 1).  kpow[k] = kappa^(2k), rounded once from FP64.
constexpr int kKpow = QAOA_MAX_CONE_QUBITS + 1;

struct RegLaunch {
    RegWork work;
    int64_t n_points;
    int32_t jpt;              // parameter points per warp task
    int32_t p;
    int32_t cmax1;            // phase-table row length (max cone edges + 1)
    const float2 *lut;        // [G][P][p][cmax1]  exp(-i gamma_l c)
    const float2 *mix;        // [G][P][p]         (tau_l, flip_l)
    const float *kpow;        // [G][P][p][kKpow]  kappa_l^(2k)
    double *energy;           // [G][P]
    double *grad;             // [G][P][2p] or null
    double *terms;            // [reps][P] or null
    int32_t *status;
    int32_t norm = 0;         // 1: the observable is the identity (terms = sum |psi|^2, energy unused)
};

struct PrepArgs {
    const double *params;     // [G][P][2p]
    int32_t G, p, cmax1;
    int64_t P;
    const double *half_edges; // [G]
    float2 *lut;
    float2 *mix;
    float *kpow;
    double *energy;
    double *grad;             // may be null
    double *terms;            // may be null
    int64_t n_reps;
    int32_t n_kpow;           // kappa powers filled per row: what the plan's mixers read (<= kKpow)
    float4 *cs;               // large-state cones: exact rotations [G][P][p]; null: none
    float2 *fa;               // their first layer's factored coefficient, hi and lo [G][P]; may be null
};

// launchers (kernels.cu)
// A launch that is prepared while the kernel before it in the stream drains
// (programmatic stream serialisation; after anything but a kernel it is a plain
// one); its kernel begins with wait_before(), so nothing runs earlier than it did.
// Measured, against plain launches of every kernel of an evaluation: 8x8 torus, p =
// 2, 128 points, allocation-free 16.8 -> 12.7 us a call; Erdos-Renyi n = 10,000, p =
// 1, 101 points, gradient 75.7 -> 69.6; cubic n = 16, p = 3, 14 points, energy 125 ->
// 115; n = 20, 4 points, gradient 375 -> 348; circulant n = 30, p = 4, 64 points,
// gradient 1233 -> 1217.
cudaError_t launch_after(const void *fn, int grid, int block, void **args, size_t smem, cudaStream_t s);
// A plain launch.  Both answer for the launch itself: cudaGetLastError() would also
// give an error that an earlier call met and reported (scratch refused by the
// allocator, say).
cudaError_t launch(const void *fn, int grid, int block, void **args, cudaStream_t s);
cudaError_t launch_prep(const PrepArgs &a, cudaStream_t s);
// wide = some cone has more than 32 edges (64-bit cut words).  Dynamic
// shared memory: 4 warps x jpt x p x cmax1 float2 (phase tables).
cudaError_t launch_reg_energy(const RegLaunch &a, bool wide, int grid, cudaStream_t s);
// rg: register qubits per thread of the adjoint kernel (4 or 5)
cudaError_t launch_reg_grad(const RegLaunch &a, bool wide, int rg, int grid, cudaStream_t s);
cudaError_t launch_cut_table(const DevCone *cone, uint8_t *out, int32_t n, int32_t *status, cudaStream_t s);
// occupancy-sized persistent grids for a given dynamic shared memory size
int reg_energy_grid(bool wide, size_t smem);
int sm_count();  // multiprocessors of the current device (cached)
// Dynamic shared memory a block may use when `blocks` blocks share one
// multiprocessor of the current device: the multiprocessor's shared memory
// split evenly, less what the hardware reserves per block (cached).
int smem_per_block(int blocks);
int reg_grad_grid(bool wide, size_t smem, int p, int rg);
cudaError_t reg_grad_prepare();
// Raises the register kernels' dynamic shared memory limit to kRegMaxSmem
// (once per device; called at upload, outside any stream capture).
cudaError_t reg_prepare();
constexpr int kRegBlock = 128;
constexpr int kRegMaxSmem = 96 * 1024;

#ifndef QAOA_REG_BITS_ENERGY
#define QAOA_REG_BITS_ENERGY 5
#endif
#ifndef QAOA_REG_BITS_GRAD
#define QAOA_REG_BITS_GRAD 4
#endif
// register qubits per thread of the energy and the adjoint kernels
constexpr int kRegBitsEnergy = QAOA_REG_BITS_ENERGY;
constexpr int kRegBitsGrad = QAOA_REG_BITS_GRAD;
constexpr int kLaneBits = 5;
// resident 128-thread blocks per SM the register allocation is sized for
// (the adjoint with four register qubits; with five it holds twice the
// amplitudes and is sized for two)
#ifndef QAOA_GRAD_MIN_BLOCKS
#define QAOA_GRAD_MIN_BLOCKS 4
#endif
constexpr int kGradMinBlocks = QAOA_GRAD_MIN_BLOCKS;
constexpr int kGradMinBlocks5 = 2;
constexpr int kEnergyMinBlocks = 3;
// largest inner part the register kernels take (both must fit)
constexpr int kRegMaxInner = (kRegBitsEnergy < kRegBitsGrad ? kRegBitsEnergy : kRegBitsGrad) + kLaneBits;

// The register kernels stage every lane's share of each output of a point
// (the energy, and with the adjoint the 2p derivatives) in shared memory and
// sum it over the warp for a group of points at once: per warp, outputs x
// group points x 32 lanes FP32 partials.
__host__ __device__ constexpr int reg_outputs(int p, bool grad) { return grad ? 1 + 2 * p : 1; }
__host__ __device__ constexpr int reg_group(int p, bool grad) {
    // at most 24 x 32 partials (3 KB) per warp, so that the point tables and
    // this buffer leave room for four blocks per SM
    return reg_outputs(p, grad) * 8 <= 24 ? 8
           : reg_outputs(p, grad) * 4 <= 24 ? 4
           : reg_outputs(p, grad) * 2 <= 24 ? 2 : 1;
}
// kappa powers a register kernel reads: kappa^(2k) for k <= its largest inner part
constexpr int kRegKpow = 10;
// 32-bit words of per-lane cone fields a register kernel keeps in shared
// memory: the layers' k (one byte each, two words), the adjoint's cut-value
// offset, and per layer the flip word M(F_l) as two words
__host__ __device__ constexpr int reg_lane_words(int p) { return 3 + 2 * p; }
// Depth-1 kernel (p1_kernel.cu): shell blocks per thread, and the resident
// blocks per SM its register allocation is sized for.  Its work lists hold
// per graph the shell blocks of all the graph's cones back to back, 16 to a
// slot; rec_cw[q * slots + s] holds blocks 2q and 2q + 1 of slot s: their count
// bytes (the cut value c_a of amplitude a = z_u + 2 z_v in byte a, scaled by 4
// unless a cone has 64 cut bits), then their weights W = multiplicity x orbit
// size x 2^-n; the amplitudes may be relabelled by X_u, X_v or both (a -> a xor
// f), with W negated for a single flip, so that c_0 is the middle one of the
// four; warp_graph as for the other lists.
constexpr int kP1Blocks = 16;
// Blocks per SM of the registers, and of the shared memory for the points of a
// task.  Measured on the 48-graph mix at 256 points, adjoint: 4, 5, 6 and 8
// blocks of registers 750, 736, 728 and 713 us, then 12 points per task (room
// for six blocks) instead of 4: 691 us; energy 361, 350, 347 and 351 us.
constexpr int kP1GradMinBlocks = 8;
constexpr int kP1EnergyMinBlocks = 6;
constexpr int kP1PointBlocks = 6;
// Points per reduction group of the depth-1 kernel (see reg_flush): four for
// the adjoint, whose three outputs would otherwise take 3 KB per warp
__host__ __device__ constexpr int reg_p1_group(bool grad) { return grad ? 4 : 8; }
// Bytes of a point's phase-table row in shared memory (see p1_kernel.cu).
constexpr int kP1RowSmall = 256, kP1RowMid = 512, kP1RowLarge = 544;
__host__ __device__ constexpr int p1_row_bytes(int cmax1) {
    return cmax1 <= 32 ? kP1RowSmall : cmax1 <= 64 ? kP1RowMid : kP1RowLarge;
}
// Dynamic shared memory of a depth-1 block: per warp jpt phase tables and (tau,
// kappa^4) pairs, the records of its 32 slots and the reduction buffer.
inline size_t reg_p1_smem_bytes(int jpt, int cmax1, bool grad) {
    return size_t(kRegBlock / 32) *
           (size_t(jpt) * (p1_row_bytes(cmax1) + sizeof(float2)) + size_t(kP1Blocks / 2) * 32 * sizeof(uint4) +
            size_t(reg_outputs(1, grad)) * reg_p1_group(grad) * 32 * sizeof(float));
}
int reg_p1_grid(bool grad, int cmax1, size_t smem);
cudaError_t reg_p1_prepare();
cudaError_t launch_reg_p1(const RegLaunch &a, bool grad, int grid, cudaStream_t s);

// Dynamic shared memory of a register-kernel block: per warp and point the
// phase tables (p x cmax1 float2), the mixer data (p float2) and the kappa
// powers (p x kRegKpow float) of jpt points, the reduction buffer, and the
// lanes' cone fields (reg_lane_words).
inline size_t reg_smem_bytes(int jpt, int p, int cmax1, bool grad) {
    return size_t(kRegBlock / 32) *
           (size_t(jpt) * p * (cmax1 + 1) * sizeof(float2) +
            (size_t(jpt) * p * kRegKpow + size_t(reg_outputs(p, grad)) * reg_group(p, grad) * 32 +
             size_t(reg_lane_words(p)) * 32) * sizeof(float));
}

// Depth-2 kernel (depth2_kernel.cuh; plans of depth 2 whose register cones are
// all pruned): bytes of one layer's phase-table row in shared memory (narrow:
// at most 31 cut bits, 32 entries), floats of a point's parameters, and a
// block's dynamic shared memory.
// Resident 128-thread blocks per SM: 128 registers for the energy and the
// adjoint with four register qubits, 255 with five (energy at 3 and 5 blocks:
// 752 and 842 against 734 us on four random cubic graphs of 2,000 vertices and
// 64 points; the adjoint with four at 3 and 5: 2858 and 2909 against 2677 us).
__host__ __device__ constexpr int depth2_blocks(bool grad, int rg) { return grad && rg == 5 ? 2 : 4; }
constexpr int kDepth2WideRow = 544;  // 2 x 68 entries, a multiple of 32 bytes
constexpr int kDepth2Params = 4 + kRegKpow;
__host__ __device__ constexpr bool depth2_narrow(int cmax1) { return cmax1 <= 32; }
__host__ __device__ constexpr int depth2_row_bytes(bool narrow) { return narrow ? 256 : kDepth2WideRow; }
inline size_t depth2_point_bytes(int cmax1) {
    return 2 * size_t(depth2_row_bytes(depth2_narrow(cmax1))) + kDepth2Params * sizeof(float);
}
inline size_t depth2_smem_bytes(int jpt, int cmax1, bool grad) {
    return size_t(kRegBlock / 32) * (size_t(jpt) * depth2_point_bytes(cmax1) +
                                     size_t(reg_outputs(2, grad)) * reg_group(2, grad) * 32 * sizeof(float));
}
// rg: register qubits per thread of the adjoint (4 or 5)
int depth2_grid(bool grad, int rg, int cmax1, size_t smem);
cudaError_t launch_depth2(const RegLaunch &a, bool grad, int rg, int grid, cudaStream_t s);
cudaError_t depth2_prepare();
// Fills the records of a depth-2 work list on the device (legacy default
// stream); start: device int64 per cone, its first slot.
cudaError_t build_depth2_records(const DevCone *cones, const uint64_t *shell, const int32_t *slot_cone,
                                 const int64_t *start, int64_t slots, int R, int cmax1, uint32_t *cnt, float *wk);

}  // namespace qaoa
