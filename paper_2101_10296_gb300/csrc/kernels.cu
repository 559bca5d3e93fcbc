// Register-resident cone kernels for sm_103a.
//
// Per (cone, parameter point) the kernel evolves the cone's state vector
// |+>^n through p layers of U_P(gamma_l) = exp(-i gamma_l C) and
// U_B(beta_l) = prod exp(-i beta_l X_q) (Sec. 2.2) and reduces
// <Z_0 Z_1> = sum_z |psi_z|^2 (-1)^(z_0 xor z_1) (Sec. 2.3-2.4).
//
// Gate pruning (Sec. 2.3, reverse causal cone): a mixer of layer l only acts
// on qubits within distance p-l of the edge -- elsewhere it commutes through
// the observable and cancels -- so layer l mixes qubits [0, k_l) and the
// outermost shell (distance p) is never mixed.  Those shell qubits therefore
// stay classical: for each assignment of them the remaining amplitudes
// evolve independently.  A thread holds 2^R amplitudes (the R lowest qubits)
// in registers; qubits R..R+4 live on lane bits of the warp (butterflies via
// shuffles); higher qubits are shell bits that index independent threads.
// This is the full 2^n state vector, computed in 2^(n-R) register-sized
// slices that never leave the SM.
//
// Stored form.  The registers hold s with psi = K X^F s: K is a scalar whose
// |K|^2 = sigma each lane tracks in FP32 from a table rounded once from FP64,
// and F is a set of bit flips.  exp(-i beta X) = kappa (I - i tau X) with
// |tau| <= 1 (tau = tan beta), or, when |tan beta| > 1, the same form for
// beta - pi/2 times exp(-i pi/2 X) = -i X; that X is not applied but added
// to F.  Each butterfly output is then two FMAs.  A phase lookup needs
// C(z xor F), which is popcount(M(z) ^ M(F)) since the cut word M is linear,
// so F costs one XOR into the per-thread part of M per flipped layer.
// Every layer flips qubits 0 and 1 together, so Z_0 Z_1 never changes sign.
//
// Numerics: complex64 amplitudes and FP32 arithmetic; the phase table
// exp(-i gamma c), tan and the kappa powers are computed in FP64 and rounded
// once; lane partial sums are reduced across the warp in FP32 and
// accumulated across warps, cones and orbits in FP64 (atomicAdd).
#include <algorithm>
#include <cstdint>
#include <map>
#include <set>
#include <mutex>
#include <tuple>

#include "cone_kernel.cuh"

namespace qaoa {
namespace {

// Per-call tables and output initialisation.  Bound: the FP64 pipe (two lanes
// per clock and SM), and for small calls its latency, so the work is spread
// over the SMs in blocks of one or two warps and a table row is cut into
// `parts` segments while the rows alone would leave SMs idle.  The first
// row_blocks blocks fill phase-table rows, the next mix_blocks the mixer
// tables, the rest initialise the outputs.
// Measured: the whole call of an 8x8 torus at p = 2, 128 points, energy 35 -> 17
// us (256 rows of 24 entries had sat on one SM, 33 kappa powers each where 10
// are read); the 48-graph mix at p = 1, 256 points 763 -> 749 us.
// The large-state kernels' rotations come from the same sincos (a launch of their
// own before: 59.1 -> 56.8 us for the 5x5 torus, p = 3, 4 points, energy).
constexpr int kPrepBlock = 64;

__global__ void __launch_bounds__(kPrepBlock) prep_kernel(const PrepArgs a, int parts, int row_blocks, int mix_blocks) {
    wait_before();
    const int64_t GP = int64_t(a.G) * a.P;
    const int p2 = 2 * a.p;
    if (int(blockIdx.x) < row_blocks) {
        // exp(-i gamma c) of one (graph, point, layer), c in the thread's segment: the segment's first
        // entry, then the recurrence z_(c+1) = z_c exp(-i gamma) in FP64 (after at most 64 steps its
        // rounding error, ~1e-14, is far below the FP32 table's own).  The first entry is not sincos of
        // the rounded product gamma c0 (off by |gamma c0| 2^-53, more than the table's own rounding from
        // |gamma| = 1e7 on): up to 2^20 the product's error is put back, beyond it exp(-i gamma), whose
        // argument sincos reduces exactly, is raised to the power by squarings.  (Squarings throughout
        // wait for the first sincos instead of running beside it: 11.7 against 10.4 us a replayed
        // evaluation of the 8x8 torus, p = 2, 8 points; 72.5 against 71.7 for Erdos-Renyi n = 10,000,
        // p = 1, 101 points, gradient.)
        const int64_t t = int64_t(blockIdx.x) * kPrepBlock + threadIdx.x;
        const int64_t r = t / parts;
        if (r >= GP * a.p) return;
        const int part = int(t - r * parts);
        const int64_t gj = r / a.p;
        const double gamma = a.params[gj * p2 + (r - gj * a.p)];
        double sn, cs;
        sincos(gamma, &sn, &cs);
        const int len = (a.cmax1 + parts - 1) / parts;
        const int c0 = part * len, c1 = min(c0 + len, a.cmax1);
        float2 *row = a.lut + r * a.cmax1;
        double zr = 1.0, zi = 0.0;
        if (c0 > 0) {
            const double first = gamma * double(c0);
            if (fabs(gamma) < 0x1p20) {
                const double e = fma(gamma, double(c0), -first);  // the product's rounding error, below 2^-27
                double se, ce;
                sincos(first, &se, &ce);
                zr = fma(-se, e, ce);
                zi = -fma(ce, e, se);
            } else {
                double br = cs, bi = -sn;
                for (int k = c0;;) {
                    if (k & 1) {
                        const double nr = fma(zr, br, -(zi * bi));
                        zi = fma(zr, bi, zi * br);
                        zr = nr;
                    }
                    k >>= 1;
                    if (k == 0) break;
                    const double nr = fma(br, br, -(bi * bi));
                    bi = 2.0 * (br * bi);
                    br = nr;
                }
            }
        }
        for (int c = c0; c < c1; ++c) {
            row[c] = make_float2(float(zr), float(zi));
            const double nr = fma(zr, cs, zi * sn);  // (zr + i zi)(cos gamma - i sin gamma)
            zi = fma(zi, cs, -(zr * sn));
            zr = nr;
        }
        return;
    }
    const int64_t u = int64_t(int(blockIdx.x) - row_blocks) * kPrepBlock + threadIdx.x;
    if (int(blockIdx.x) < row_blocks + mix_blocks) {
        if (u >= GP * a.p) return;
        const int64_t gj = u / a.p, l = u - gj * a.p;
        double sn, cs;
        sincos(a.params[gj * p2 + a.p + l], &sn, &cs);
        const bool flip = fabs(sn) > fabs(cs);
        const double tau = flip ? -cs / sn : sn / cs;
        const double k2 = flip ? sn * sn : cs * cs;
        a.mix[u] = make_float2(float(tau), flip ? 1.f : 0.f);
        double pw = 1.0;
        for (int k = 0; k < a.n_kpow; ++k) {
            a.kpow[u * kKpow + k] = float(pw);
            pw *= k2;
        }
        // (cos beta, sin beta) for the large-state kernels' exact rotations, each as an FP32 pair hi + lo.
        // Rounded to one FP32 number each, the gate becomes r exp(-i beta' X) with beta' - beta up to
        // ~4e-8: the same shift for every amplitude, layer after layer, which a small gradient (near a
        // stationary point, a second derivative times that shift) feels in full.  The lo parts (two more
        // FMAs per output) take the shift away; what remains is per-operation rounding.
        if (a.cs) {
            const float ch = float(cs), sh = float(sn);
            a.cs[u] = make_float4(ch, sh, float(cs - double(ch)), float(sn - double(sh)));
        }
        if (a.fa && l == 0) {
            // the first layer's factored coefficient: tan beta, or cot beta where |tan beta| > 1 (tau's
            // choice and rounded hi part, but for the sign), with its FP32 rounding error
            const double f = flip ? cs / sn : sn / cs;
            const float fh = float(f);
            a.fa[gj] = make_float2(fh, float(f - double(fh)));
        }
        return;
    }
    const int64_t first = u - int64_t(mix_blocks) * kPrepBlock;
    const int64_t stride = int64_t(int(gridDim.x) - row_blocks - mix_blocks) * kPrepBlock;
    for (int64_t i = first; i < GP; i += stride) a.energy[i] = a.half_edges[i / a.P];
    if (a.grad)
        for (int64_t i = first; i < GP * p2; i += stride) a.grad[i] = 0.0;
    if (a.terms)
        for (int64_t i = first; i < a.n_reps * a.P; i += stride) a.terms[i] = 0.0;
}

// C(z) for every z of one cone, through the same cut-word routine.
template <typename MT>
__global__ void cut_table_kernel(const DevCone *__restrict__ C, uint8_t *__restrict__ out, int32_t n,
                                 int32_t *status) {
    constexpr int R = kRegBitsEnergy;
    const int64_t threads = int64_t(1) << (n > R ? n - R : 0);
    const int nreg = n < R ? n : R;
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < threads;
         t += int64_t(gridDim.x) * blockDim.x) {
        CutWords<R, MT> cw;
        cw.init(C, n, t);
        cw.visit([&](int i, int c) {
            if (!(i >> nreg)) out[(t << R) | i] = uint8_t(c);
        });
    }
    if (n != C->n && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, 1);
}

}  // namespace

// Persistent grid size for (kernel, block, dynamic shared memory) on the
// current device, computed once and cached (the runtime query is not free
// and small evaluations are dominated by host overhead).
int occupancy_grid(const void *fn, int block, size_t smem) {
    struct Key {
        const void *fn;
        int block, dev;
        size_t smem;
        bool operator<(const Key &o) const {
            return std::tie(fn, block, dev, smem) < std::tie(o.fn, o.block, o.dev, o.smem);
        }
    };
    static std::mutex mu;
    static std::map<Key, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    const Key key{fn, block, dev, smem};
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) return it->second;
    }
    int sms = 0, per = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, block, smem);
    if (per < 1) per = 1;
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = sms * per;
    return sms * per;
}

int sm_count() {
    static std::mutex mu;
    static std::map<int, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(dev);
    if (it != cache.end()) return it->second;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cache[dev] = sms;
    return sms;
}

int smem_per_block(int blocks) {
    static std::mutex mu;
    static std::map<std::pair<int, int>, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find({dev, blocks});
    if (it != cache.end()) return it->second;
    int per_sm = 0, reserved = 0;
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    const int v = std::max(0, per_sm / std::max(blocks, 1) - reserved);
    cache[{dev, blocks}] = v;
    return v;
}

cudaError_t launch_after(const void *fn, int grid, int block, void **args, size_t smem, cudaStream_t s) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(unsigned(grid));
    c.blockDim = dim3(unsigned(block));
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &attr;
    c.numAttrs = 1;
    return cudaLaunchKernelExC(&c, fn, args);
}

cudaError_t launch(const void *fn, int grid, int block, void **args, cudaStream_t s) {
    return cudaLaunchKernel(fn, dim3(unsigned(grid)), dim3(unsigned(block)), args, 0, s);
}

cudaError_t launch_prep(const PrepArgs &a, cudaStream_t s) {
    const int64_t rows = int64_t(a.G) * a.P * a.p;
    // segments per table row while rows x segments fit one block per SM
    int parts = 1;
    while (parts < 8 && rows * parts * 2 <= int64_t(sm_count()) * kPrepBlock) parts *= 2;
    auto blocks = [](int64_t threads) { return (threads + kPrepBlock - 1) / kPrepBlock; };
    const int64_t row_blocks = blocks(rows * parts), mix_blocks = blocks(rows);
    int64_t out = int64_t(a.G) * a.P * (a.grad ? 2 * a.p : 1);
    if (a.terms) out = std::max<int64_t>(out, a.n_reps * a.P);
    const int64_t out_blocks = std::min<int64_t>(blocks(out), int64_t(sm_count()) * 8);
    if (row_blocks + mix_blocks + out_blocks > INT32_MAX) return cudaErrorInvalidValue;
    PrepArgs arg = a;
    int rb = int(row_blocks), mb = int(mix_blocks);
    void *args[] = {&arg, &parts, &rb, &mb};
    return launch_after((const void *)prep_kernel, int(row_blocks + mix_blocks + out_blocks), kPrepBlock, args, 0, s);
}

int reg_energy_grid(bool wide, size_t smem) {
    return wide ? occupancy_grid((const void *)reg_cone_kernel<kRegBitsEnergy, uint64_t, false, 0>, kRegBlock, smem)
                : occupancy_grid((const void *)reg_cone_kernel<kRegBitsEnergy, uint32_t, false, 0>, kRegBlock, smem);
}
cudaError_t reg_prepare() {
    static std::mutex mu;
    static std::set<int> done;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (done.count(dev)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute((const void *)reg_cone_kernel<kRegBitsEnergy, uint32_t, false, 0>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kRegMaxSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)reg_cone_kernel<kRegBitsEnergy, uint64_t, false, 0>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kRegMaxSmem);
    if (e == cudaSuccess) e = reg_grad_prepare();
    if (e == cudaSuccess) e = reg_p1_prepare();
    if (e == cudaSuccess) e = depth2_prepare();
    if (e == cudaSuccess) done.insert(dev);
    return e;
}

cudaError_t launch_reg_energy(const RegLaunch &a, bool wide, int grid, cudaStream_t s) {
    const size_t sm = reg_smem_bytes(a.jpt, a.p, a.cmax1, false);
    RegLaunch arg = a;
    void *args[] = {&arg};
    const void *fn = wide ? (const void *)reg_cone_kernel<kRegBitsEnergy, uint64_t, false, 0>
                          : (const void *)reg_cone_kernel<kRegBitsEnergy, uint32_t, false, 0>;
    return launch_after(fn, grid, kRegBlock, args, sm, s);
}

cudaError_t launch_cut_table(const DevCone *cone, uint8_t *out, int32_t n, int32_t *status, cudaStream_t s) {
    int64_t threads = int64_t(1) << (n > kRegBitsEnergy ? n - kRegBitsEnergy : 0);
    int64_t blocks = (threads + 127) / 128;
    if (blocks > 65535) blocks = 65535;
    void *args[] = {&cone, &out, &n, &status};
    return launch((const void *)cut_table_kernel<uint64_t>, int(blocks), 128, args, s);
}

}  // namespace qaoa
