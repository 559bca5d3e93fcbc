// Large-state cones, core-tile schedule.
//
// In a pruned cone, layer l mixes the qubits within distance p - l of the
// edge (Sec. 2.3), so the outer inner qubits -- those at distance p - 1 --
// are mixed by the first layer only.  When every later layer mixes only the
// T = RB + 5 core qubits [0, T) of a warp tile, the state after the first
// layer's mixer decouples into 2^(n_in - T) independent core tiles:
//
//   forward   outer passes build V_U exp(-i gamma_1 C)|+> (V_U: the first
//             mixer on the outer qubits), five outer qubits per pass; the
//             core pass loads one tile, applies the first mixer to the core
//             qubits, runs layers 2..p in registers and reduces <Z_0 Z_1>.
//   adjoint   the core pass continues with lambda = -1/2 Z_0 Z_1 psi, runs
//             both states back through layers p..2 (the derivative terms of
//             those layers), takes the first mixer's terms of the core
//             qubits, un-mixes lambda alone on the core qubits and stores it
//             in place of psi.  Outer passes un-mix lambda on the outer
//             qubits; the last one evaluates the first layer's phase term
//             and the outer qubits' mixer terms against the state before the
//             first mixer, exp(-i gamma_1 C)|+>, which is known in closed
//             form (amplitude = phase-table entry of C(z)).
//
// Both derivative identities rest on the first mixer commuting with every
// X_q it contains: <lambda|X_q|psi> is the same before and after it.  Only
// one state block per item is ever stored (the general schedule stores psi
// and lambda), and psi is never written back after the core pass.
//
// Storage: address bits 0..4 = qubits RB..RB+4, bits 5..RB+4 = qubits
// 0..RB-1, higher bits = the outer qubits themselves.  A core tile is one
// warp: lane = qubits RB..RB+4, register i = qubits 0..RB-1, so the most
// often mixed qubits 0, 1 are register butterflies and <Z_0 Z_1>'s sign is a
// compile-time function of the register.  Every load and store moves 256
// contiguous bytes per warp instruction.
#include <cuda.h>  // CUtensorMap and its enums (the encoder itself is fetched from the driver at run time)

#include <mutex>
#include <set>

#include "big.cuh"
#include "big_common.cuh"

namespace qaoa {
namespace {

// The first layer's mixer in factored form, without bit flips:
// exp(-i beta X) = kappa D with D = I - i a X (a = tan beta, kappa = cos beta)
// when |tan beta| <= 1, else D = a I - i X (a = cot beta, kappa = sin beta);
// its inverse up to the same factor, D' = exp(+i beta X) / kappa, is I + i a X
// or a I + i X.  Two FMAs per output amplitude in both cases (the exact
// rotation takes four).  Only the first layer uses it: every state of the
// schedule then carries one known factor, kappa^(n_in) per amplitude of psi,
// and every derivative term is taken either before any of the first mixer
// is undone or after all of it, so (D'D = 1 / kappa^2 per qubit) nothing else
// changes.
//
// With LO the coefficient is a + alo (FP32 hi and lo parts of the FP64 value),
// one FMA more per output: a single FP32 a is tan or cot of a slightly
// different angle (|delta beta| ~ 1e-8), which moves the gradient by the
// Hessian times that shift -- as large as the whole 1e-4 tolerance at points
// where |grad E| ~ 1e-3 |E|.  The adjoint's passes use it; the energy's need
// not (E moves by grad E . delta beta).
//
// Here on one amplitude, its real and imaginary parts a packed pair: the partner
// enters with the halves exchanged.
template <bool B, bool INV, bool LO>
__device__ __forceinline__ P2 fmix(P2 me, P2 o, float a, float alo) {
    const P2 so = swap(o);
    if (!B) {
        const P2 ox = LO ? fma2(INV ? p2(-alo, alo) : p2(alo, -alo), so, me) : me;
        return fma2(INV ? p2(-a, a) : p2(a, -a), so, ox);
    }
    const float2 h = halves(so);
    const P2 io = INV ? p2(-h.x, h.y) : p2(h.x, -h.y);  // i o, or -i o
    return fma2(splat(a), me, LO ? fma2(splat(alo), me, io) : io);
}

// D (or D') on register bits [r0, r1).
template <int NR, bool B, bool INV, bool LO>
__device__ __forceinline__ void fmix_regs(P2 (&x)[NR], int r0, int r1, float a, float alo) {
#pragma unroll
    for (int rb = 0; (1 << rb) < NR; ++rb) {
        if (rb >= r0 && rb < r1) {
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                if (i & (1 << rb)) continue;
                const int i2 = i | (1 << rb);
                const P2 u = x[i], v = x[i2];
                x[i] = fmix<B, INV, LO>(u, v, a, alo);
                x[i2] = fmix<B, INV, LO>(v, u, a, alo);
            }
        }
    }
}

// The first layer's a (hi and lo), form (b: the a I - i X form) and
// kappa^(2 n_in) of one (graph, point): a and the form from the register
// kernels' mixer tables, the lo part from L.fa where the launch has it.
struct FirstMix {
    float a, alo, k2n;
    bool b;
};
__device__ __forceinline__ FirstMix first_mix(const BigLaunch &L, int64_t gj, int n_in) {
    const float2 m = __ldg(L.mix + gj * L.p);  // (tau, flip) of the factored form with bit flips
    FirstMix f;
    f.b = m.y != 0.f;
    f.a = f.b ? -m.x : m.x;  // flip form: tau = -cot beta
    f.alo = L.fa ? __ldg(L.fa + gj).y : 0.f;
    f.k2n = __ldg(L.kpow + gj * L.p * kKpow + n_in);
    return f;
}

// The same factored form for layer l mixing k qubits (kappa_l^(2k) in k2n).
__device__ __forceinline__ FirstMix layer_mix(const BigLaunch &L, int64_t gj, int l, int k) {
    const float2 m = __ldg(L.mix + gj * L.p + l);
    FirstMix f;
    f.b = m.y != 0.f;
    f.a = f.b ? -m.x : m.x;
    f.alo = 0.f;
    f.k2n = __ldg(L.kpow + (gj * L.p + l) * kKpow + k);
    return f;
}

template <int NR, bool INV, bool LO>
__device__ __forceinline__ void first_mix_regs(P2 (&x)[NR], int r0, int r1, const FirstMix &f) {
    if (f.b)
        fmix_regs<NR, true, INV, LO>(x, r0, r1, f.a, f.alo);
    else
        fmix_regs<NR, false, INV, LO>(x, r0, r1, f.a, f.alo);
}

// ---------------------------------------------------------------- core pass
// The tile in packed FP32x2 pairs (packed.cuh): C2 number h holds registers h
// and h + NR/2, every operation of the sweep is one instruction for both, and
// the highest register qubit's partner is the other half.  Sums that run over
// the registers in order (the observable, the derivative terms) take the lower
// halves first, then the upper ones.

// fmix on two amplitudes
template <bool B, bool INV, bool LO>
__device__ __forceinline__ C2 fmix2(const C2 &me, const C2 &o, float a, float alo) {
    const P2 oi = INV ? neg(o.i) : o.i, nor = INV ? o.r : neg(o.r);  // -i o, or i o
    if (!B) {
        const P2 ox = LO ? fma2(splat(alo), oi, me.r) : me.r, oy = LO ? fma2(splat(alo), nor, me.i) : me.i;
        return C2{fma2(splat(a), oi, ox), fma2(splat(a), nor, oy)};
    }
    const P2 px = LO ? fma2(splat(alo), me.r, oi) : oi, py = LO ? fma2(splat(alo), me.i, nor) : nor;
    return C2{fma2(splat(a), me.r, px), fma2(splat(a), me.i, py)};
}

// op on register qubits [0, nr) and lane qubits [0, nl)
template <int NP, class F>
__device__ __forceinline__ void on_qubits(C2 (&x)[NP], int nr, int nl, F &&op) {
#pragma unroll
    for (int q = 0; (1 << q) <= NP; ++q)
        if (q < nr) on_reg<NP>(x, q, op);
#pragma unroll 1
    for (int lb = 0; lb < nl; ++lb) {
#pragma unroll
        for (int h = 0; h < NP; ++h) x[h] = op(x[h], shfl_xor(x[h], 1 << lb));
    }
}

template <int NP, bool INV, bool LO>
__device__ __forceinline__ void first_mix2(C2 (&x)[NP], int nr, int nl, const FirstMix &f) {
    if (__any_sync(kFull, f.b))  // the same in every lane: the vote tells the compiler
        on_qubits<NP>(x, nr, nl, [&](const C2 &u, const C2 &v) { return fmix2<true, INV, LO>(u, v, f.a, f.alo); });
    else
        on_qubits<NP>(x, nr, nl, [&](const C2 &u, const C2 &v) { return fmix2<false, INV, LO>(u, v, f.a, f.alo); });
}

// <Z_0 Z_1> sign of register i (qubits 0 and 1 are register bits 0 and 1).
__host__ __device__ constexpr float zz_sign(int i) { return ((i ^ (i >> 1)) & 1) ? -1.f : 1.f; }

// Resident CTAs per SM.  Adjoint: 3 (168 registers, no spills; 2, 4 and 5:
// 16.4, 17.4 and 18.8 against 15.8 ms on four cubic graphs n = 24, p = 3, 25
// points); energy: 4 (128 registers; 2, 3 and 5: 10.0, 9.2 and 9.4 against 9.0
// ms on the 6x6 torus).
constexpr int kCoreGradBlocks = 3, kCoreEnergyBlocks = 4;

inline size_t core_smem_bytes(int p, bool grad) { return size_t(4) * (p * kCoreRow + (grad ? 2 * p * kTileSum * sizeof(float) : 0)); }

// A warp takes L.tpw consecutive tiles of one item: the item's decoding, its
// phase tables (staged in shared memory, rows of real parts and of imaginary
// parts) and the warp reductions and atomics of the sums are per item and not
// per tile.  Meanwhile the tiles' energies and terms gather in FP64, their derivatives
// per lane in shared memory (Tfl).
//
// Bound: the adjoint by the operand reads of its packed FMAs (ncu, p = 3: FP32 pipe
// 63% of the cycles, where packed FMAs of three fresh register pairs reach about 70%,
// 55% of the issue slots; 5,000 instructions of straight-line code, so that the
// block's warps start each tile together, which lets them share fetched code: 14.4 ->
// 13.7 ms; further barriers within the tile or larger blocks were slower), the energy
// by shuffles and shared memory (61%).  Measured
// against the unpacked kernel with one tile per task: four cubic graphs n = 24,
// p = 3, 25 points, gradient 21.6 -> 15.8 ms; 6x6 torus, p = 3, 32 points, energy
// 10.1 -> 8.8 ms (both with their outer passes).
template <bool GRAD, int RB>
__global__ void __launch_bounds__(128, GRAD ? kCoreGradBlocks : kCoreEnergyBlocks) split_core_kernel(const __grid_constant__ BigLaunch L) {
    wait_before();
    constexpr int NR = 1 << RB, NP = NR / 2;
    constexpr int T = RB + 5;
    constexpr int NW = NR / 4;  // packed cut counts, 4 registers per word
    extern __shared__ __align__(256) unsigned char s_core[];
    const int lane = threadIdx.x & 31, warp = warp_index();
    const int64_t gw = int64_t(blockIdx.x) * (blockDim.x >> 5) + warp;
    const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
    const int nin = L.n_in;
    const int p = L.p;
    const int tpw = L.tpw;
    const int64_t per_item = (int64_t(1) << (nin - T)) / tpw;
    const int64_t ntask = L.n_items * per_item;
    const int64_t block_amps = int64_t(1) << nin;
    unsigned char *tab = s_core + warp * (p * kCoreRow);
    float *sums = reinterpret_cast<float *>(s_core + (blockDim.x >> 5) * (p * kCoreRow)) + warp * (2 * p * kTileSum) + lane;
    const uint32_t tab0 = smem_addr(tab);
    // the block's warps start every tile together (a warp past the last task, or of a
    // foreign shape, only keeps step)
    for (int64_t t0 = gw - warp; t0 < ntask; t0 += nw) {
        const int64_t task = min(t0 + warp, ntask - 1);
        const int64_t it = task / per_item;
        const int64_t u0 = (task - it * per_item) * tpw;
        int ci;
        int64_t j, y;
        decode_item(L, L.item0 + it, ci, j, y);
        const DevCone *__restrict__ C = L.cones + L.cone_ids[ci];
        const bool ours = t0 + warp < ntask && !__any_sync(kFull, C->n_in != nin);
        if (t0 + warp < ntask && !ours && lane == 0) atomicOr(L.status, 1);
        const int64_t gj = int64_t(C->graph) * L.P + j;
        const float4 *__restrict__ cs = L.cs + gj * p;
        __syncwarp();
        {
            stage_rows(tab, L.lut + gj * p * L.cmax1, p, L.cmax1, lane);
            if (GRAD)
                for (int c = 0; c < 2 * p; ++c) tile_sum_clear(sums + kTileSum * c);
        }
        __syncwarp();
        // cut word of the item's fixed bits: shell block, lane qubits
        float mult = 1.f;
        uint64_t base = shell_block(C, L.shell, uint32_t(y), mult);
#pragma unroll
        for (int lb = 0; lb < 5; ++lb)
            if ((lane >> lb) & 1) base ^= C->col[RB + lb];
        const FirstMix f1 = first_mix(L, gj, nin);
        const float wgt = float(C->weight);
        const float sig0 = __int_as_float((127 - C->n) << 23) * f1.k2n;
        // In d/d gamma_l, C may be replaced by C - c0: Im<lambda|psi> =
        // <psi_end|O|psi_end> is zero within every core tile, and c0 = m/2
        // (the mean cut value) removes most of the cancellation in the FP32
        // sums.  Counts are bytes of kCoreScale c; 2^23 + kCoreScale c0 here.
        const float b0 = 8388608.f + 0.5f * kCoreScale * float(C->m);
        auto add_sum = [&](int c, Dfl v) { tile_sum_add(sums + kTileSum * c, v); };
        double e_sum = 0.0, t_sum = 0.0;  // of the warp's tile sums
        for (int64_t u = u0; u < u0 + tpw; ++u) {
            __syncthreads();
            if (!ours) continue;
            uint64_t tb = base;
            for (int q = T; q < nin; ++q)
                if ((u >> (q - T)) & 1) tb ^= C->col[q];
            // cut value of every register, one byte each, times kCoreScale (a cone has at most 64 cut bits)
            uint32_t cnt[NW];
            {
                const uint64_t c0 = C->col[0], c1 = C->col[1];
                const uint64_t lo[4] = {0ull, c0, c1, c0 ^ c1};
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    uint64_t h = tb;
#pragma unroll
                    for (int t = 0; t < RB - 2; ++t)
                        if ((w >> t) & 1) h ^= C->col[2 + t];
                    uint32_t packed = 0;
#pragma unroll
                    for (int a = 0; a < 4; ++a) packed |= uint32_t(__popcll(lo[a] ^ h)) << (8 * a);
                    cnt[w] = packed * uint32_t(kCoreScale);
                }
            }
            // table entries of registers h and h + NP in the row of layer l
            auto entry = [&](int h, int l) { return row_entry(tab0 + l * kCoreRow, cnt[h >> 2], cnt[(h >> 2) + NW / 2], h & 3); };
            float2 *__restrict__ sp = L.psi + it * block_amps + (u << T) + lane;
            C2 x[NP];
            if (L.load) {
#pragma unroll
                for (int h = 0; h < NP; ++h) x[h] = load_pair(sp, h << 5, (h + NP) << 5);
            } else {
#pragma unroll
                for (int h = 0; h < NP; ++h) x[h] = entry(h, 0);
            }
            // |psi|^2 = 2^-n kappa_1^(2 n_in) |x|^2 (the first mixer's factored form)
            float sig = sig0;
            // first mixer on the core qubits
            first_mix2<NP, false, GRAD>(x, RB, 5, f1);
            for (int l = 1; l < p; ++l) {
#pragma unroll
                for (int w = 0; w < NW; ++w) opaque(cnt[w]);
#pragma unroll
                for (int h = 0; h < NP; ++h) x[h] = cmul_ri(x[h], entry(h, l));
                const int kl = uniform(C->k[l]);
                if (GRAD) {  // the adjoint keeps exact rotations (its derivative terms need them)
                    const float4 c_s = __ldg(cs + l);
                    on_qubits<NP>(x, kl, kl - RB, [&](const C2 &a, const C2 &b) { return rot2<false>(a, b, c_s); });
                } else {  // the energy: the factored form, two FMAs per output, kappa^(2 k_l) into sigma
                    const FirstMix fl = layer_mix(L, gj, l, kl);
                    first_mix2<NP, false, false>(x, kl, kl - RB, fl);
                    sig *= fl.k2n;
                }
            }
            float acc = 0.f;
            {
                float up[NP];
                const bool norm = !GRAD && L.norm;
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    const float2 v = halves(fma2(x[h].r, x[h].r, mul2(x[h].i, x[h].i)));
                    const float s = norm ? 1.f : zz_sign(h);
                    acc = fmaf(s, v.x, acc);
                    up[h] = s * v.y;  // registers h and h + NP have the same sign
                }
#pragma unroll
                for (int h = 0; h < NP; ++h) acc += up[h];
            }
            {
                const float tv = acc * sig * mult;  // this tile's share of <Z_0 Z_1>
                e_sum += f2d(warp_sum(-0.5f * wgt * tv));
                if (L.terms) t_sum += f2d(warp_sum(tv));
            }
            if (GRAD) {
                C2 r[NP];
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    const P2 s = splat(-0.5f * zz_sign(h));
                    r[h] = C2{mul2(s, x[h].r), mul2(s, x[h].i)};
                }
                for (int l = p - 1; l >= 1; --l) {
                    const float4 c_s = __ldg(cs + l);
                    const int kl = uniform(C->k[l]);
                    auto un = [&](const C2 &a, const C2 &b) { return rot2<true>(a, b, c_s); };
                    Dfl d{0.f, 0.f};
#pragma unroll
                    for (int q = 0; q < RB; ++q) {
                        if (q < kl) {
                            dfl_add(d, xterm_reg<NP>(x, r, q));
                            on_reg<NP>(x, q, un);
                            on_reg<NP>(r, q, un);
                        }
                    }
#pragma unroll 1
                    for (int lb = 0; lb < kl - RB; ++lb) {
                        C2 xo[NP];
#pragma unroll
                        for (int h = 0; h < NP; ++h) xo[h] = shfl_xor(x[h], 1 << lb);
                        dfl_add(d, xterm_lane<NP>(xo, r));
#pragma unroll
                        for (int h = 0; h < NP; ++h) {
                            x[h] = un(x[h], xo[h]);
                            r[h] = un(r[h], shfl_xor(r[h], 1 << lb));
                        }
                    }
                    add_sum(p + l, d);
#pragma unroll
                    for (int w = 0; w < NW; ++w) opaque(cnt[w]);
                    float dg = 0.f, uw[NP], uv[NP];
#pragma unroll
                    for (int h = 0; h < NP; ++h) {
                        const float2 w = halves(row_weight(cnt[h >> 2], cnt[(h >> 2) + NW / 2], h & 3, b0)), v = halves(imconj(r[h], x[h]));
                        dg = fmaf(w.x, v.x, dg);
                        uw[h] = w.y;
                        uv[h] = v.y;
                        const C2 ph = entry(h, l);
                        x[h] = cmulc(x[h], ph);
                        r[h] = cmulc(r[h], ph);
                    }
#pragma unroll
                    for (int h = 0; h < NP; ++h) dg = fmaf(uw[h], uv[h], dg);
                    add_sum(l, Dfl{dg * (1.f / kCoreScale), 0.f});
                }
                // first mixer: the core qubits' terms, then lambda alone un-mixed
                // At p = 1 the first layer is the last: lambda = O psi with
                // O = -1/2 Z_0 Z_1, and <psi|O X_q|psi> is real for every q other
                // than 0 and 1 (X_q and O commute), so only those two contribute.
                {
                    Dfl d{0.f, 0.f};
#pragma unroll
                    for (int q = 0; q < RB; ++q)
                        if (q < 2 || p > 1) dfl_add(d, xterm_reg<NP>(x, r, q));
                    if (p > 1) {
#pragma unroll 1
                        for (int lb = 0; lb < 5; ++lb) {
                            C2 xo[NP];
#pragma unroll
                            for (int h = 0; h < NP; ++h) xo[h] = shfl_xor(x[h], 1 << lb);
                            dfl_add(d, xterm_lane<NP>(xo, r));
                        }
                    }
                    add_sum(p, d);
                }
                first_mix2<NP, true, true>(r, RB, 5, f1);
#pragma unroll
                for (int h = 0; h < NP; ++h) store_pair(sp, h << 5, (h + NP) << 5, r[h]);
            }
        }
        if (!ours) continue;
        if (lane == 0) {
            atomicAdd(L.energy + gj, e_sum);
            if (L.terms) atomicAdd(L.terms + C->rep * L.P + j, t_sum);
        }
        if (GRAD) {
            const float wgt2 = 2.f * wgt * mult * sig0;
            for (int l = 1; l < p; ++l) {
                add_gp(tile_sum(sums + kTileSum * (p + l)), wgt2, L.grad, gj * 2 * p + p + l);
                add_gp(tile_sum(sums + kTileSum * l), wgt2, L.grad, gj * 2 * p + l);
            }
            add_gp(tile_sum(sums + kTileSum * p), wgt2, L.grad, gj * 2 * p + p);
        }
    }
}

// ---------------------------------------------------------------- outer passes
constexpr int kOuterRow = 68;  // table entries: a cone has at most 64 cut bits
template <bool V>
struct BoolTag {
    static constexpr bool value = V;
};

// Qubit held by storage address bit a (see the layout above).
__device__ __forceinline__ int qubit_of(int a, int rb) { return a < 5 ? rb + a : (a < rb + 5 ? a - 5 : a); }

// A warp takes L.tpw consecutive tiles of an item (lanes = address bits 0..4,
// registers = the window).  The item's first-layer table sits in shared memory,
// a lane holds the cut word of one address bit outside the window (a tile's
// fixed word is one XOR reduction), and the derivative sums gather over the
// tiles (Tfl).  The state is held an amplitude per packed pair; kOuterFirst, which
// forms pair terms, holds registers h and h + 16 together as the core pass does.
// Blocks per SM: 4 and 3 (generation at 3 and 5, the others at 2 and 4: no faster).
// Generation was bound by the integer pipe (64-bit popcounts and table lookups in
// global memory, 50%).  With the chunk passes changed alike, against scalar
// registers and one tile per task: four cubic graphs n = 24, p = 3, 25 points,
// gradient 15.8 -> 14.4 ms, energy 3.7 -> 3.3 ms; 6x6 torus, p = 3, 32 points,
// energy 8.8 -> 8.3 ms; Q_12 full cone, 32 points, energy 4.5 -> 4.15 ms.
template <int MODE, bool LO, typename MT>
__global__ void __launch_bounds__(128, MODE == kOuterGen ? 4 : 3) split_outer_kernel(const __grid_constant__ BigLaunch L) {
    wait_before();
    __shared__ __align__(16) float s_tab[4][MODE == kOuterMix ? 4 : 2 * kOuterRow];
    const int lane = threadIdx.x & 31, warp = warp_index();
    const int64_t gw = int64_t(blockIdx.x) * (blockDim.x >> 5) + warp;
    const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
    const int nin = L.n_in, b = L.b, RB = L.rb;
    const int r0 = L.w0 - b, r1 = L.w1 - b;  // register bits of the outer qubits to mix
    const int p = L.p;
    const int tpw = L.tpw;
    const int64_t per_item = (int64_t(1) << (nin - 10)) / tpw;
    const int64_t ntask = L.n_items * per_item;
    const int64_t block_amps = int64_t(1) << nin;
    const int64_t lowmask = (int64_t(1) << (b - 5)) - 1;
    for (int64_t task = gw; task < ntask; task += nw) {
        const int64_t it = task / per_item;
        const int64_t tile0 = (task - it * per_item) * tpw;
        int ci;
        int64_t j, y;
        decode_item(L, L.item0 + it, ci, j, y);
        const DevCone *__restrict__ C = L.cones + L.cone_ids[ci];
        if (__any_sync(kFull, C->n_in != nin)) {
            if (lane == 0) atomicOr(L.status, 1);
            continue;
        }
        const int64_t gj = int64_t(C->graph) * L.P + j;
        const FirstMix f1 = first_mix(L, gj, nin);
        float mult = 1.f;
        MT item_w = 0, bit_w = 0, col[5];
        int pairs[kPairs5];
        if (MODE != kOuterMix) {
            // first layer's phase table: entries (kOuterGen), or real parts, then imaginary parts
            __syncwarp();
            const float2 *__restrict__ lut = L.lut + gj * p * L.cmax1;
            for (int e = lane; e < L.cmax1; e += 32) {
                const float2 v = __ldg(lut + e);
                if (MODE == kOuterGen) {
                    reinterpret_cast<float2 *>(s_tab[warp])[e] = v;
                } else {
                    s_tab[warp][e] = v.x;
                    s_tab[warp][kOuterRow + e] = v.y;
                }
            }
            __syncwarp();
            item_w = MT(shell_block(C, L.shell, uint32_t(y), mult));
#pragma unroll
            for (int lb = 0; lb < 5; ++lb)
                if ((lane >> lb) & 1) item_w ^= MT(C->col[RB + lb]);
            if (lane >= 5 && lane < nin && (lane < b || lane >= b + 5)) bit_w = MT(C->col[qubit_of(lane, RB)]);
#pragma unroll
            for (int q = 0; q < 5; ++q) col[q] = MT(C->col[qubit_of(b + q, RB)]);
#pragma unroll
            for (int q = 1; q < 5; ++q)
#pragma unroll
                for (int t = 0; t < q; ++t) pairs[q * (q - 1) / 2 + t] = uniform(window_pair(col[q], col[t], MT(C->neg)));
        }
        Tfl s_dg{0.f, 0.f, 0.f}, s_db{0.f, 0.f, 0.f};  // of the lane's tiles
        for (int64_t tile = tile0; tile < tile0 + tpw; ++tile) {
            // address of (lane, register i) = xb | (i << b) | lane
            const int64_t xb = ((tile & lowmask) << 5) | ((tile >> (b - 5)) << (b + 5));
            float2 *__restrict__ sp = L.psi + it * block_amps + xb + lane;
            MT base = 0;
            if (MODE != kOuterMix) base = item_w ^ warp_xor(((xb >> lane) & 1) ? bit_w : MT(0));
            if constexpr (MODE == kOuterFirst) {
                C2 x[16];  // lambda
#pragma unroll
                for (int h = 0; h < 16; ++h) x[h] = load_pair(sp, int64_t(h) << b, int64_t(h + 16) << b);
                auto unmix = [&](auto form) {
#pragma unroll
                    for (int q = 0; q < 5; ++q)
                        if (q >= r0 && q < r1)
                            on_reg<16>(x, q, [&](const C2 &u, const C2 &v) {
                                return fmix2<decltype(form)::value, true, LO>(u, v, f1.a, f1.alo);
                            });
                };
                if (f1.b)
                    unmix(BoolTag<true>{});
                else
                    unmix(BoolTag<false>{});
                // the outer qubits' mixer terms vanish at p = 1, where the first
                // layer is the last (only qubits 0 and 1 contribute there)
                const bool outer_terms = p > 1;
                const float b0 = 4194304.f + 0.5f * float(C->m);  // Im<lambda|psi> = 0: C - c0 in place of C
                const float *tr = s_tab[warp], *ti = s_tab[warp] + kOuterRow;
                // state before the first mixer, times 2^(n/2), of registers h and h + 16
                int cnt[32];
                window_counts<5, 1>(base, col, pairs, cnt);
                C2 ph[16];
                float dg = 0.f, uw[16], uv[16];
#pragma unroll
                for (int h = 0; h < 16; ++h) {
                    const int cl = cnt[h], cu = cnt[h + 16];
                    ph[h] = C2{p2(tr[cl], tr[cu]), p2(ti[cl], ti[cu])};
                    const float2 v = halves(imconj(x[h], ph[h]));
                    dg = fmaf(cut_minus(cl, b0), v.x, dg);
                    uw[h] = cut_minus(cu, b0);
                    uv[h] = v.y;
                }
#pragma unroll
                for (int h = 0; h < 16; ++h) dg = fmaf(uw[h], uv[h], dg);
                tfl_add(s_dg, Dfl{dg, 0.f});
                if (outer_terms) {
                    Dfl db{0.f, 0.f};
#pragma unroll
                    for (int rb = 0; rb < 5; ++rb) {  // per window qubit
                        float d = 0.f;
                        if (rb >= r0 && rb < r1) {
#pragma unroll
                            for (int h = 0; h < 16; ++h) {
                                const float2 v = halves(imconj(rb == 4 ? swap(x[h]) : x[h ^ ((1 << rb) & 15)], ph[h]));
                                d += v.x;
                                uv[h] = v.y;
                            }
#pragma unroll
                            for (int h = 0; h < 16; ++h) d += uv[h];
                        }
                        dfl_add(db, d);
                    }
                    for (int q = L.x0; q < L.x1; ++q) {  // outer qubits outside the window
                        // (qubit q's edges into the window shift its counts: the sums start over)
                        window_counts<5, 1>(MT(base ^ MT(C->col[q])), col, pairs, cnt);
                        float t = 0.f;
#pragma unroll
                        for (int h = 0; h < 16; ++h) {
                            const int cl = cnt[h], cu = cnt[h + 16];
                            const float2 v = halves(imconj(x[h], C2{p2(tr[cl], tr[cu]), p2(ti[cl], ti[cu])}));
                            t += v.x;
                            uv[h] = v.y;
                        }
#pragma unroll
                        for (int h = 0; h < 16; ++h) t += uv[h];
                        dfl_add(db, t);
                    }
                    tfl_add(s_db, db);
                }
            } else {
                P2 x[32];
                if (MODE == kOuterGen) {
                    const float2 *tab = reinterpret_cast<const float2 *>(s_tab[warp]);
                    int cnt[32];
                    window_counts<5, 1>(base, col, pairs, cnt);
#pragma unroll
                    for (int i = 0; i < 32; ++i) x[i] = load_amp(tab + cnt[i]);
                    first_mix_regs<32, false, LO>(x, r0, r1, f1);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) x[i] = load_amp(sp + (int64_t(i) << b));
                    if (L.sign > 0)
                        first_mix_regs<32, false, LO>(x, r0, r1, f1);
                    else
                        first_mix_regs<32, true, LO>(x, r0, r1, f1);
                }
#pragma unroll
                for (int i = 0; i < 32; ++i) store_amp(sp + (int64_t(i) << b), x[i]);
            }
        }
        if (MODE == kOuterFirst) {
            // lambda = 2^(-n/2) kappa_1^(2 n_in) x once the first mixer is undone
            const float wgt2 = 2.f * float(C->weight) * mult * __int_as_float((127 - C->n) << 23) * f1.k2n;
            add_gp(tfl_pair(s_dg), wgt2, L.grad, gj * 2 * p);
            if (p > 1) add_gp(tfl_pair(s_db), wgt2, L.grad, gj * 2 * p + p);
        }
    }
}

// ------------------------------------------------------------ chunk passes
// An outer pass over more than five outer qubits stages a chunk of the block
// in shared memory: 2^13 amplitudes made of the lowest lo = 13 - w address
// bits (contiguous runs of at least 64 bytes) and a window of w <=
// kChunkMaxW outer qubits.  The window is mixed five qubits at a time by
// register butterflies over amplitudes gathered from shared memory, so one
// HBM round trip covers all of it.  The chunk moves between HBM and shared
// memory by the tensor memory accelerator: one cp.async.bulk.tensor per
// chunk and direction, described by a tensor map of the block (the run, the
// address bits between run and window, the window in two dimensions of at
// most 256, the bits above it times the wave's items), completion of a load
// tracked by an mbarrier.  The copies use the natural order (element e at
// e); the rounds in between use a bank-swizzled order.
constexpr int kChunkBits = 13;
constexpr int kChunkMaxW = 10;
constexpr int kChunkThreads = 256;

// Bank swizzle for runs of eight amplitudes (a window of ten): bit 3 of the
// shared-memory index (which 64-byte half of a 128-byte row) is flipped by
// the parity of the bits above it, so the four 64-byte runs that a warp
// touches fall two in each half.  With runs of 16 or more the rounds' lanes
// read 16 consecutive amplitudes per half-warp, free of conflicts as they
// are, and no swizzle is applied.
__device__ __forceinline__ int swz(int s) { return s ^ ((__popc(s >> 4) & 1) << 3); }
__device__ __forceinline__ int sidx(int s, bool swizzled) { return swizzled ? swz(s) : s; }

// ---- tensor-memory-accelerator helpers (one thread issues, an mbarrier tracks loads)
__device__ __forceinline__ void mbar_init(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Orders this thread's earlier shared-memory accesses before later accesses
// of the asynchronous (TMA) proxy.
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Load of one box into shared memory, completing on bar (issued by one thread).
__device__ __forceinline__ void tma_load(const CUtensorMap *map, void *dst, uint64_t *bar, uint32_t bytes,
                                         const int (&c)[5]) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, "
        "%6}], [%7];" ::"r"(smem_addr(dst)),
        "l"(map), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]), "r"(c[4]), "r"(smem_addr(bar))
        : "memory");
}

// Store of one box from shared memory; returns once the box has been read
// (issued by one thread, after every writer's fence_async_smem and a barrier).
__device__ __forceinline__ void tma_store(const CUtensorMap *map, const void *src, const int (&c)[5]) {
    asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4, %5}], [%6];" ::"l"(
                     map),
                 "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]), "r"(c[4]), "r"(smem_addr(src))
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

__device__ __forceinline__ void tma_store_drain() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Waits for phase `phase` of bar to complete, for at most limit_ns; false if
// it has not.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t phase, uint64_t limit_ns) {
    const uint32_t a = smem_addr(bar);
    const uint64_t t0 = global_ns();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(a), "r"(phase)
            : "memory");
        if (done) return true;
        if (global_ns() - t0 > limit_ns) return false;
    }
}
constexpr uint64_t kTmaWaitNs = 2000000000ull;  // 2 s: a load of 64 KB takes microseconds

// slot with gn zero bits inserted at bit position pos
__device__ __forceinline__ int spread_slot(int slot, int pos, int gn) {
    return (slot & ((1 << pos) - 1)) | ((slot >> pos) << (pos + gn));
}

// What the slots of a chunk share, in shared memory: the first layer's phase
// table and the cut words of the chunk's 13 bits.
template <typename MT>
struct ChunkItem {
    float2 tab[kOuterRow];
    MT col[kChunkBits];
    int pairs[kPairs5];  // of the first round's window bits (see window_counts)
};

// First-layer cut values over the G register bits from chunk bit pos on (the
// window's lowest), with the slot's fixed bits sb and cw.
template <int G, typename MT>
__device__ __forceinline__ void slot_counts(const ChunkItem<MT> &I, MT cw, int sb, int pos, int (&c)[1 << G]) {
    MT base = cw;
#pragma unroll
    for (int b = 0; b < kChunkBits; ++b)
        if ((sb >> b) & 1) base ^= I.col[b];  // the register bits of sb are zero
    MT col[5];
    int pairs[kPairs5];
#pragma unroll
    for (int b = 0; b < 5; ++b) col[b] = b < G ? I.col[pos + b] : MT(0);
#pragma unroll
    for (int k = 0; k < kPairs5; ++k) pairs[k] = I.pairs[k];
    window_counts<G, 1>(base, col, pairs, c);
}

// A chunk element's place: the swizzled one where asked for (SW: the chunk's
// geometry has a swizzle at all).
template <bool SW>
__device__ __forceinline__ int place(int s, bool swizzled) {
    return SW ? sidx(s, swizzled) : s;
}

// One round of a chunk pass: every slot gathers the 2^G amplitudes that
// differ in chunk bits [pos, pos+G), applies the mixer to those G qubits and
// writes them back.  GEN in its first round generates the amplitudes instead.
template <int G, bool GEN, bool INV, bool LO, bool SW, typename MT>
__device__ __forceinline__ void chunk_round(float2 *__restrict__ sm, int n_el, int pos, const FirstMix &f,
                                            const ChunkItem<MT> &I, MT cw, bool rd_swz, bool wr_swz) {
    constexpr int NR = 1 << G;
    for (int slot = threadIdx.x; slot < (n_el >> G); slot += kChunkThreads) {
        const int sb = spread_slot(slot, pos, G);
        P2 x[NR];
        if (GEN) {
            int c[NR];
            slot_counts<G>(I, cw, sb, pos, c);
#pragma unroll
            for (int i = 0; i < NR; ++i) x[i] = load_amp(I.tab + c[i]);
        } else {
#pragma unroll
            for (int i = 0; i < NR; ++i) x[i] = load_amp(sm + place<SW>(sb + (i << pos), rd_swz));
        }
        first_mix_regs<NR, INV, LO>(x, 0, G, f);
#pragma unroll
        for (int i = 0; i < NR; ++i) store_amp(sm + place<SW>(sb + (i << pos), wr_swz), x[i]);
    }
}

template <bool GEN, bool INV, bool LO, bool SW, typename MT>
__device__ __forceinline__ void chunk_round_g(int G, float2 *sm, int n_el, int pos, const FirstMix &f,
                                              const ChunkItem<MT> &I, MT cw, bool rd_swz, bool wr_swz) {
    switch (G) {
        case 1: chunk_round<1, GEN, INV, LO, SW>(sm, n_el, pos, f, I, cw, rd_swz, wr_swz); break;
        case 2: chunk_round<2, GEN, INV, LO, SW>(sm, n_el, pos, f, I, cw, rd_swz, wr_swz); break;
        case 3: chunk_round<3, GEN, INV, LO, SW>(sm, n_el, pos, f, I, cw, rd_swz, wr_swz); break;
        case 4: chunk_round<4, GEN, INV, LO, SW>(sm, n_el, pos, f, I, cw, rd_swz, wr_swz); break;
        default: chunk_round<5, GEN, INV, LO, SW>(sm, n_el, pos, f, I, cw, rd_swz, wr_swz); break;
    }
}

// sw: the chunk's runs are short enough (eight amplitudes, a window of ten, whose
// rounds all have five bits) for the swizzle.  A first round always has five.
template <bool GEN, bool INV, bool LO, typename MT>
__device__ __forceinline__ void chunk_round_any(int G, float2 *sm, int n_el, int pos, const FirstMix &f,
                                                const ChunkItem<MT> &I, MT cw, bool sw, bool rd_swz, bool wr_swz) {
    if (sw)
        chunk_round<5, GEN, INV, LO, true>(sm, n_el, pos, f, I, cw, rd_swz, wr_swz);
    else if (GEN)
        chunk_round<5, GEN, INV, LO, false>(sm, n_el, pos, f, I, cw, false, false);
    else
        chunk_round_g<GEN, INV, LO, false>(G, sm, n_el, pos, f, I, cw, false, false);
}

template <int MODE, bool LO, typename MT>
__global__ void __launch_bounds__(kChunkThreads, 2)
    split_chunk_kernel(const __grid_constant__ BigLaunch L, const __grid_constant__ CUtensorMap tmap) {
    wait_before();
    extern __shared__ __align__(1024) float2 sm[];
    __shared__ uint64_t s_bar;  // completion of the chunk's load
    __shared__ ChunkItem<MT> s_item;
    const int tid = threadIdx.x;
    if (tid == 0) mbar_init(&s_bar);
    __syncthreads();
    uint32_t phase = 0;
    const int nin = L.n_in, RB = L.rb, w0 = L.w0, w = L.w1 - L.w0;
    const int lo_bits = kChunkBits - w;  // lowest address bits of the chunk (w0 >= lo_bits)
    const int n_el = 1 << kChunkBits;
    const int p = L.p;
    const int64_t chunks = int64_t(1) << (nin - kChunkBits);
    const int64_t ntask = L.n_items * chunks;
    const int64_t lowmask = (int64_t(1) << (w0 - lo_bits)) - 1;
    for (int64_t task = blockIdx.x; task < ntask; task += gridDim.x) {
        const int64_t it = task / chunks;
        const int64_t ch = task - it * chunks;
        int ci;
        int64_t j, y;
        decode_item(L, L.item0 + it, ci, j, y);
        const DevCone *__restrict__ C = L.cones + L.cone_ids[ci];
        if (C->n_in != nin) {  // uniform over the CTA
            if (tid == 0) atomicOr(L.status, 1);
            continue;
        }
        const int64_t gj = int64_t(C->graph) * L.P + j;
        const FirstMix f1 = first_mix(L, gj, nin);
        // element e of the chunk <-> address xb + (e & runmask) + ((e >> lo_bits) << w0) of
        // item it; tensor coordinates: run, middle bits, window (two dimensions), high bits x item
        const int64_t xb = ((ch & lowmask) << lo_bits) | ((ch >> (w0 - lo_bits)) << (w0 + w));
        const int crd[5] = {0, int(ch & lowmask), 0, 0,
                            int(it * (int64_t(1) << (nin - w0 - w)) + (ch >> (w0 - lo_bits)))};
        if (MODE != kOuterGen && tid == 0) {
            fence_async_smem();  // the previous task's accesses come before the copy's writes
            tma_load(&tmap, sm, &s_bar, uint32_t(n_el * sizeof(float2)), crd);
        }
        // the item's table and the chunk bits' cut words, and the cut word of its
        // fixed bits (shell block and address bits outside the chunk)
        float mult = 1.f;
        MT cw = 0;
        if (MODE != kOuterMix) {
            const float2 *__restrict__ lut = L.lut + gj * p * L.cmax1;  // first layer's phase table
            for (int e = tid; e < L.cmax1; e += kChunkThreads) s_item.tab[e] = __ldg(lut + e);
            if (tid < kChunkBits)
                s_item.col[tid] = MT(C->col[tid < lo_bits ? qubit_of(tid, RB) : w0 + tid - lo_bits]);
            if (tid < kPairs5) {  // pair (q, t), t < q
                const int q = tid < 1 ? 1 : tid < 3 ? 2 : tid < 6 ? 3 : 4, t = tid - q * (q - 1) / 2;
                s_item.pairs[tid] = window_pair(MT(C->col[w0 + q]), MT(C->col[w0 + t]), MT(C->neg));
            }
            cw = MT(shell_block(C, L.shell, uint32_t(y), mult));
            for (int a = lo_bits; a < nin; ++a)
                if ((a < w0 || a >= w0 + w) && ((xb >> a) & 1)) cw ^= MT(C->col[qubit_of(a, RB)]);
        }
        if (MODE != kOuterGen) {
            // bounded wait; should it ever run out (never expected), record it,
            // give the copy the same time again to land, and stop this block
            const bool ok = mbar_wait(&s_bar, phase, kTmaWaitNs);
            if (__syncthreads_or(!ok)) {
                if (tid == 0) atomicOr(L.status, 4);
                mbar_wait(&s_bar, phase, kTmaWaitNs);
                return;
            }
            phase ^= 1u;
        }
        __syncthreads();
        for (int g0 = 0; g0 < w; g0 += 5) {
            const int gn = min(5, w - g0);  // this round's qubits: chunk bits lo_bits + g0 ..
            // the copies use the natural order, the rounds between them the swizzled one
            const bool swz_on = lo_bits < 4;
            const bool rd_swz = swz_on && g0 > 0, wr_swz = swz_on && (g0 + gn < w || MODE == kOuterFirst);
            if (MODE == kOuterGen && g0 == 0)
                chunk_round_any<true, false, LO>(gn, sm, n_el, lo_bits, f1, s_item, cw, swz_on, rd_swz, wr_swz);
            else if (MODE == kOuterGen || (MODE == kOuterMix && L.sign > 0))
                chunk_round_any<false, false, LO>(gn, sm, n_el, lo_bits + g0, f1, s_item, cw, swz_on, rd_swz, wr_swz);
            else
                chunk_round_any<false, true, LO>(gn, sm, n_el, lo_bits + g0, f1, s_item, cw, swz_on, rd_swz, wr_swz);
            __syncthreads();
        }
        if (MODE == kOuterFirst) {
            // lambda is now fully un-mixed: the first layer's phase term and the
            // outer qubits' mixer terms against exp(-i gamma_1 C)|+>
            const bool outer_terms = p > 1;
            const float b0 = 4194304.f + 0.5f * float(C->m);  // Im<lambda|psi> = 0: C - c0 in place of C
            const int gn = min(5, w);
            const int nreg = 1 << gn;
            Dfl dg{0.f, 0.f}, db{0.f, 0.f};  // this thread's slots, compensated
            for (int slot = tid; slot < (n_el >> gn); slot += kChunkThreads) {
                const int sb = spread_slot(slot, lo_bits, gn);
                float2 x[32];
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    x[i] = i < nreg ? sm[sidx(sb | (i << lo_bits), lo_bits < 4)] : make_float2(0.f, 0.f);
                int cnt[32];
                slot_counts<5>(s_item, cw, sb, lo_bits, cnt);  // w > 5 here: five window qubits in registers
                float dgs = 0.f, dq[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int c = cnt[i];
                    const float2 ph = s_item.tab[c];
                    dgs = fmaf(cut_minus(c, b0), imconj(x[i], ph), dgs);
                    if (outer_terms) {
#pragma unroll
                        for (int rb = 0; rb < 5; ++rb) dq[rb] += imconj(x[i ^ (1 << rb)], ph);
                    }
                }
                dfl_add(dg, dgs);
                if (outer_terms) {
#pragma unroll
                    for (int rb = 0; rb < 5; ++rb) dfl_add(db, dq[rb]);
                    // the other outer qubits: the rest of the window, then beyond it
                    for (int q = w0 + 5; q < L.x1; ++q) {
                        slot_counts<5>(s_item, MT(cw ^ MT(C->col[q])), sb, lo_bits, cnt);
                        float t = 0.f;
#pragma unroll
                        for (int i = 0; i < 32; ++i) t += imconj(x[i], s_item.tab[cnt[i]]);
                        dfl_add(db, t);
                    }
                }
            }
            // lambda = 2^(-n/2) kappa_1^(2 n_in) x once the first mixer is undone
            const float wgt2 = 2.f * float(C->weight) * mult * __int_as_float((127 - C->n) << 23) * f1.k2n;
            add_gp(dg, wgt2, L.grad, gj * 2 * p);
            if (outer_terms) add_gp(db, wgt2, L.grad, gj * 2 * p + p);
        } else {
            fence_async_smem();  // every thread's writes, before the copy reads them
            __syncthreads();
            if (tid == 0) tma_store(&tmap, sm, crd);
        }
        __syncthreads();  // the next task reuses the shared chunk
    }
    if (tid == 0) tma_store_drain();
}

// Tensor map of a wave's blocks as the chunk passes of window [w0, w0 + w) see
// them (8-byte elements): the run of the lo = 13 - w lowest address bits,
// the bits between run and window, the window in two dimensions of at most 2^8,
// the bits above it times the items.  Dense: every stride is the previous one
// times the previous extent.
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encoder() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    });
    return fn;
}

cudaError_t chunk_map(const BigLaunch &B, int w0, int w, CUtensorMap *map) {
    EncodeTiledFn enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    const int nin = B.n_in, lo = kChunkBits - w, wa = w < 8 ? w : 8;
    const cuuint64_t dim[5] = {cuuint64_t(1) << lo, cuuint64_t(1) << (w0 - lo), cuuint64_t(1) << wa,
                               cuuint64_t(1) << (w - wa), cuuint64_t(B.n_items) << (nin - w0 - w)};
    const cuuint64_t stride[4] = {cuuint64_t(8) << lo, cuuint64_t(8) << w0, cuuint64_t(8) << (w0 + wa),
                                  cuuint64_t(8) << (w0 + w)};
    const cuuint32_t box[5] = {1u << lo, 1u, 1u << wa, 1u << (w - wa), 1u};
    const cuuint32_t estride[5] = {1u, 1u, 1u, 1u, 1u};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 5, B.psi, dim, stride, box, estride,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

int occupancy_grid(const void *fn, int block, size_t smem);

bool split_ok(int n_in, int p, const int32_t *k, bool grad) {
    const int T = (grad ? kSplitRbGrad : kSplitRbEnergy) + 5;
    if (n_in < 10 || n_in < T || n_in > QAOA_MAX_CONE_QUBITS || k[0] != n_in) return false;
    if (grad && n_in == T) return false;
    for (int l = 1; l < p; ++l)
        if (k[l] > T) return false;
    return true;
}

namespace {

// The variants of a pass: lo, the first mixer's coefficient as a hi + lo pair (the
// adjoint's passes); wide, 64-bit cut words.  kOuterFirst is the adjoint's alone.
template <int MODE, bool LO>
const void *outer_fn(bool wide) {
    return wide ? (const void *)split_outer_kernel<MODE, LO, uint64_t> : (const void *)split_outer_kernel<MODE, LO, uint32_t>;
}
const void *outer_fn(int mode, bool lo, bool wide) {
    if (mode == kOuterGen) return lo ? outer_fn<kOuterGen, true>(wide) : outer_fn<kOuterGen, false>(wide);
    if (mode == kOuterMix) return lo ? outer_fn<kOuterMix, true>(false) : outer_fn<kOuterMix, false>(false);
    return outer_fn<kOuterFirst, true>(wide);
}
template <int MODE, bool LO>
const void *chunk_fn(bool wide) {
    return wide ? (const void *)split_chunk_kernel<MODE, LO, uint64_t> : (const void *)split_chunk_kernel<MODE, LO, uint32_t>;
}
const void *chunk_fn(int mode, bool lo, bool wide) {
    if (mode == kOuterGen) return lo ? chunk_fn<kOuterGen, true>(wide) : chunk_fn<kOuterGen, false>(wide);
    if (mode == kOuterMix) return lo ? chunk_fn<kOuterMix, true>(false) : chunk_fn<kOuterMix, false>(false);
    return chunk_fn<kOuterFirst, true>(wide);
}

constexpr size_t kChunkSmem = sizeof(float2) << kChunkBits;

}  // namespace

// Chunk kernels need more than the default 48 KB of dynamic shared memory:
// raised once per device, at upload.
cudaError_t split_prepare() {
    static std::mutex mu;
    static std::set<int> done;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (done.count(dev)) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    for (int mode : {kOuterGen, kOuterMix, kOuterFirst})
        for (int v = 0; v < 4 && e == cudaSuccess; ++v)
            e = cudaFuncSetAttribute(chunk_fn(mode, v & 1, v & 2), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     int(kChunkSmem));
    if (e == cudaSuccess) done.insert(dev);
    return e;
}

cudaError_t launch_split_wave(BigLaunch B, bool grad, int chunk_window, int64_t &launches, cudaStream_t s) {
    const int cw_max = chunk_window < 6 ? 6 : (chunk_window > kChunkMaxW ? kChunkMaxW : chunk_window);
    const int RB = grad ? kSplitRbGrad : kSplitRbEnergy, T = RB + 5;
    const int nin = B.n_in, p = B.p;
    B.rb = RB;
    // Outer qubit windows: shared-memory chunks of up to kChunkMaxW qubits
    // while more than five remain, then one register window of at most five.
    struct Win {
        int w0, w1;
        bool chunk;
    };
    std::vector<Win> win;
    for (int w0 = T; w0 < nin;) {
        const int left = nin - w0;
        const int n = left > 5 ? std::min(left, cw_max) : left;
        win.push_back({w0, w0 + n, left > 5});
        w0 += n;
    }
    auto outer = [&](int mode, size_t w, int sign) -> cudaError_t {
        B.mode = mode;
        B.w0 = win[w].w0;
        B.w1 = win[w].w1;
        B.b = std::min(B.w0, nin - 5);
        B.x0 = win[w].w1;
        B.x1 = nin;
        B.sign = sign;
        const bool wide = B.cmax1 - 1 > 32;
        if (win[w].chunk) {
            CUtensorMap map;
            if (cudaError_t e = chunk_map(B, B.w0, B.w1 - B.w0, &map); e != cudaSuccess) return e;
            const int64_t tasks = B.n_items << (nin - kChunkBits);
            const void *fn = chunk_fn(mode, grad, wide);
            const int grid = int(std::min<int64_t>(occupancy_grid(fn, kChunkThreads, kChunkSmem), std::max<int64_t>(tasks, 1)));
            void *args[] = {&B, &map};
            if (cudaError_t e = launch_after(fn, grid, kChunkThreads, args, kChunkSmem, s); e != cudaSuccess) return e;
        } else {
            const void *fn = outer_fn(mode, grad, wide);
            const int full = occupancy_grid(fn, 128, 0);
            B.tpw = tiles_per_task(B.n_items, nin - 10, full);
            const int64_t tasks = (B.n_items << (nin - 10)) / B.tpw;
            const int grid = int(std::min<int64_t>(full, std::max<int64_t>(1, (tasks + 3) / 4)));
            void *args[] = {&B};
            if (cudaError_t e = launch_after(fn, grid, 128, args, 0, s); e != cudaSuccess) return e;
        }
        ++launches;
        return cudaSuccess;
    };
    if (grad && win.empty()) return cudaErrorInvalidValue;  // excluded by split_ok
    cudaError_t e = cudaSuccess;
    for (size_t w = 0; w < win.size() && e == cudaSuccess; ++w) e = outer(w == 0 ? kOuterGen : kOuterMix, w, 1);
    if (e != cudaSuccess) return e;
    B.load = win.empty() ? 0 : 1;
    const void *core = grad ? (const void *)split_core_kernel<true, kSplitRbGrad>
                            : (const void *)split_core_kernel<false, kSplitRbEnergy>;
    const size_t core_smem = core_smem_bytes(p, grad);
    const int core_grid = occupancy_grid(core, 128, core_smem);
    B.tpw = tiles_per_task(B.n_items, nin - T, core_grid);
    const int64_t core_tasks = (B.n_items << (nin - T)) / B.tpw;
    const int grid = int(std::min<int64_t>(core_grid, std::max<int64_t>(1, (core_tasks + 3) / 4)));
    void *args[] = {&B};
    if ((e = launch_after(core, grid, 128, args, core_smem, s)) != cudaSuccess) return e;
    ++launches;
    if (!grad) return cudaSuccess;
    for (size_t w = win.size(); w-- > 1 && e == cudaSuccess;) e = outer(kOuterMix, w, -1);
    if (e != cudaSuccess) return e;
    return outer(kOuterFirst, 0, -1);
}

}  // namespace qaoa
