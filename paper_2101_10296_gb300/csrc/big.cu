// Large-state cone path: cones whose inner part (the qubits any mixer
// touches, within distance p-1 of the edge) is too large for registers.
//
// Every (cone, point, shell assignment) owns a block of 2^n_in complex64
// amplitudes in scratch memory.  A pass streams a block once through
// registers: a warp tile covers 10 qubits -- qubits 0..4 on the lanes, so
// that each load or store instruction of the warp touches 256 contiguous
// bytes, and qubits b..b+4 in registers -- and applies a short list of
// operations (phase, mixer on the tile's qubits, reduction, and in the
// adjoint their inverses with the derivative terms).  Gates are the exact
// unitaries exp(-i gamma C) and exp(-i beta X) (Sec. 2.2); the adjoint uses
// exp(+i beta X) and exp(+i gamma C), which keep <lambda|X_q|psi> invariant
// under the un-mixing of any qubit of the same layer.
#include "big.cuh"
#include "big_common.cuh"

namespace qaoa {
namespace {

constexpr int NP = 1 << (kBigRegBits - 1);  // packed registers: h holds registers h and h + 16
constexpr int NW = 8;                       // packed cut counts, 4 registers per word

// A warp takes L.tpw consecutive tiles of an item: its phase tables sit in
// shared memory, a lane holds the cut word of one address bit outside the window
// (a tile's fixed word is one XOR reduction), cut values are counted once per
// tile (bytes of kCoreScale c), and the derivative sums gather per lane in
// shared memory (Tfl) until the item's tiles are done.  Sums over the registers run
// in register order: lower halves, then upper ones.
//
// Bound: FP32 and latency at two blocks per SM (three, with 168 registers, spill:
// 1.96 against 1.24 ms).  Against scalar registers, a popcount per amplitude and
// operation and one tile per task, C_30(1,2) at p = 4, 64 points: gradient 1.78 ->
// 1.24 ms, energy 0.50 -> 0.30 ms.
template <bool GRAD, typename MT>
__global__ void __launch_bounds__(128) big_pass_kernel(const __grid_constant__ BigLaunch L) {
    wait_before();
    extern __shared__ __align__(256) unsigned char s_big[];
    const int lane = threadIdx.x & 31, warp = warp_index();
    const int64_t gw = int64_t(blockIdx.x) * (blockDim.x >> 5) + warp;
    const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
    const BigPass &ps = L.pass;
    const int b = ps.b;
    const int nin = L.n_in;
    const int p = L.p;
    const int tpw = L.tpw;
    const int64_t per_item = (int64_t(1) << (nin - 10)) / tpw;
    const int64_t ntask = L.n_items * per_item;
    const int64_t block_amps = int64_t(1) << nin;
    const int64_t lowmask = (int64_t(1) << (b - 5)) - 1;
    unsigned char *tab = s_big + warp * (p * kCoreRow);
    float *sums = reinterpret_cast<float *>(s_big + 4 * (p * kCoreRow)) + warp * (2 * p * kTileSum) + lane;
    const uint32_t tab0 = smem_addr(tab);
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
        const float4 *__restrict__ cs = L.cs + gj * p;
        __syncwarp();
        stage_rows(tab, L.lut + gj * p * L.cmax1, p, L.cmax1, lane);
        if (GRAD)
            for (int c = 0; c < 2 * p; ++c) tile_sum_clear(sums + kTileSum * c);
        __syncwarp();
        // cut words: shell block ^ lane part, the address bits outside the window (one per lane), the window's
        float mult = 1.f;
        MT item_w = MT(shell_block(C, L.shell, uint32_t(y), mult));
#pragma unroll
        for (int q = 0; q < 5; ++q)
            if ((lane >> q) & 1) item_w ^= MT(C->col[q]);
        MT bit_w = 0, wc[5];
        if (lane >= 5 && lane < nin && (lane < b || lane >= b + 5)) bit_w = MT(C->col[lane]);
#pragma unroll
        for (int q = 0; q < 5; ++q) wc[q] = MT(C->col[b + q]);
        const float wgt = float(C->weight) * mult;             // orbit size x shell multiplicity
        const float sig = __int_as_float((127 - C->n) << 23);  // 2^-n
        // Im<r|x> = 0: C - m/2 in place of C in the derivatives
        const float b0 = 8388608.f + 0.5f * kCoreScale * float(C->m);
        auto add_sum = [&](int c, Dfl v) { tile_sum_add(sums + kTileSum * c, v); };
        double e_sum = 0.0, t_sum = 0.0;  // of the warp's tile sums
        for (int64_t tile = tile0; tile < tile0 + tpw; ++tile) {
            // inner index of (lane, register i): xb | (i << b) | lane
            const int64_t xb = ((tile & lowmask) << 5) | ((tile >> (b - 5)) << (b + 5));
            uint32_t cnt[NW];
            {
                const MT base = item_w ^ warp_xor(((xb >> lane) & 1) ? bit_w : MT(0));
                const MT lo[4] = {MT(0), wc[0], wc[1], MT(wc[0] ^ wc[1])};
#pragma unroll
                for (int k = 0; k < NW; ++k) {
                    const MT h = base ^ ((k & 1) ? wc[2] : MT(0)) ^ ((k & 2) ? wc[3] : MT(0)) ^ ((k & 4) ? wc[4] : MT(0));
                    uint32_t packed = 0;
#pragma unroll
                    for (int a = 0; a < 4; ++a) packed |= uint32_t(popc_w(MT(lo[a] ^ h))) << (8 * a);
                    cnt[k] = packed * uint32_t(kCoreScale);
                }
            }
            auto entry = [&](int h, int l) { return row_entry(tab0 + l * kCoreRow, cnt[h >> 2], cnt[(h >> 2) + NW / 2], h & 3); };
            float2 *__restrict__ sp = L.psi + it * block_amps + xb + lane;
            float2 *__restrict__ lp = GRAD ? L.lam + it * block_amps + xb + lane : nullptr;
            C2 x[NP], r[GRAD ? NP : 1];
            if (ps.load_psi) {
#pragma unroll
                for (int h = 0; h < NP; ++h) x[h] = load_pair(sp, int64_t(h) << b, int64_t(h + NP) << b);
            }
            if constexpr (GRAD) {
                if (ps.load_lam) {
#pragma unroll
                    for (int h = 0; h < NP; ++h) r[h] = load_pair(lp, int64_t(h) << b, int64_t(h + NP) << b);
                }
            }
            for (int o = 0; o < ps.nops; ++o) {
                const BigOp op = ps.ops[o];
                const int l = op.layer;
#pragma unroll
                for (int k = 0; k < NW; ++k) opaque(cnt[k]);
                switch (op.type) {
                    case kOpGenPhase: {  // |+> (amplitude 1) times exp(-i gamma_1 C)
#pragma unroll
                        for (int h = 0; h < NP; ++h) x[h] = entry(h, 0);
                        break;
                    }
                    case kOpPhase: {
#pragma unroll
                        for (int h = 0; h < NP; ++h) x[h] = cmul_ri(x[h], entry(h, l));
                        break;
                    }
                    case kOpMix: {
                        const float4 c_s = __ldg(cs + l);
                        auto f = [&](const C2 &u, const C2 &v) { return rot2<false>(u, v, c_s); };
#pragma unroll 1
                        for (int q = op.q0; q < op.q1 && q < 5; ++q) {
#pragma unroll
                            for (int h = 0; h < NP; ++h) x[h] = f(x[h], shfl_xor(x[h], 1 << q));
                        }
#pragma unroll
                        for (int rb = 0; rb < kBigRegBits; ++rb)
                            if (b + rb >= op.q0 && b + rb < op.q1) on_reg<NP>(x, rb, f);
                        break;
                    }
                    case kOpReduce: {
                        const float sg = ((lane ^ (lane >> 1)) & 1) && !L.norm ? -1.f : 1.f;
                        float acc = 0.f;
#pragma unroll
                        for (int h = 0; h < NP; ++h) acc = fmaf(lo(x[h].r), lo(x[h].r), fmaf(lo(x[h].i), lo(x[h].i), acc));
#pragma unroll
                        for (int h = 0; h < NP; ++h) acc = fmaf(hi(x[h].r), hi(x[h].r), fmaf(hi(x[h].i), hi(x[h].i), acc));
                        const float tv = sg * acc * sig * mult;  // this block's share of <Z_0 Z_1>
                        e_sum += f2d(warp_sum(-0.5f * float(C->weight) * tv));
                        if (L.terms) t_sum += f2d(warp_sum(tv));
                        break;
                    }
                    case kOpLamInit: {
                        if constexpr (GRAD) {
                            const P2 sg = splat(((lane ^ (lane >> 1)) & 1) ? 0.5f : -0.5f);
#pragma unroll
                            for (int h = 0; h < NP; ++h) r[h] = C2{mul2(sg, x[h].r), mul2(sg, x[h].i)};
                        }
                        break;
                    }
                    case kOpUnmix: {
                        if constexpr (GRAD) {
                            const float4 c_s = __ldg(cs + l);
                            auto f = [&](const C2 &u, const C2 &v) { return rot2<true>(u, v, c_s); };
                            // At the last layer lambda = O psi (O = -1/2 Z_0 Z_1), and
                            // <psi|O X_q|psi> is real for every q other than 0 and 1 (X_q
                            // commutes with O and with the mixers of other qubits): only
                            // those two enter d/d beta_p, the others are rounding noise.
                            const int qd = l == p - 1 ? 2 : QAOA_MAX_CONE_QUBITS;
                            Dfl acc{0.f, 0.f};
#pragma unroll 1
                            for (int q = op.q0; q < op.q1 && q < 5; ++q) {
                                C2 xo[NP];
#pragma unroll
                                for (int h = 0; h < NP; ++h) xo[h] = shfl_xor(x[h], 1 << q);
                                if (q < qd) dfl_add(acc, xterm_lane<NP>(xo, r));  // this qubit's terms, then added compensated
#pragma unroll
                                for (int h = 0; h < NP; ++h) {
                                    x[h] = f(x[h], xo[h]);
                                    r[h] = f(r[h], shfl_xor(r[h], 1 << q));
                                }
                            }
#pragma unroll
                            for (int rb = 0; rb < kBigRegBits; ++rb) {
                                if (b + rb >= op.q0 && b + rb < op.q1) {
                                    if (b + rb < qd) dfl_add(acc, xterm_reg<NP>(x, r, rb));
                                    on_reg<NP>(x, rb, f);
                                    on_reg<NP>(r, rb, f);
                                }
                            }
                            add_sum(p + l, acc);
                        }
                        break;
                    }
                    case kOpUnphase: {  // q0 = 1: also undo the phase
                        if constexpr (GRAD) {
                            // eight terms at a time into the compensated sum: the halves' groups side by side
                            P2 d[2] = {splat(0.f), splat(0.f)};
#pragma unroll
                            for (int h = 0; h < NP; ++h) {
                                const P2 w = row_weight(cnt[h >> 2], cnt[(h >> 2) + NW / 2], h & 3, b0);
                                d[h / 8] = fma2(w, imconj(r[h], x[h]), d[h / 8]);
                                if (op.q0) {
                                    const C2 ph = entry(h, l);
                                    x[h] = cmulc(x[h], ph);
                                    r[h] = cmulc(r[h], ph);
                                }
                            }
                            Dfl acc{0.f, 0.f};
                            dfl_add(acc, lo(d[0]));
                            dfl_add(acc, lo(d[1]));
                            dfl_add(acc, hi(d[0]));
                            dfl_add(acc, hi(d[1]));
                            add_sum(l, Dfl{acc.hi * (1.f / kCoreScale), acc.lo * (1.f / kCoreScale)});
                        }
                        break;
                    }
                    default:
                        break;
                }
            }
            if (ps.store_psi) {
#pragma unroll
                for (int h = 0; h < NP; ++h) store_pair(sp, int64_t(h) << b, int64_t(h + NP) << b, x[h]);
            }
            if constexpr (GRAD) {
                if (ps.store_lam) {
#pragma unroll
                    for (int h = 0; h < NP; ++h) store_pair(lp, int64_t(h) << b, int64_t(h + NP) << b, r[h]);
                }
            }
        }
        bool reduces = false;
        for (int o = 0; o < ps.nops; ++o) {
            const BigOp op = ps.ops[o];
            reduces = reduces || op.type == kOpReduce;
            if (GRAD && (op.type == kOpUnmix || op.type == kOpUnphase)) {
                // an op's sums, once: a layer's mixer may come in several ops of a pass
                const int c = op.type == kOpUnmix ? p + op.layer : op.layer;
                add_gp(tile_sum(sums + kTileSum * c), 2.f * wgt * sig, L.grad, gj * 2 * p + c);
                tile_sum_clear(sums + kTileSum * c);
            }
        }
        if (reduces && lane == 0) {
            atomicAdd(L.energy + gj, e_sum);
            if (L.terms) atomicAdd(L.terms + C->rep * L.P + j, t_sum);
        }
    }
}

// A pass made only of mixers: load, butterflies on the tile's qubits, store.
// No cut words or tables, so far fewer registers and more loads in flight.  An
// amplitude per packed register.
__global__ void __launch_bounds__(128, 4) big_mix_kernel(const __grid_constant__ BigLaunch L) {
    wait_before();
    constexpr int NR = 2 * NP;
    const int lane = threadIdx.x & 31;
    const int64_t gw = int64_t(blockIdx.x) * (blockDim.x >> 5) + warp_index();
    const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
    const BigPass &ps = L.pass;
    const int b = ps.b;
    const int64_t tiles = int64_t(1) << (L.n_in - 10);
    const int64_t ntask = L.n_items * tiles;
    const int64_t block_amps = int64_t(1) << L.n_in;
    for (int64_t task = gw; task < ntask; task += nw) {
        const int64_t it = task / tiles;
        const int64_t tile = task - it * tiles;
        int ci;
        int64_t j, y;
        decode_item(L, L.item0 + it, ci, j, y);
        const DevCone *__restrict__ C = L.cones + L.cone_ids[ci];
        const float4 *__restrict__ cs = L.cs + (int64_t(C->graph) * L.P + j) * L.p;
        const int64_t lowmask = (int64_t(1) << (b - 5)) - 1;
        const int64_t xb = ((tile & lowmask) << 5) | ((tile >> (b - 5)) << (b + 5));
        float2 *__restrict__ sp = L.psi + it * block_amps + xb + lane;
        P2 x[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) x[i] = load_amp(sp + (int64_t(i) << b));
        for (int o = 0; o < ps.nops; ++o) {
            const BigOp op = ps.ops[o];
            const float4 c_s = __ldg(cs + op.layer);
#pragma unroll 1
            for (int q = op.q0; q < op.q1 && q < 5; ++q) {
#pragma unroll
                for (int i = 0; i < NR; ++i) x[i] = rot1(x[i], shfl_xor(x[i], 1 << q), c_s);
            }
#pragma unroll
            for (int rb = 0; rb < kBigRegBits; ++rb) {
                if (b + rb < op.q0 || b + rb >= op.q1) continue;
#pragma unroll
                for (int i = 0; i < NR; ++i) {
                    if (i & (1 << rb)) continue;
                    const int i2 = i | (1 << rb);
                    const P2 u = x[i], v = x[i2];
                    x[i] = rot1(u, v, c_s);
                    x[i2] = rot1(v, u, c_s);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < NR; ++i) store_amp(sp + (int64_t(i) << b), x[i]);
    }
}

}  // namespace

int occupancy_grid(const void *fn, int block, size_t smem);

namespace {

int mix_grid() { return occupancy_grid((const void *)big_mix_kernel, 128, 0); }

const void *pass_fn(bool grad, bool wide) {
    if (grad) return wide ? (const void *)big_pass_kernel<true, uint64_t> : (const void *)big_pass_kernel<true, uint32_t>;
    return wide ? (const void *)big_pass_kernel<false, uint64_t> : (const void *)big_pass_kernel<false, uint32_t>;
}

}  // namespace

static bool mix_only(const BigPass &ps) {
    if (!ps.load_psi || !ps.store_psi || ps.load_lam || ps.store_lam) return false;
    for (int o = 0; o < ps.nops; ++o)
        if (ps.ops[o].type != kOpMix) return false;
    return true;
}

cudaError_t launch_big_pass(BigLaunch a, bool grad, cudaStream_t s) {
    const int bits = a.n_in - 10;
    const int64_t tiles = a.n_items << bits;
    if (mix_only(a.pass)) {
        const int64_t need = std::max<int64_t>(1, (tiles + 3) / 4);
        void *args[] = {&a};
        return launch_after((const void *)big_mix_kernel, int(std::min<int64_t>(mix_grid(), need)), 128, args, 0, s);
    }
    const size_t smem = size_t(4) * (a.p * kCoreRow + (grad ? 2 * a.p * kTileSum * sizeof(float) : 0));
    const void *fn = pass_fn(grad, a.cmax1 - 1 > 32);
    const int full = occupancy_grid(fn, 128, smem);
    a.tpw = tiles_per_task(a.n_items, bits, full);
    const int64_t need = std::max<int64_t>(1, (tiles / a.tpw + 3) / 4);
    void *args[] = {&a};
    return launch_after(fn, int(std::min<int64_t>(full, need)), 128, args, smem, s);
}

// ------------------------------------------------------------ pass lists

namespace {

// Register window [b, b+5) of the tile that holds qubits [lo, hi)
int window_for(int lo, int n_in) { return lo < 10 ? 5 : std::min(lo, n_in - 5); }

bool fits(const BigPass &ps, int q0, int q1) {
    for (int q = q0; q < q1; ++q)
        if (!(q < 5 || (q >= ps.b && q < ps.b + 5))) return false;
    return true;
}

}  // namespace

// Forward op list for one cone shape, split into passes.  Layer l applies
// its phase, then its mixer on the qubit groups [10,15), [15,20), ... (each
// in its own register window) and finally on [0, 10) in window 5, so that
// the low group fuses with the next layer's phase and, when that layer only
// mixes low qubits, with its mixer too.
std::vector<BigPass> big_forward_passes(int n_in, int p, const int32_t *k) {
    std::vector<BigPass> out;
    auto push_op = [&](uint8_t type, int layer, int q0, int q1, int want_b) {
        if (out.empty() || (type == kOpMix && !fits(out.back(), q0, q1)) || out.back().nops >= kBigMaxOps) {
            BigPass ps{};
            ps.b = want_b;
            out.push_back(ps);
        }
        BigPass &ps = out.back();
        ps.ops[ps.nops++] = BigOp{type, uint8_t(layer), uint8_t(q0), uint8_t(q1)};
    };
    for (int l = 0; l < p; ++l) {
        const int kl = k[l];
        std::vector<std::pair<int, int>> groups;
        for (int lo = 10; lo < kl; lo += 5) groups.emplace_back(lo, std::min(lo + 5, kl));
        groups.emplace_back(0, std::min(kl, 10));
        const int first_b = window_for(groups.front().first, n_in);
        push_op(l == 0 ? kOpGenPhase : kOpPhase, l, 0, 0, first_b);
        for (auto &gq : groups) push_op(kOpMix, l, gq.first, gq.second, window_for(gq.first, n_in));
    }
    push_op(kOpReduce, 0, 0, 0, 5);
    for (size_t i = 0; i < out.size(); ++i) {
        out[i].load_psi = i > 0;
        out[i].store_psi = i + 1 < out.size();
    }
    return out;
}

// Adjoint: the forward passes, except that the last one continues with the
// co-state initialisation and the inverse of its own ops; then the earlier
// passes in reverse order with inverted ops.  An inverted phase of layer 0
// only contributes its derivative.
std::vector<BigPass> big_grad_passes(int n_in, int p, const int32_t *k) {
    std::vector<BigPass> fwd = big_forward_passes(n_in, p, k);
    std::vector<BigPass> out;
    auto invert = [](const BigPass &src, BigPass &dst) {
        for (int o = src.nops - 1; o >= 0; --o) {
            const BigOp &op = src.ops[o];
            BigOp inv = op;
            if (op.type == kOpReduce) continue;
            if (op.type == kOpMix) inv.type = kOpUnmix;
            if (op.type == kOpPhase) inv = BigOp{kOpUnphase, op.layer, 1, 0};
            if (op.type == kOpGenPhase) inv = BigOp{kOpUnphase, op.layer, 0, 0};
            dst.ops[dst.nops++] = inv;
        }
    };
    for (size_t i = 0; i < fwd.size(); ++i) {
        BigPass ps = fwd[i];
        if (i + 1 < fwd.size()) {
            out.push_back(ps);  // forward part, stores psi
            continue;
        }
        // last forward pass: forward ops, reduce, co-state, inverse ops
        ps.ops[ps.nops++] = BigOp{kOpLamInit, 0, 0, 0};
        invert(fwd[i], ps);
        ps.store_psi = fwd.size() > 1;
        ps.store_lam = fwd.size() > 1;
        out.push_back(ps);
    }
    for (int i = int(fwd.size()) - 2; i >= 0; --i) {
        BigPass ps{};
        ps.b = fwd[i].b;
        invert(fwd[i], ps);
        ps.load_psi = true;
        ps.load_lam = true;
        ps.store_psi = i > 0;
        ps.store_lam = i > 0;
        out.push_back(ps);
    }
    return out;
}

}  // namespace qaoa
