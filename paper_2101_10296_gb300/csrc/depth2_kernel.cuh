// Register-resident kernel of pruned cones at p = 2: the depth-2 form of
// cone_kernel.cuh (same states, same sums in the same order, so the same
// numbers), laid out for packed FP32x2 instructions.
//
// As there, a thread holds 2^R amplitudes of inner blocks, lanes hold the inner
// qubits from R on, higher bits index threads and blocks; psi = K X^F s with
// |K|^2 = sigma from a table, F the bit flips of layers with |tan beta| > 1.
//
// Layout.  Register h of the thread is the packed pair (amplitude h, amplitude
// h + 2^(R-1)), real and imaginary parts in registers of their own.  Every
// operation of the sweep -- butterflies, phases, pair terms, the observable --
// treats the two halves alike, so it is one packed instruction for both; the
// butterfly on the paired qubit itself reads its partner with the halves
// exchanged, which the instruction does for free.  Only the pair terms of that
// qubit and the sums over a thread's groups of four are scalar.  The FP32 pipe
// spends two cycles on a packed instruction (its peak does not rise), but half
// the issue slots: they go to the lookups, shuffles and conversions, which kept
// the unpacked kernel at 37% of the FP32 pipe.
//
// Lookups.  Without flips a thread's cut values never change, and the last
// layer is preceded by one flip set, so both sets of counts are taken at upload,
// one byte each, scaled so that the byte is the entry's offset in its table row:
// a byte permute forms the address (the row starts at a multiple of 256), and
// two 4-byte loads (real and imaginary rows, free of bank conflicts) fill the
// halves of the packed registers.
//
// The last layer mixes qubits 0 and 1 alone (gate pruning, Sec. 2.3), so its
// phase, mixer, observable, derivative terms and their inverses stay within
// groups of four amplitudes: they run group by group in one pass with one
// lookup per amplitude, psi and the co-state r = Z_u Z_v psi leaving it undone
// to the state before that layer.
//
// Numerics as in cone_kernel.cuh.  Bound: the FP32 pipe, 71 lane operations per
// amplitude and point with the adjoint at six inner qubits (22 for the energy).
// Measured on four random cubic graphs of 2,000 vertices at 64 points (638 M
// amplitude-points), against the unpacked kernel: adjoint 3.59 -> 2.32 ms (55%
// of the FP32 pipe's cycles, 70 instructions per amplitude instead of 131; two
// warps per scheduler leave the rest to fixed latencies), energy 0.93 -> 0.73 ms
// (51%, shared memory and shuffles at 55%).
#pragma once

#include "packed.cuh"
#include "reg_common.cuh"

namespace qaoa {
namespace {

// (I - i tau X) on register qubit q
template <int R>
__device__ __forceinline__ void mix_q(C2 (&x)[1 << (R - 1)], int q, float tau) {
    constexpr int NP = 1 << (R - 1);
    if (q == R - 1) {  // the paired qubit: the partner is the other half
#pragma unroll
        for (int h = 0; h < NP; ++h) x[h] = bfly(x[h], swap(x[h]), tau);
    } else {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            if (h & (1 << q)) continue;
            const int j = h | (1 << q);
            const C2 a = x[h], b = x[j];
            x[h] = bfly(a, b, tau);
            x[j] = bfly(b, a, tau);
        }
    }
}

// Counts as bytes.  NARROW (at most 31 cut bits): 4 c, the entry's offset in a
// 256-byte row (32 real, 32 imaginary parts); otherwise 2 c (c <= 64), rows of
// kWideRow bytes.
template <bool NARROW>
struct Counts {
    static constexpr float kScale = NARROW ? 4.f : 2.f;
    static constexpr uint32_t kIm = NARROW ? 128u : kDepth2WideRow / 2;
    static __device__ __forceinline__ uint32_t addr(uint32_t pk, int a, uint32_t row) {
        if constexpr (NARROW)
            return __byte_perm(pk, row, 0x7650u | uint32_t(a));
        else
            return row + (__byte_perm(pk, 0u, 0x4440u | uint32_t(a)) << 1);
    }
    // table entries of byte a of two packed words
    static __device__ __forceinline__ C2 entry(uint32_t lo, uint32_t hi, int a, uint32_t row) {
        const uint32_t p = addr(lo, a, row), q = addr(hi, a, row);
        return C2{p2(lds1(p), lds1(q)), p2(lds1(p + kIm), lds1(q + kIm))};
    }
    // kScale (c - c0), given b0 = 2^23 + kScale c0: the byte permute makes the FP32
    // value 2^23 + kScale c, and the difference is exact
    static __device__ __forceinline__ P2 weight(uint32_t lo, uint32_t hi, int a, float b0) {
        const P2 v = p2(__uint_as_float(__byte_perm(lo, 0x4B000000u, 0x7540u | uint32_t(a))),
                        __uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7540u | uint32_t(a))));
        return add2(v, splat(-b0));
    }
};

template <int R, bool GRAD, bool NARROW>
__global__ void __launch_bounds__(kRegBlock, depth2_blocks(GRAD, R)) depth2_kernel(const RegLaunch L) {
    wait_before();
    using CT = Counts<NARROW>;
    constexpr int NP = 1 << (R - 1), NG = 1 << (R - 2), HG = NG / 2, kWarps = kRegBlock / 32;
    constexpr int NOUT = reg_outputs(2, GRAD), G = reg_group(2, GRAD);
    extern __shared__ __align__(256) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, warp = warp_index();
    const RegWork &W = L.work;
    const int cm1 = L.cmax1;
    constexpr int row_b = depth2_row_bytes(NARROW);
    // per warp: phase tables [point][layer], point parameters, reduction buffer (reg_flush)
    unsigned char *my_tab = s_raw + size_t(warp) * L.jpt * 2 * row_b;
    float *pars = reinterpret_cast<float *>(s_raw + size_t(kWarps) * L.jpt * 2 * row_b);
    float *my_par = pars + warp * (L.jpt * kDepth2Params);
    float *red = pars + kWarps * (L.jpt * kDepth2Params) + warp * (NOUT * G * 32);
    const uint32_t tab0 = static_cast<uint32_t>(__cvta_generic_to_shared(my_tab));
    const int64_t gw = int64_t(blockIdx.x) * kWarps + warp;
    const int64_t nw = int64_t(gridDim.x) * kWarps;
    const int64_t nblk = (L.n_points + L.jpt - 1) / L.jpt;
    const int64_t ntask = W.warps * nblk;
    // Few tasks per warp: neighbouring tasks take different points, so that the
    // warps running at one time do not all add to the same outputs (random cubic
    // n = 600, 25 points, gradient: 106 -> 88 us); many: different slots, the
    // points' tables stay in L1 (four cubic graphs n = 2000, 64 points: 2344 ->
    // 2304 us).
    const bool spread = ntask < 8 * nw;
    for (int64_t task = gw; task < ntask; task += nw) {
        const int64_t slow = spread ? nblk : W.warps;
        const int64_t t_hi = task / slow, t_lo = task - t_hi * slow;
        const int64_t jb = spread ? t_lo : t_hi, w = spread ? t_hi : t_lo;
        const int64_t j0 = jb * L.jpt;
        const int jn = int(L.n_points - j0 < L.jpt ? L.n_points - j0 : L.jpt);
        const int64_t slot = w * 32 + lane;  // < W.slots, a multiple of 32
        const int g = __ldg(W.warp_graph + w);
        const int64_t row0 = int64_t(g) * L.n_points + j0;
        __syncwarp();  // the previous task's reads of the staged data are done
        {
            const float *__restrict__ src = reinterpret_cast<const float *>(L.lut + row0 * 2 * cm1);
            for (int r = 0; r < jn * 2; ++r)
                for (int e = lane; e < cm1; e += 32) {
                    cp_async4(my_tab + size_t(r) * row_b + 4 * e, src + 2 * (r * cm1 + e));
                    cp_async4(my_tab + size_t(r) * row_b + CT::kIm + 4 * e, src + 2 * (r * cm1 + e) + 1);
                }
            // parameters of a point: tau_1, flip_1, tau_2, kappa_2^4, kappa_1^(2k) (k < kRegKpow)
            for (int e = lane; e < jn * kDepth2Params; e += 32) {
                const int pt = e / kDepth2Params, i = e - pt * kDepth2Params;
                const int64_t gp = (row0 + pt) * 2;
                const float *s = i < 3    ? reinterpret_cast<const float *>(L.mix + gp) + i
                                 : i == 3 ? L.kpow + (gp + 1) * kKpow + 2
                                          : L.kpow + gp * kKpow + (i - 4);
                cp_async4(my_par + e, s);
            }
        }
        const int32_t sc = __ldg(W.slot_cone + slot);
        const int ci = sc & 0x7fffffff;
        const DevCone *__restrict__ C = W.cones + ci;
        uint32_t cnt[NG], cnf[NG];  // counts, and counts after the first layer's flips
        float wk[NG];
#pragma unroll
        for (int k = 0; k < NG; ++k) {
            cnt[k] = __ldg(W.rec_cnt + k * W.slots + slot);
            cnf[k] = __ldg(W.rec_cnt + (NG + k) * W.slots + slot);
            wk[k] = __ldg(W.rec_wk + k * W.slots + slot);
        }
        const int n = C->n;
        bool active = sc >= 0;
        if (n < 2 || n > QAOA_MAX_CONE_QUBITS || C->n_in < 2 || C->n_in > R + kLaneBits || C->k[1] != 2 ||
            C->k[0] > kRegKpow - 1 || C->graph != g) {  // never made by the planner
            if (active) atomicOr(L.status, 1);
            active = false;
        }
        if (!active) {
#pragma unroll
            for (int k = 0; k < NG; ++k) wk[k] = 0.f;
        }
        const float wgt = float(C->weight);
        const float sig0 = __int_as_float((127 - (n & 63)) << 23);  // 2^-n
        const int k1 = min(C->k[0], kRegKpow - 1);
        // 2^23 + kScale m / 2: C enters the derivatives as C - m/2 (see cone_kernel.cuh)
        const float b0 = 8388608.f + 0.5f * CT::kScale * float(C->m);
        cp_async_wait_all();
        __syncwarp();  // the staged data are complete and visible to the warp
        for (int jj = 0; jj < jn; ++jj) {
            const uint32_t row1 = tab0 + uint32_t(jj * 2 * row_b), row2 = row1 + row_b;
            const float *par = my_par + jj * kDepth2Params;
            const float tau1 = par[0], tau2 = par[2];
            const bool flip = par[1] != 0.f;
            auto stash = [&](int c, float v) { red[(c * G + (jj & (G - 1))) * 32 + ((lane + jj) & 31)] = v; };
            C2 x[NP];
            // layer 1: phase on |+>, mixer on the lane's k1 qubits
#pragma unroll
            for (int k = 0; k < NG; ++k) opaque(cnt[k]);
#pragma unroll
            for (int h = 0; h < NP; ++h) x[h] = CT::entry(cnt[h >> 2], cnt[(h >> 2) + HG], h & 3, row1);
#pragma unroll
            for (int q = 0; q < R; ++q)
                mix_q<R>(x, q, q < k1 ? tau1 : 0.f);
#pragma unroll 1
            for (int q = R; __any_sync(kFull, q < k1); ++q) {
                const float t = q < k1 ? tau1 : 0.f;
#pragma unroll
                for (int h = 0; h < NP; ++h) x[h] = bfly(x[h], shfl_xor(x[h], 1 << (q - R)), t);
            }
            float sig = sig0;
            sig *= par[4 + k1];
            // layer 2, four amplitudes (twice: groups k and k + HG) at a time
            C2 r[GRAD ? NP : 1];
            P2 zz[HG], db2[HG], dg2[HG];
#pragma unroll
            for (int k = 0; k < HG; ++k) {
                uint32_t ca = flip ? cnf[k] : cnt[k], cb = flip ? cnf[k + HG] : cnt[k + HG];
                opaque(ca);
                opaque(cb);
                C2 ph[4], y[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    ph[a] = CT::entry(ca, cb, a, row2);
                    y[a] = cmul(x[4 * k + a], ph[a]);
                }
                mix01(y, tau2);
                // |y_0|^2 + |y_3|^2 - |y_1|^2 - |y_2|^2 (norm: plus)
                const P2 pos =
                    fma2(y[0].r, y[0].r, fma2(y[0].i, y[0].i, fma2(y[3].r, y[3].r, mul2(y[3].i, y[3].i))));
                const P2 ngv =
                    fma2(y[1].r, y[1].r, fma2(y[1].i, y[1].i, fma2(y[2].r, y[2].r, mul2(y[2].i, y[2].i))));
                zz[k] = fma2(splat(!GRAD && L.norm ? 1.f : -1.f), ngv, pos);
                if constexpr (GRAD) {
                    // half of Im<r|X_0 + X_1|y> with r = Z_0 Z_1 y (the two terms of a pair coincide)
                    P2 d = splat(0.f);
                    acc_imconj(d, y[0], y[1]);
                    acc_imconj(d, y[0], y[2]);
                    d = fma2(neg(y[2].r), y[3].i, d);
                    d = fma2(y[2].i, y[3].r, d);
                    d = fma2(neg(y[1].r), y[3].i, d);
                    d = fma2(y[1].i, y[3].r, d);
                    db2[k] = d;
                    // the mixer undone: r' = Z_0 Z_1 (I - i tau X_0)(I - i tau X_1) y
                    C2 u[4] = {y[0], y[1], y[2], y[3]};
                    mix01(u, tau2);
                    mix01(y, -tau2);
                    u[1] = neg(u[1]);
                    u[2] = neg(u[2]);
                    P2 dg = splat(0.f);
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        dg = fma2(CT::weight(ca, cb, a, b0), imconj(u[a], y[a]), dg);
                        x[4 * k + a] = cmulc(y[a], ph[a]);
                        r[4 * k + a] = cmulc(u[a], ph[a]);
                    }
                    dg2[k] = dg;
                }
            }
            // sums over the thread's groups, in order
            auto over_groups = [&](const P2(&v)[HG]) {
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < HG; ++k) s = fmaf(wk[k], lo(v[k]), s);
#pragma unroll
                for (int k = 0; k < HG; ++k) s = fmaf(wk[k + HG], hi(v[k]), s);
                return s;
            };
            sig *= par[3];
            const float tl = over_groups(zz);
            stash(0, -0.5f * wgt * sig * tl);
            if (L.terms) {
                float tv = sig * tl;
                if (seg_sum(tv, active ? ci : -1) && active) atomicAdd(L.terms + C->rep * L.n_points + j0 + jj, f2d(tv));
            }
            if constexpr (GRAD) {
                const float gw2 = active ? -wgt : 0.f;  // 2 x (-1/2) x orbit weight
                const float sig_end = sig;
                constexpr float kInv = 1.f / CT::kScale;
                stash(4, gw2 * sig * (2.f * over_groups(db2)));
                sig *= par[3];
                stash(2, gw2 * sig * (kInv * over_groups(dg2)));
                // layer 1: d/d beta_1 = 2 sigma Im <r|sum_q X_q|x>, register qubits on the untouched states
                P2 d[HG];
#pragma unroll
                for (int k = 0; k < HG; ++k) d[k] = splat(0.f);
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    if (q < 2 || q < k1) {
#pragma unroll
                        for (int hh = 0; hh < NP; ++hh) {
                            const int h = 4 * (hh % HG) + hh / HG;  // the groups' chains side by side
                            if (q == R - 1) {
                                // amplitude h with amplitude h + NP: the lower group's sum alone
                                const float2 rr = halves(r[h].r), ri = halves(r[h].i);
                                const float2 xr = halves(x[h].r), xi = halves(x[h].i);
                                float e = lo(d[h >> 2]);
                                e = fmaf(rr.x, xi.y, e);
                                e = fmaf(-ri.x, xr.y, e);
                                e = fmaf(rr.y, xi.x, e);
                                e = fmaf(-ri.y, xr.x, e);
                                d[h >> 2] = p2(e, hi(d[h >> 2]));
                            } else if (!(h & (1 << q))) {
                                const int j = h | (1 << q);
                                acc_imconj(d[h >> 2], r[h], x[j]);
                                acc_imconj(d[h >> 2], r[j], x[h]);
                            }
                        }
                    }
                }
                float db = over_groups(d);
                // lane qubits: each term is taken after the lane qubits before it were undone, which
                // scales it by (1 + tau^2) each; kappa^2 per undone qubit takes that back out.  The
                // last one's is evaluated with the partner's r -- the partner's term, sent back -- so
                // that x, which nothing reads after it, is neither exchanged nor undone.  (The votes
                // make the branches warp-uniform for the compiler, which otherwise adds a warp
                // synchronisation to every shuffle.)
                int q = R;
#pragma unroll 1
                for (; __any_sync(kFull, q + 1 < k1); ++q) {
                    const float t = q < k1 ? -tau1 : 0.f;
                    P2 e[HG];
#pragma unroll
                    for (int k = 0; k < HG; ++k) e[k] = splat(0.f);
#pragma unroll
                    for (int h = 0; h < NP; ++h) {
                        const C2 xo = shfl_xor(x[h], 1 << (q - R)), ro = shfl_xor(r[h], 1 << (q - R));
                        acc_imconj(e[h >> 2], r[h], xo);
                        x[h] = bfly(x[h], xo, t);
                        r[h] = bfly(r[h], ro, t);
                    }
                    if (q < k1) db = fmaf(over_groups(e), par[4 + q - R], db);
                }
                if (__any_sync(kFull, q < k1)) {
                    const int m = 1 << (q - R);
                    const float t = q < k1 ? -tau1 : 0.f;
                    P2 e[HG];
#pragma unroll
                    for (int k = 0; k < HG; ++k) e[k] = splat(0.f);
#pragma unroll
                    for (int h = 0; h < NP; ++h) {
                        const C2 ro = shfl_xor(r[h], m);
                        acc_imconj(e[h >> 2], ro, x[h]);
                        r[h] = bfly(r[h], ro, t);
                    }
                    const float v = __shfl_xor_sync(kFull, over_groups(e), m);
                    if (q < k1) db = fmaf(v, par[4 + q - R], db);
                }
#pragma unroll
                for (int q = 0; q < R; ++q)
                    mix_q<R>(r, q, q < k1 ? -tau1 : 0.f);
                stash(3, gw2 * sig * db);
                // d/d gamma_1: the un-mixed psi would be Lambda exp(-i gamma_1 C) with Lambda the scale of
                // the unnormalised inverse mixers, and sigma Lambda = sigma at the end of the forward sweep
#pragma unroll
                for (int k = 0; k < NG; ++k) opaque(cnt[k]);
#pragma unroll
                for (int k = 0; k < HG; ++k) {
                    P2 dg = splat(0.f);
#pragma unroll
                    for (int a = 0; a < 4; ++a)
                        dg = fma2(CT::weight(cnt[k], cnt[k + HG], a, b0),
                                  imconj(r[4 * k + a], CT::entry(cnt[k], cnt[k + HG], a, row1)), dg);
                    dg2[k] = dg;
                }
                stash(1, gw2 * sig_end * (kInv * over_groups(dg2)));
            }
            if ((jj & (G - 1)) == G - 1 || jj == jn - 1) {
                __syncwarp();
                reg_flush<1>(red, NOUT, G, jj, lane, row0, 4, L.energy, L.grad);
                __syncwarp();
            }
        }
    }
}

}  // namespace
}  // namespace qaoa
