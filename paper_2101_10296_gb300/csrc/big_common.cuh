// Device helpers shared by the large-state kernels.
#pragma once

#include "big.cuh"
#include "dev_math.cuh"
#include "packed.cuh"

namespace qaoa {
namespace {

// One output of exp(-i beta X) on the pair (me, o), c me - i s o, or of
// exp(+i beta X) (INV), with c = cs.x + cs.z and s = cs.y + cs.w (hi and lo FP32
// parts), on the amplitudes of two packed registers.
template <bool INV>
__device__ __forceinline__ C2 rot2(const C2 &me, const C2 &o, float4 cs) {
    const float s = INV ? -cs.y : cs.y, w = INV ? -cs.w : cs.w;
    return C2{fma2(splat(cs.x), me.r, fma2(splat(s), o.i, fma2(splat(cs.z), me.r, mul2(splat(w), o.i)))),
              fma2(splat(cs.x), me.i, fma2(splat(-s), o.r, fma2(splat(cs.z), me.i, mul2(splat(-w), o.r))))};
}

// The same (forward) on one amplitude, its real and imaginary parts a packed pair.
__device__ __forceinline__ P2 rot1(P2 me, P2 o, float4 cs) {
    const P2 so = swap(o);
    return fma2(splat(cs.x), me, fma2(p2(cs.y, -cs.y), so, fma2(splat(cs.z), me, mul2(p2(cs.w, -cs.w), so))));
}

// op(me, partner) on register qubit q of a tile
template <int NP, class F>
__device__ __forceinline__ void on_reg(C2 (&x)[NP], int q, F &&op) {
    if ((1 << q) == NP) {
#pragma unroll
        for (int h = 0; h < NP; ++h) x[h] = op(x[h], swap(x[h]));
    } else {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            if (h & (1 << q)) continue;
            const int j = h | (1 << q);
            const C2 u = x[h], v = x[j];
            x[h] = op(u, v);
            x[j] = op(v, u);
        }
    }
}

// Im<r|X_q|x> over register qubit q: the pairs' terms in register order.
template <int NP>
__device__ __forceinline__ float xterm_reg(const C2 (&x)[NP], const C2 (&r)[NP], int q) {
    float d = 0.f;
    if ((1 << q) == NP) {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            const float2 t = halves(imconj(r[h], swap(x[h])));
            d += t.x + t.y;
        }
    } else {
        float up[NP / 2];
        int n = 0;
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            if (h & (1 << q)) continue;
            const int j = h | (1 << q);
            const float2 t = halves(add2(imconj(r[h], x[j]), imconj(r[j], x[h])));
            d += t.x;
            up[n++] = t.y;
        }
#pragma unroll
        for (int k = 0; k < NP / 2; ++k) d += up[k];
    }
    return d;
}

// The same over a lane qubit, given the partner's x.
template <int NP>
__device__ __forceinline__ float xterm_lane(const C2 (&xo)[NP], const C2 (&r)[NP]) {
    float d = 0.f, up[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        const float2 t = halves(imconj(r[h], xo[h]));
        d += t.x;
        up[h] = t.y;
    }
#pragma unroll
    for (int h = 0; h < NP; ++h) d += up[h];
    return d;
}

// An amplitude as a packed pair.
__device__ __forceinline__ P2 load_amp(const float2 *p) { return P2{*reinterpret_cast<const unsigned long long *>(p)}; }
__device__ __forceinline__ void store_amp(float2 *p, P2 v) { *reinterpret_cast<unsigned long long *>(p) = v.v; }

// Cut words as 32 bits where every cone of the plan fits them, else 64.
__device__ __forceinline__ int popc_w(uint32_t x) { return __popc(x); }
__device__ __forceinline__ int popc_w(uint64_t x) { return __popcll(x); }
// Scaled cut values over G window bits.  With the fixed bits' word base, setting
// bit q adds d_q = popc(base ^ col_q) - popc(base), and setting q and q' together
// adds pair_qq' more, -2 for each positive (+2 for each negative) cut bit of an
// edge that joins them, whatever base is: so a lane counts G + 1 words and adds up
// the others (two integer additions per value instead of a 64-bit exclusive or, two
// popcounts and an addition).  The pairs are uniform: pairs[q (q - 1) / 2 + q'].
// With rounds that leave the swizzle's address work out where there is none: 6x6
// torus, p = 3, 32 points, energy 8.27 -> 7.49 ms, gradient, 8 points 8.84 -> 8.58
// (64-bit words); no change with 32-bit words (cubic n = 24).
constexpr int kPairs5 = 10;
template <typename MT>
__device__ __forceinline__ int window_pair(MT a, MT b, MT neg) {
    return 2 * (popc_w(MT(a & b & neg)) - popc_w(MT(a & b & ~neg)));
}
template <int G, int SCALE, typename MT>
__device__ __forceinline__ void window_counts(MT base, const MT (&col)[5], const int (&pairs)[kPairs5], int (&c)[1 << G]) {
    const int n = popc_w(base);
    c[0] = SCALE * n;
#pragma unroll
    for (int q = 0; q < G; ++q) {
        int e[1 << (G - 1)];
        e[0] = SCALE * (popc_w(MT(base ^ col[q])) - n);
#pragma unroll
        for (int i = 0; i < (1 << q); ++i) {
            const int t = i < 2 ? 0 : i < 4 ? 1 : i < 8 ? 2 : 3;  // the highest bit of i > 0
            if (i > 0) e[i] = e[i ^ (1 << t)] + SCALE * pairs[q * (q - 1) / 2 + t];
            c[i | (1 << q)] = c[i] + e[i];
        }
    }
}
// XOR over the lanes.
__device__ __forceinline__ uint32_t warp_xor(uint32_t x) { return __reduce_xor_sync(kFull, x); }
__device__ __forceinline__ uint64_t warp_xor(uint64_t x) {
    return (uint64_t(__reduce_xor_sync(kFull, uint32_t(x >> 32))) << 32) | __reduce_xor_sync(kFull, uint32_t(x));
}
// c - c0 of a cut value, given b0 = 2^22 + c0 (halves are exact at that size)
__device__ __forceinline__ float cut_minus(int c, float b0) { return __uint_as_float(0x4A800000u + 2u * uint32_t(c)) - b0; }

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return uint32_t(__cvta_generic_to_shared(p)); }

// Rows of a warp's phase tables: 68 real parts, then 68 imaginary parts (a cone
// has at most 64 cut bits); count bytes hold 2 c.
constexpr int kCoreRow = 544, kCoreIm = 272;
constexpr float kCoreScale = 2.f;
// Stages p layers' phase tables in rows (above); called by the whole warp.
__device__ __forceinline__ void stage_rows(unsigned char *tab, const float2 *__restrict__ lut, int p, int cmax1, int lane) {
    for (int l = 0; l < p; ++l)
        for (int e = lane; e < cmax1; e += 32) {
            const float2 v = __ldg(lut + l * cmax1 + e);
            *reinterpret_cast<float *>(tab + l * kCoreRow + 4 * e) = v.x;
            *reinterpret_cast<float *>(tab + l * kCoreRow + kCoreIm + 4 * e) = v.y;
        }
}
// Entries of count byte a of two packed words in a row.
__device__ __forceinline__ C2 row_entry(uint32_t row, uint32_t wa, uint32_t wb, int a) {
    const uint32_t p = row + (__byte_perm(wa, 0u, 0x4440u | uint32_t(a)) << 1);
    const uint32_t q = row + (__byte_perm(wb, 0u, 0x4440u | uint32_t(a)) << 1);
    return C2{p2(lds1(p), lds1(q)), p2(lds1(p + kCoreIm), lds1(q + kCoreIm))};
}
// kCoreScale (c - c0) of the same bytes, given b0 = 2^23 + kCoreScale c0.
__device__ __forceinline__ P2 row_weight(uint32_t wa, uint32_t wb, int a, float b0) {
    return add2(p2(__uint_as_float(__byte_perm(wa, 0x4B000000u, 0x7540u | uint32_t(a))),
                   __uint_as_float(__byte_perm(wb, 0x4B000000u, 0x7540u | uint32_t(a)))),
                splat(-b0));
}
// Amplitudes at offsets i and j of p in one packed register.
__device__ __forceinline__ C2 load_pair(const float2 *p, int64_t i, int64_t j) {
    const float2 u = p[i], v = p[j];
    return C2{p2(u.x, v.x), p2(u.y, v.y)};
}
__device__ __forceinline__ void store_pair(float2 *p, int64_t i, int64_t j, const C2 &x) {
    const float2 a = halves(x.r), b = halves(x.i);
    p[i] = make_float2(a.x, b.x);
    p[j] = make_float2(a.y, b.y);
}

// Warp sum in FP32 (every lane gets it).
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Compensated warp sum of a derivative partial times w, then one FP64
// atomic into base[idx].
__device__ __forceinline__ void add_gp(Dfl v, float w, double *base, int64_t idx) {
    v = dfl_warp_sum(dfl_scale(v, w));
    if ((threadIdx.x & 31) == 0) atomicAdd(base + idx, dfl_value(v));
}

// Derivative sums of a warp's tiles in shared memory: per output and lane a Tfl, its
// parts 32 floats apart (s points at the lane's first).
constexpr int kTileSum = 96;
__device__ __forceinline__ void tile_sum_clear(float *s) { s[0] = s[32] = s[64] = 0.f; }
__device__ __forceinline__ void tile_sum_add(float *s, Dfl v) {
    Tfl a{s[0], s[32], s[64]};
    tfl_add(a, v);
    s[0] = a.hi;
    s[32] = a.lo;
    s[64] = a.lo2;
}
__device__ __forceinline__ Dfl tile_sum(const float *s) { return tfl_pair(Tfl{s[0], s[32], s[64]}); }

// Item -> (cone of the shape, point j, shell block y).  Cone c owns the items
// P * [ystart[c], ystart[c+1]), ordered point-major.
__device__ __forceinline__ void decode_item(const BigLaunch &L, int64_t item, int &ci, int64_t &j, int64_t &y) {
    int lo = 0, hi = L.n_shape - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (L.P * L.ystart[mid] <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    const int64_t Y = L.ystart[lo + 1] - L.ystart[lo];
    const int64_t rem = item - L.P * L.ystart[lo];
    j = rem / Y;
    y = rem - j * Y;
    ci = lo;
}

}  // namespace
}  // namespace qaoa
