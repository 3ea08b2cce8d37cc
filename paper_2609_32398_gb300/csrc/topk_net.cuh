// Top-K of a token held one row per lane in a swizzled 32-token tile: sorting
// networks on packed fp16 pairs, a bit per candidate, and the drop of the
// excess ones (the selection of select.cuh and router.cu).
#pragma once

#include <cuda_fp16.h>

#include <climits>

#include "dol_internal.cuh"

namespace dol {

constexpr int kSelBoxBytes = 32 * 128;  // 32 rows x 32 fp32

namespace {

// Transpose a 32x32 bit matrix held one row per lane (bit c of lane t is
// element (t, c)); on return lane c holds column c (bit t = element (t, c)).
// Each step exchanges j x j blocks: a rotation of the partner's word by j (up
// or down, by lane) and one bit select.
__device__ __forceinline__ uint32_t transpose32_bits(uint32_t x, int lane) {
    const uint32_t lo_mask[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int j = 16 >> s;
        const uint32_t p = __shfl_xor_sync(kFull, x, j);
        const uint32_t keep = (lane & j) ? ~lo_mask[s] : lo_mask[s];
        const uint32_t r = __funnelshift_l(p, p, (lane & j) ? 32 - j : j);
        x = (x & keep) | (r & ~keep);
    }
    return x;
}

__device__ __forceinline__ uint32_t h2max(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t h2min(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
// two values rounded towards zero to fp16: lo in the low half
__device__ __forceinline__ uint32_t pack_rz(float lo, float hi) {
    uint32_t d;
    asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// v[i] >= v[j] in both halves
__device__ __forceinline__ void ce(uint32_t &a, uint32_t &b) {
    const uint32_t hi = h2max(a, b), lo = h2min(a, b);
    a = hi;
    b = lo;
}

// Batcher's odd-even merge sort of positions LO .. LO + N - 1; cx(i, j) puts
// the larger of two positions first.
template <int LO, int N, int R, class Cx>
__device__ __forceinline__ void net_merge(const Cx &cx) {
    if constexpr (2 * R < N) {
        net_merge<LO, N, 2 * R>(cx);
        net_merge<LO + R, N, 2 * R>(cx);
#pragma unroll
        for (int i = LO + R; i + R < LO + N; i += 2 * R) cx(i, i + R);
    } else {
        cx(LO, LO + R);
    }
}
template <int LO, int N, class Cx>
__device__ __forceinline__ void net_sort(const Cx &cx) {
    if constexpr (N > 1) {
        net_sort<LO, N / 2>(cx);
        net_sort<LO + N / 2, N / 2>(cx);
        net_merge<LO, N, 1>(cx);
    }
}

// N packed pairs sorted in both halves, largest first.
template <int N>
__device__ __forceinline__ void sort_desc(uint32_t (&v)[N]) {
    net_sort<0, N>([&](int i, int j) { ce(v[i], v[j]); });
}

// a = the N largest of two lists a and b sorted largest first, sorted again:
// max(a_i, b_(N-1-i)) are those N as a bitonic sequence.
template <int N>
__device__ __forceinline__ void merge_top(uint32_t (&a)[N], const uint32_t (&b)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) a[i] = h2max(a[i], b[N - 1 - i]);
#pragma unroll
    for (int h = N / 2; h >= 1; h >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i)
            if ((i & h) == 0) ce(a[i], a[i + h]);
}

// Byte address of float4 chunk c of box b of this lane's row in a swizzled tile.
__device__ __forceinline__ unsigned char *sel_chunk(unsigned char *tile, int b, int c, int lane) {
    return tile + b * kSelBoxBytes + lane * 128 + ((c ^ (lane & 7)) << 4);
}
__device__ __forceinline__ float sel_value(unsigned char *tile, int e, int lane) {
    return reinterpret_cast<const float *>(sel_chunk(tile, e >> 5, (e & 31) >> 2, lane))[e & 3];
}

// The KP largest values of boxes [b0, b1) of this lane's row at fp16 precision,
// largest first (the same list in both halves).
template <int KP>
__device__ __forceinline__ void topk_lists(unsigned char *tile, int b0, int b1, int lane,
                                           uint32_t (&top)[KP]) {
    // one copy of the code for every box: with two boxes unrolled the warps,
    // each at another place of a longer kernel, waited for instructions
    // (2.2 cycles per issue against 0.4)
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        constexpr int G = 16 / KP;  // packed groups of KP pairs in 32 experts
        uint32_t h[G][KP];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int c = 0; c < KP / 4; ++c) {
                const float4 x = *reinterpret_cast<const float4 *>(
                    sel_chunk(tile, b, (2 * g) * (KP / 4) + c, lane));
                const float4 y = *reinterpret_cast<const float4 *>(
                    sel_chunk(tile, b, (2 * g + 1) * (KP / 4) + c, lane));
                h[g][4 * c] = pack_rz(x.x, y.x);
                h[g][4 * c + 1] = pack_rz(x.y, y.y);
                h[g][4 * c + 2] = pack_rz(x.z, y.z);
                h[g][4 * c + 3] = pack_rz(x.w, y.w);
            }
#pragma unroll
        for (int g = 0; g < G; ++g) sort_desc<KP>(h[g]);
#pragma unroll
        for (int s = 1; s < G; s <<= 1)
#pragma unroll
            for (int g = 0; g + s < G; g += 2 * s) merge_top<KP>(h[g], h[g + s]);
        if (b == b0) {
#pragma unroll
            for (int i = 0; i < KP; ++i) top[i] = h[0][i];
        } else {
            merge_top<KP>(top, h[0]);
        }
    }
    // the halves' lists against each other: the same list in both
    uint32_t other[KP];
#pragma unroll
    for (int i = 0; i < KP; ++i) other[i] = __byte_perm(top[i], 0u, 0x1032);
    merge_top<KP>(top, other);
}

// The smallest fp32 that rounds (towards zero) to the k-th largest value of
// the sorted list top, or of top and other together.
template <int KP>
__device__ __forceinline__ float topk_bound(uint32_t (&top)[KP], const uint32_t *other, int k) {
    uint32_t kth;
    if (other && k == KP) {  // the smallest of the KP largest of both
        kth = h2max(top[0], other[(KP - 1) * 32]);
#pragma unroll
        for (int i = 1; i < KP; ++i) kth = h2min(kth, h2max(top[i], other[(KP - 1 - i) * 32]));
    } else {
        if (other) {
            uint32_t o[KP];
#pragma unroll
            for (int i = 0; i < KP; ++i) o[i] = other[i * 32];
            merge_top<KP>(top, o);
        }
        kth = top[0];
#pragma unroll
        for (int i = 1; i < KP; ++i) kth = (i < k) ? top[i] : kth;
    }
    kth &= 0xFFFFu;
    if (kth > 0u && kth < 0x8000u) return __half2float(__ushort_as_half((unsigned short)kth));
    // minus infinity is the image of nothing else (-inf - -inf is a NaN without
    // a sign bit: not below)
    if (kth == 0xFC00u) return -INFINITY;
    // zero or negative: the fp32 values that round to it reach down to, but
    // not as far as, the next fp16 below
    uint32_t mag = kth & 0x7FFFu;
    if (mag > 0x7BFFu) mag = 0x7BFFu;
    const float next = __half2float(__ushort_as_half((unsigned short)(mag + 1u)));
    return __uint_as_float((__float_as_uint(next) - 1u) | 0x80000000u);
}

// Top-K of this lane's row of NB boxes (the tile is only read): the chosen
// experts in ascending order.  Two passes without data-dependent branches or
// addresses (see topk_lists and select.cuh), then the drop of the candidates
// that share the k-th value's fp16 image beyond k, a row at a time by the whole
// warp.  (The router step at T = 32768, H = 2048 takes 129.6 us with it against
// 130.3 with K rounds of an argmax over 16 group maxima.)
template <int NB, int K>
__device__ __forceinline__ void select_net(unsigned char *tile, int lane, bool valid, int (&sel)[K]) {
    constexpr int KP = K <= 4 ? 4 : K;
    static_assert(KP == 4 || KP == 8 || KP == 16, "list length");
    uint32_t top[KP];
    topk_lists<KP>(tile, 0, NB, lane, top);
    const float bound = topk_bound<KP>(top, nullptr, K);
    uint32_t cand[NB];  // bit 31 - j of word b: expert 32 b + j
    int cnt = 0;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        uint32_t below = 0u;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float4 v = *reinterpret_cast<const float4 *>(sel_chunk(tile, b, c, lane));
            below = __funnelshift_l(__float_as_uint(v.x - bound), below, 1);
            below = __funnelshift_l(__float_as_uint(v.y - bound), below, 1);
            below = __funnelshift_l(__float_as_uint(v.z - bound), below, 1);
            below = __funnelshift_l(__float_as_uint(v.w - bound), below, 1);
        }
        cand[b] = valid ? ~below : 0u;
        cnt += __popc(cand[b]);
    }
    // rows with more than K: the smallest values first, equal ones from the
    // highest index on (a lane per expert of a box)
    unsigned todo = __ballot_sync(kFull, cnt > K);
    while (todo) {
        const int r = __ffs(todo) - 1;
        todo &= todo - 1;
        int rem = __shfl_sync(kFull, cnt, r) - K;
        while (rem > 0) {
            uint32_t key[NB], low = 0xFFFFFFFFu;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const uint32_t m = __shfl_sync(kFull, cand[b], r);
                const float v = *reinterpret_cast<const float *>(sel_chunk(tile, b, lane >> 2, r) + 4 * (lane & 3)) + 0.0f;
                const uint32_t x = __float_as_uint(v);
                const uint32_t o = x ^ ((x >> 31) ? 0xFFFFFFFFu : 0x80000000u);
                key[b] = ((m >> (31 - lane)) & 1u) ? o : 0xFFFFFFFFu;
                low = min(low, key[b]);
            }
            low = __reduce_min_sync(kFull, low);
            if (low == 0xFFFFFFFFu) break;
#pragma unroll
            for (int b = NB - 1; b >= 0; --b) {
                unsigned eq = __ballot_sync(kFull, key[b] == low);
                while (__popc(eq) > rem) eq &= eq - 1;  // the lowest ones stay
                rem -= __popc(eq);
                if (lane == r) cand[b] &= ~__brev(eq);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
        uint32_t w = cand[0];
        int b = 0;
#pragma unroll
        for (int i = 1; i < NB; ++i)
            if (w == 0u) {
                w = cand[i];
                b = i;
            }
        const int j = __clz(w) & 31;
        sel[q] = 32 * b + j;
        const uint32_t bit = 0x80000000u >> j;
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (i == b) cand[i] &= ~bit;
    }
}

}  // namespace
}  // namespace dol
