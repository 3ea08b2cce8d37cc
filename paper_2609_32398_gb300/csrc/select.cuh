// Step 1 (and, with E <= 256, the co-occurrence counts of the Hamming matrix):
// Top-K signatures (Sec. 3.1.1, Eq. 1) with one token per lane, for any
// E <= 512 that is a multiple of 4, k <= 16 and 16-byte aligned logits.
//
// A persistent CTA per SM owns a contiguous range of 32-token tiles.  One
// producer warp streams each tile [32 tokens x E] into a ring of shared
// memory slots with 2-D TMA loads (32 x 32 fp32 boxes, 128-byte swizzle, so a
// lane reading its own row is bank-conflict free); the consumer warps take the
// tiles in turn.  A lane finds the Top-K of its token in two passes over its
// row, neither of which has a data-dependent branch or address:
//   1. the k-th largest value at 11-bit precision: every value is rounded
//      towards zero to fp16 (a monotone map, one conversion per two values),
//      and a register list of the KP = 4, 8 or 16 largest is kept by sorting
//      networks on packed pairs (two lists per register, min/max on both at
//      once), merged 32 experts at a time;
//   2. a bit per expert: z >= L, L the smallest fp32 that rounds to the k-th
//      largest fp16 value, taken as the sign of z - L.
// The bits hold every member of the Top-K (the map is monotone) and, where
// values share the k-th one's fp16 image, a few more: those lanes drop the
// smallest of their candidates (equal values: the highest index first) until k
// are left.  At E = 128, k = 6 a tile takes 2,480 warp instructions in all, about
// half of them in either warp of its team (the argmax rounds of sig_fast.cuh, at
// k = 8: 1,780 in one warp).
//
// The lanes' rows of bits are turned into signature words by 32 x 32 bit
// transposes.  With kCooc the words are also written as fp8 columns of F^T
// (the tile's own slot holds them once the logits are read) and one thread
// adds F^T F on the tensor cores into an accumulator that stays in TMEM for
// the whole CTA: c_ab = sum_t f_at f_bt, exact (0/1 products, fp32 sums), in
// place of k (k - 1) / 2 shared-memory atomics per token.  At the end it goes
// out as the CTA's triangle of distances n_a + n_b - 2 c_ab.
// With routing outputs the lane also writes the chosen experts in selection
// order and their re-normalized combine weights (Sec. 3.1.1).
#pragma once

#include <climits>

#include "dol_internal.cuh"
#include "tma.cuh"
#include "topk_net.cuh"

namespace dol {

constexpr int kSelMaxSlots = 16;
// Most teams (pairs of consumer warps) and block size for lists of KP values
// (the launch bound of 896 threads keeps 72 registers a thread for KP <= 8).
constexpr int sel_max_teams(int KP) { return KP <= 8 ? 9 : 6; }
constexpr int sel_threads(int KP) { return (2 * sel_max_teams(KP) + 2) * 32; }
// Leaves room for two small CTAs of the next kernel on the SM.
constexpr int kSelMaxSmem = 226304;

// Shared memory of one launch: ring | barriers and flags | lists | masks | counters.
struct SelLayout {
    int nb;         // boxes of 32 experts per row
    int slots;      // ring slots (tiles in flight)
    int split;      // consumer warps per tile (a team): 2, each with half of the boxes (1 for one box)
    int teams;      // teams, each working on one tile at a time
    int consumers;  // consumer warps, at least four
    int off_bar;    // byte offsets behind the ring
    int off_list;
    int off_mask;
    int off_cnt;
    int total;      // bytes with the 1024-byte alignment slack
};

// tiles: the most tiles a CTA takes (no more slots and warps than those).
inline SelLayout sel_layout(int E, int KP, int64_t tiles) {
    SelLayout l;
    l.nb = (E + 31) / 32;
    l.split = l.nb > 1 ? 2 : 1;
    const int slot = l.nb * kSelBoxBytes;
    const int max_teams = l.split == 1 ? 2 * sel_max_teams(KP) : sel_max_teams(KP);
    for (int s = (int)min64(kSelMaxSlots, tiles); s >= 1; --s) {
        const int ring = s * slot;
        l.slots = s;
        l.teams = s;
        if (l.teams > max_teams) l.teams = max_teams;
        // the four lane quadrants of TMEM are read by four warps at least
        l.consumers = l.teams * l.split < 4 ? 4 : l.teams * l.split;
        l.off_bar = ring;
        l.off_list = (l.off_bar + 8 * (3 * s + 1) + 16 + 15) / 16 * 16;
        l.off_mask = l.off_list + (l.split > 1 ? l.teams * 2 * KP * 128 : 0);
        l.off_cnt = l.off_mask + l.teams * (l.nb + 2) * 128;
        l.total = l.off_cnt + 32 * l.nb * 4 + 1024;
        if (l.total <= kSelMaxSmem) break;
    }
    return l;
}

struct SelArgs {
    int64_t T, W;
    int E, k;
    int whole;        // E a multiple of 32: the tensor map is [E / 32][L T][32]
    SelLayout lay;
    uint32_t *bits;
    int *counts;      // not kCooc: the counts (zero on entry) or null
    uint32_t *cooc;   // kCooc: per-CTA triangles of distances of EP = 32 nb experts
    ZeroSpans zero;
    int *status;      // may be null
    uint8_t *idx;     // may be null: the chosen experts of every token, one byte each
    RouteOut route;
};

namespace {

// Barrier of the `n` threads of one tile's warps; the AND of ok over them.
__device__ __forceinline__ bool tile_sync_and(int id, int n, bool ok) {
    if (n == 32) return __all_sync(kFull, ok);
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %3, 0;\n\t"
        "barrier.cta.red.and.pred q, %1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(id), "r"(n), "r"((uint32_t)ok)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void tile_sync(int id, int n) {
    if (n == 32) __syncwarp();
    else asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Drops candidates of the rows of todo (a bit per row that holds cnt > k of
// them; cnt in the row's lane): the smallest values first, equal ones from the
// highest index on.  The warp takes one such row at a time, a lane per expert
// of a box, four boxes at once (0.5 rows of a tile of random logits at E = 128;
// a lane walking its own candidates one by one took 1 us per dropped
// candidate).  rows: word b * 32 + r holds row r's candidates of box b, bit
// 31 - j for expert 32 b + j.
__device__ __forceinline__ void drop_excess(unsigned char *tile, uint32_t *rows, int nb, int lane,
                                            unsigned todo, int cnt, int k) {
    while (todo) {
        const int r = __ffs(todo) - 1;
        todo &= todo - 1;
        int rem = __shfl_sync(kFull, cnt, r) - k;
        // this lane's experts of boxes b0 .. b0 + 3: their values as ordered
        // integers (-0.0 as +0.0), the largest one for no candidate
        uint32_t key[4];
        auto load = [&](int b0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int b = min(b0 + u, nb - 1);
                const uint32_t m = b0 + u < nb ? rows[b * 32 + r] : 0u;
                const float v = *reinterpret_cast<const float *>(sel_chunk(tile, b, lane >> 2, r) + 4 * (lane & 3)) + 0.0f;
                const uint32_t x = __float_as_uint(v);
                const uint32_t o = x ^ ((x >> 31) ? 0xFFFFFFFFu : 0x80000000u);
                key[u] = ((m >> (31 - lane)) & 1u) ? o : 0xFFFFFFFFu;
            }
        };
        bool dropped = true;
        while (rem > 0 && dropped) {
            uint32_t low = 0xFFFFFFFFu;
            for (int b0 = 0; b0 < nb; b0 += 4) {
                load(b0);
                low = min(low, min(min(key[0], key[1]), min(key[2], key[3])));
            }
            low = __reduce_min_sync(kFull, low);
            dropped = false;
            if (low == 0xFFFFFFFFu) break;
            for (int b0 = (nb - 1) & ~3; b0 >= 0 && rem > 0; b0 -= 4) {
                if (nb > 4) load(b0);
#pragma unroll
                for (int u = 3; u >= 0; --u) {
                    unsigned eq = __ballot_sync(kFull, key[u] == low);
                    const int n = __popc(eq);
                    if (n == 0 || rem <= 0) continue;
                    while (n > rem && __popc(eq) > rem) eq &= eq - 1;  // keep the lowest ones as candidates
                    rem -= __popc(eq);
                    __syncwarp();
                    if (lane == 0) rows[(b0 + u) * 32 + r] &= ~__brev(eq);
                    dropped = true;
                }
            }
            __syncwarp();
        }
    }
}

// The chosen experts of one token in selection order (largest value first,
// equal values lower index first) and their values, from the candidate masks.
template <int KP>
__device__ __forceinline__ void chosen_sorted(unsigned char *tile, const uint32_t *masks, int nb,
                                              int lane, int k, int (&sel)[KP], float (&val)[KP]) {
    int b = 0;
    uint32_t m = masks[0];
#pragma unroll
    for (int q = 0; q < KP; ++q) {
        sel[q] = INT_MAX;
        val[q] = -INFINITY;
        if (q < k) {
            while (m == 0u && b + 1 < nb) m = masks[32 * ++b];
            const int j = m ? __clz(m) : 0;
            m &= ~(0x80000000u >> j);
            sel[q] = 32 * b + j;
            val[q] = sel_value(tile, sel[q], lane);
        }
    }
    net_sort<0, KP>([&](int x, int y) {
        const bool swap = val[y] > val[x] || (val[y] == val[x] && sel[y] < sel[x]);
        const float vx = val[x], vy = val[y];
        const int ex = sel[x], ey = sel[y];
        val[x] = swap ? vy : vx;
        val[y] = swap ? vx : vy;
        sel[x] = swap ? ey : ex;
        sel[y] = swap ? ex : ey;
    });
}

// ids and weights of one token (Sec. 3.1.1): w_q = u_q / sum_q' u_q', u from
// route_raw_weight, summed in selection order.
template <int KP>
__device__ __forceinline__ void write_route(const RouteOut &r, int64_t off, int k, const int (&sel)[KP],
                                            const float (&val)[KP]) {
    float w[KP], part[KP];
#pragma unroll
    for (int q = 0; q < KP; ++q) part[q] = w[q] = q < k ? route_raw_weight(val[q], val[0], r.gate) : 0.0f;
    // by halves: a third of the rounding error of a running sum at k = 8
#pragma unroll
    for (int h = KP / 2; h >= 1; h >>= 1)
#pragma unroll
        for (int q = 0; q < h; ++q) part[q] += part[q + h];
    const float sum = part[0];
    // w / sum by the reciprocal of the sum and one Newton step
    const float inv = 1.0f / sum;
#pragma unroll
    for (int q = 0; q < KP; ++q) {
        const float t = w[q] * inv;
        w[q] = fmaf(inv, fmaf(-t, sum, w[q]), t);
    }
    int *ids = r.ids + off;
    float *cw = r.combine + off;
    const uintptr_t al = reinterpret_cast<uintptr_t>(r.ids) | reinterpret_cast<uintptr_t>(r.combine);
    if ((k & 3) == 0 && (al & 15) == 0) {
#pragma unroll
        for (int q = 0; q < KP; q += 4)
            if (q < k) {
                *reinterpret_cast<int4 *>(ids + q) = make_int4(sel[q], sel[q + 1], sel[q + 2], sel[q + 3]);
                *reinterpret_cast<float4 *>(cw + q) = make_float4(w[q], w[q + 1], w[q + 2], w[q + 3]);
            }
    } else {
#pragma unroll
        for (int q = 0; q < KP; ++q)
            if (q < k) {
                ids[q] = sel[q];
                cw[q] = w[q];
            }
    }
}

// The chosen experts as one byte each (E <= 256).
template <int KP>
__device__ __forceinline__ void write_idx(uint8_t *p, int k, const int (&sel)[KP]) {
#pragma unroll
    for (int q = 0; q < KP; q += 4) {
        const uint32_t v = (uint32_t)(sel[q] & 255) | ((uint32_t)(sel[q + 1] & 255) << 8) |
                           ((uint32_t)(sel[q + 2] & 255) << 16) | ((uint32_t)(sel[q + 3] & 255) << 24);
        if ((k & 3) == 0) {  // rows of 4 or 8 bytes
            if (q < k) *reinterpret_cast<uint32_t *>(p + q) = v;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q + u < k) p[q + u] = (uint8_t)(v >> (8 * u));
        }
    }
}

// Shared-memory matrix descriptor of a K-major operand without swizzle: 8-row
// x 16-byte core matrices, `lbo` bytes between the two 16-byte columns of one
// K = 32-byte step, `sbo` bytes between 8-row groups, descriptor version 1.
__device__ __forceinline__ uint64_t umma_desc_plain(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) |
           ((uint64_t)(sbo >> 4) << 32) | ((uint64_t)1 << 46);
}

// D[tmem] (+)= A[smem] B[smem], kind::f8f6f4 (e4m3), one CTA.
__device__ __forceinline__ void umma_f8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                        uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Row e of F^T for the tile's 32 tokens (the signature word of expert e) as 32
// fp8 values 0 or 2 (0x40), in the tile's core matrices.  The tokens are taken
// in the order bit j, 8 + j, 16 + j, 24 + j of byte group j: any order will do
// for a sum over tokens, as long as it is the same for every expert.
__device__ __forceinline__ void write_f_row(unsigned char *f, int e, uint32_t word) {
    uint32_t r[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        r[j] = (j <= 6 ? word << (6 - j) : word >> 1) & 0x40404040u;
    unsigned char *p = f + (e >> 3) * 256 + (e & 7) * 16;
    *reinterpret_cast<uint4 *>(p) = make_uint4(r[0], r[1], r[2], r[3]);
    *reinterpret_cast<uint4 *>(p + 128) = make_uint4(r[4], r[5], r[6], r[7]);
}

template <int KP, bool kCooc>
__global__ void __launch_bounds__(KP <= 8 ? 896 : sel_threads(KP), 1)
select_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ SelArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = smem_align<1024>(smem_raw);
    const int nb = a.lay.nb, slots = a.lay.slots, consumers = a.lay.consumers;
    const int slot_bytes = nb * kSelBoxBytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + a.lay.off_bar);  // logits loaded
    uint64_t *empty = full + slots;    // slot free again
    uint64_t *fready = empty + slots;  // kCooc: F^T of the tile written
    uint64_t *acc_done = fready + slots;
    volatile int *s_abort = reinterpret_cast<volatile int *>(acc_done + 1);
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(const_cast<int *>(s_abort + 1));
    int *s_cnt = reinterpret_cast<int *>(smem + a.lay.off_cnt);  // [32 nb]

    pdl_trigger();
    // this CTA: layer blockIdx.y, a contiguous range of its 32-token tiles
    const int64_t layer = blockIdx.y;
    const int64_t tb = a.W * (int64_t)blockIdx.x / gridDim.x;
    const int n = (int)(a.W * (int64_t)(blockIdx.x + 1) / gridDim.x - tb);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int E = a.E, k = a.k;
    if (!kCooc)
        for (int i = threadIdx.x; i < 32 * nb; i += blockDim.x) s_cnt[i] = 0;
    if (warp == 0) {  // a lane per slot (at most 16)
        if (lane < slots) {
            mbar_init(&full[lane], 1);
            mbar_init(&empty[lane], kCooc ? 1 : a.lay.split);
            mbar_init(&fready[lane], a.lay.split);
        }
        if (lane == 31) {
            mbar_init(acc_done, 1);
            *s_abort = 0;
        }
        fence_barrier_init();
    }
    if (warp == consumers && lane == 0) prefetch_tensormap(&tmap);
    __syncthreads();
    // Launched as a programmatic dependent of whatever ran before on the
    // stream: wait for it before touching global memory (it may have written
    // the logits, or still read the accumulators cleared below) and before
    // taking TMEM (a kernel before this one may still have to allocate its own).
    pdl_wait();

    const int tmem_cols = nb <= 4 ? 128 : 512;
    if (warp == consumers) {  // producer
        if (lane == 0 && n > 0) {
            int issued = 0;
            for (int q = 0, s = 0, round = 0; q < n; ++q) {
                if (round > 0 && !mbar_wait(&empty[s], (round - 1) & 1, a.status)) {
                    *s_abort = 1;
                    break;
                }
                if (*s_abort) break;
                const int y = (int)(layer * a.T + 32 * (tb + q));
                mbar_arrive_expect_tx(&full[s], slot_bytes);
                unsigned char *dst = smem + (size_t)s * slot_bytes;
                if (a.whole) {  // the tile's boxes in one copy
                    tma_load_3d(dst, &tmap, 0, y, 0, &full[s]);
                } else {
                    for (int b = 0; b < nb; ++b)
                        tma_load_2d(dst + b * kSelBoxBytes, &tmap, b * 32, y, &full[s]);
                }
                issued = q + 1;
                if (++s == slots) {
                    s = 0;
                    ++round;
                }
            }
            // Every issued load completes before the CTA may exit.
            for (int q = issued > slots ? issued - slots : 0; q < issued; ++q)
                mbar_wait(&full[q % slots], (q / slots) & 1, a.status);
        }
        __syncwarp();
    } else if (warp == consumers + 1) {  // accumulators to clear, tensor-core issuer
        for (int z = 0; z < 3; ++z)
            for (int64_t i = (int64_t)blockIdx.x * 32 + lane; i < a.zero.n[z]; i += (int64_t)gridDim.x * 32)
                a.zero.p[z][i] = 0;
        if (kCooc) {
            tmem_alloc(s_tmem, tmem_cols);
            __syncwarp();
            const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(s_tmem);
            if (lane == 0 && n > 0) {
                const int EP = 32 * nb;
                // kind::f8f6f4: fp32 accumulate, e4m3 A and B, both K-major, M = 128
                const uint32_t base = (1u << 4) | (8u << 24);
                const uint32_t idesc1 = base | ((uint32_t)(EP >> 3) << 17);
                const uint32_t idesc2 = base | ((uint32_t)((EP - 128) >> 3) << 17);
                for (int q = 0, s = 0, round = 0; q < n; ++q) {
                    if (!mbar_wait(&fready[s], round & 1, a.status)) *s_abort = 1;
                    if (*s_abort) break;
                    tc_fence_after();
                    const uint32_t f = smem_u32(smem + (size_t)s * slot_bytes);
                    umma_f8(tmem, umma_desc_plain(f, 128, 256), umma_desc_plain(f, 128, 256), idesc1,
                            q > 0 ? 1u : 0u);
                    if (EP > 128)  // experts 128 .. against themselves
                        umma_f8(tmem + 256, umma_desc_plain(f + 4096, 128, 256),
                                umma_desc_plain(f + 4096, 128, 256), idesc2, q > 0 ? 1u : 0u);
                    umma_commit(&empty[s]);
                    if (++s == slots) {
                        s = 0;
                        ++round;
                    }
                }
                umma_commit(acc_done);
                // the tensor cores must be done with the slots and TMEM
                if (!mbar_wait(acc_done, 0, a.status)) *s_abort = 1;
            }
            __syncwarp();
        }
    } else if (warp < a.lay.teams * a.lay.split) {  // consumers: a team takes every teams-th tile
        const int split = a.lay.split, teams = a.lay.teams;
        const int team = split > 1 ? warp >> 1 : warp, part = split > 1 ? warp & 1 : 0;
        const int threads = 32 * split, bar_id = 1 + team;
        const int bm = (nb + 1) / 2;  // boxes of the first warp
        const int b0 = part == 0 ? 0 : bm, b1 = (part == 0 && split > 1) ? bm : nb;
        const uint32_t in_last = (E & 31) ? kFull << (32 - (E & 31)) : kFull;  // columns of the last box below E
        uint32_t *list = reinterpret_cast<uint32_t *>(smem + a.lay.off_list) + team * 2 * KP * 32 + lane;
        uint32_t *masks = reinterpret_cast<uint32_t *>(smem + a.lay.off_mask) + team * (nb + 2) * 32 + lane;
        for (int q = team, s = team, round = 0; q < n; q += teams, s += teams) {
            if (s >= slots) {  // teams <= slots
                s -= slots;
                ++round;
            }
            unsigned char *tile = smem + (size_t)s * slot_bytes;
            // The slot's previous tile was another team's: until it is freed
            // a test of `full` by parity could still see the round before it.
            // Both warps of the team go on, or leave, together.
            const bool ok = !*s_abort &&
                            (round == 0 || mbar_wait(&empty[s], (round - 1) & 1, a.status)) &&
                            mbar_wait(&full[s], round & 1, a.status);
            const int64_t w = tb + q;
            const int64_t t = 32 * w + lane;
            const bool valid = t < a.T;
            if ((E & 31) && part == split - 1) {  // the last box's columns past E: never chosen
                const float4 none = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                for (int c = (E & 31) >> 2; c < 8; ++c)
                    *reinterpret_cast<float4 *>(sel_chunk(tile, nb - 1, c, lane)) = none;
            }
            uint32_t top[KP];
            topk_lists<KP>(tile, b0, b1, lane, top);
            if (split > 1) {
#pragma unroll
                for (int i = 0; i < KP; ++i) list[(part * KP + i) * 32] = top[i];
            }
            if (!tile_sync_and(bar_id, threads, ok)) {
                *s_abort = 1;
                break;
            }
            const float bound = topk_bound<KP>(top, split > 1 ? list + (part ^ 1) * KP * 32 : nullptr, k);
            int cnt = 0;
#pragma unroll 1
            for (int b = b0; b < b1; ++b) {
                uint32_t below = 0u;  // bit 31 - j: expert 32 b + j is below the bound
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 v = *reinterpret_cast<const float4 *>(sel_chunk(tile, b, c, lane));
                    below = __funnelshift_l(__float_as_uint(v.x - bound), below, 1);
                    below = __funnelshift_l(__float_as_uint(v.y - bound), below, 1);
                    below = __funnelshift_l(__float_as_uint(v.z - bound), below, 1);
                    below = __funnelshift_l(__float_as_uint(v.w - bound), below, 1);
                }
                const uint32_t cand = valid ? ~below & (b == nb - 1 ? in_last : kFull) : 0u;
                cnt += __popc(cand);
                masks[b * 32] = cand;
            }
            if (split > 1) masks[(nb + part) * 32] = (uint32_t)cnt;
            tile_sync(bar_id, threads);
            // each warp of the team takes half of the rows with too many
            if (split > 1) cnt += (int)masks[(nb + (part ^ 1)) * 32];
            unsigned todo = __ballot_sync(kFull, cnt > k);
            if (split > 1) todo &= part ? 0xFFFF0000u : 0xFFFFu;
            if (todo) drop_excess(tile, masks - lane, nb, lane, todo, cnt, k);
            if (a.route.ids || a.idx) {
                tile_sync(bar_id, threads);
                if (part == 0 && valid) {
                    int sel[KP];
                    float val[KP];
                    chosen_sorted<KP>(tile, masks, nb, lane, k, sel, val);
                    const int64_t off = (layer * a.T + t) * k;
                    if (a.route.ids) write_route<KP>(a.route, off, k, sel, val);
                    if (a.idx) write_idx<KP>(a.idx + off, k, sel);
                }
            }
            tile_sync(bar_id, threads);  // masks final, every row read: the slot may hold F^T
            uint32_t *words = a.bits + layer * E * a.W + w;
#pragma unroll 1
            for (int b = b0; b < b1; ++b) {
                const uint32_t word = transpose32_bits(__brev(masks[b * 32]), lane);
                const int e = 32 * b + lane;
                if (e < E) words[(int64_t)e * a.W] = word;
                if (kCooc) write_f_row(tile, e, word);
                else if (a.counts && word) atomicAdd(&s_cnt[e], __popc(word));
            }
            // hand the slot on: to the tensor cores, which free it, or back to
            // the producer
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(kCooc ? &fready[s] : &empty[s]);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (kCooc) {
        // this CTA's triangle, TMEM -> registers -> global, for the reduction
        // kernel: first the counts n_a = c_aa, then n_a + n_b - 2 c_ab (2 n_a on
        // the diagonal)
        const int EP = 32 * nb;
        const int words = tri_words(EP);
        uint32_t *tri = a.cooc + ((size_t)layer * gridDim.x + blockIdx.x) * (size_t)words;
        const bool any = n > 0 && !*s_abort;
        const uint32_t tmem = any ? *s_tmem : 0u;
        const int quad = warp & 3;
        const uint32_t tquad = tmem + ((uint32_t)(32 * quad) << 16);
        auto block_col = [](int blk, int cb) { return (uint32_t)(blk ? 256 + 32 * (cb - 4) : 32 * cb); };
        uint32_t r[32];
        if (any && warp < 4) {
            for (int cb = quad; cb < nb; cb += 4) {  // the diagonal block of rows 32 cb ..
                tmem_ld32(tquad + block_col(cb >> 2, cb), r);
                tmem_wait_ld();
                uint32_t na = r[0];
#pragma unroll
                for (int c = 1; c < 32; ++c) na = lane == c ? r[c] : na;
                s_cnt[32 * cb + lane] = (int)(__uint_as_float(na) * 0.25f);
            }
        }
        __syncthreads();
        if (!any) {
            for (int i = threadIdx.x; i < words; i += blockDim.x) tri[i] = 0u;
        } else if (warp < (consumers & ~3)) {
            const int per = consumers >> 2;
            const int nblk = nb <= 4 ? 1 : 2;
            for (int item = warp >> 2; item < nblk * nb; item += per) {
                const int blk = item / nb, cb = item - blk * nb;
                const int row0 = 128 * blk + 32 * quad;
                if (row0 >= EP || 32 * cb + 31 < row0) continue;
                const int row = row0 + lane;
                tmem_ld32(tquad + block_col(blk, cb), r);
                tmem_wait_ld();
                const int na = s_cnt[row];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int4 nc = *reinterpret_cast<const int4 *>(s_cnt + 32 * cb + 4 * c);
                    const int n4[4] = {nc.x, nc.y, nc.z, nc.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        // 2 c_ab (F holds 2 instead of 1: the accumulator is 4 c_ab)
                        const int both = 32 * cb + 4 * c + u == row ? 0 : (int)(__uint_as_float(r[4 * c + u]) * 0.5f);
                        r[4 * c + u] = (uint32_t)(na + n4[u] - both);
                    }
                    if (32 * cb + 4 * c + 4 > row)
                        *reinterpret_cast<uint4 *>(tri + tri_chunk(8 * cb + c) + 4 * row) =
                            make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
                }
            }
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (warp == consumers + 1) tmem_dealloc(*s_tmem, tmem_cols);
    } else if (a.counts) {
        for (int e = threadIdx.x; e < E; e += blockDim.x)
            if (s_cnt[e]) atomicAdd(&a.counts[layer * E + e], s_cnt[e]);
    }
}

}  // namespace
}  // namespace dol
