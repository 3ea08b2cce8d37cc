// Reduction of the selection CTAs' triangles of distances (tri_chunk): the
// Hamming distance
//   D_ab = n_a + n_b - 2 c_ab, c_ab = sum_t f_at f_bt           (App. C.3)
// is a sum over tokens, and so the sum of the CTAs' own; the diagonal holds 2 n_a.
// Alongside, Eq. origin_do: sum over a != b of D_ab^2 (exact integer
// adds, one per CTA).
// A CTA owns 32 consecutive triangle words; its warps
// each sum a strided subset of the partials with independent loads, and the
// warp sums are added in a fixed order, so D is an exact integer result
// independent of scheduling.  The kernel writes both halves of the symmetric D
// and the counts.
#include <cuda_fp16.h>

#include <climits>

#include "dol_internal.cuh"
#include "tma.cuh"

namespace dol {
namespace {

// Bound by L2 latency (1.75 us of the E = 128, T = 65536 step, whose partials are
// 5 MB).  256 threads with 20 loads in flight: with 128, 512 and 1024 threads the
// step took 30.5, 31.0 and 31.1 against 30.2 us (the routed step with 1024: 55.8
// against 52.4), and with the search for (a, b) moved ahead of the dependency wait
// 31.3.
constexpr int kRedWarps = 8;
constexpr int kRedThreads = kRedWarps * 32;
constexpr int kRedLoads = 20;  // partials a warp requests at once
constexpr int kImgThreads = 1024;

template <int EP>
__global__ void __launch_bounds__(kRedThreads)
cooc_reduce_kernel(const uint32_t *__restrict__ partials, int P1, int E, int *__restrict__ D, int *__restrict__ counts, unsigned char *__restrict__ bimg,
                   int big, long long *__restrict__ origin_do, long long r_base, int r_mult) {
    constexpr int kWords = tri_words(EP);
    __shared__ uint32_t s_sum[kRedWarps][33];
    const int e = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int word = blockIdx.x * 32 + e;
    const int layer = blockIdx.y;
    pdl_wait();
    pdl_trigger();
    uint32_t acc = 0u;
    const uint32_t *base = partials + (size_t)layer * P1 * kWords + word;
    for (int p0 = wp; p0 < P1; p0 += kRedLoads * kRedWarps) {
        uint32_t v[kRedLoads];
#pragma unroll
        for (int u = 0; u < kRedLoads; ++u) {
            const int p = p0 + u * kRedWarps;
            v[u] = (word < kWords && p < P1) ? __ldg(base + (size_t)p * kWords) : 0u;
        }
#pragma unroll
        for (int u = 0; u < kRedLoads; ++u) acc += v[u];
    }
    s_sum[wp][e] = acc;
    __syncthreads();
    if (wp != 0) return;
    long long sq = 0;  // this word's part of sum_{a != b} D_ab^2
    if (word < kWords) {
        uint32_t c = 0;
#pragma unroll
        for (int q = 0; q < kRedWarps; ++q) c += s_sum[q][e];
        // word -> (a, b): the chunk of four columns whose range holds it
        int lo = 0, hi = EP / 4 - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tri_chunk(mid) <= word) lo = mid;
            else hi = mid - 1;
        }
        const int a = (word - tri_chunk(lo)) >> 2;
        const int b = 4 * lo + (word & 3);
        int *Dl = D + (size_t)layer * E * E;
        unsigned char *img = (EP <= 128 && bimg) ? bimg + (size_t)layer * bimg_bytes(EP) : nullptr;
        if (b < a) {
            // below the diagonal: nothing to write
        } else if (b >= E) {
            // padding of the width: the image's operand is zero there
            if (img) {
                put_pieces(img, EP, a, b, 0, 0);
                put_pieces(img, EP, b, a, 0, 0);
            }
        } else if (a == b) {
            const int n = (int)(c >> 1);
            Dl[a * E + a] = 0;
            counts[(size_t)layer * E + a] = n;
            // R_a = (E - 2k) n_a + T k (every row of the co-occurrence sums to k n_a)
            const long long r = r_base + (long long)r_mult * (long long)n;
            if (img) {
                reinterpret_cast<float *>(img + bimg_r_offset(EP))[a] = (float)r;
                if (big) put_pieces(img, EP, a, a, -32768, 0);
                else put_dprime(img, EP, a, a, true, (int)r);
            }
        } else {
            const int d = (int)c;
            Dl[a * E + b] = d;
            Dl[b * E + a] = d;
            if (img) {
                put_dprime(img, EP, a, b, false, d);
                put_dprime(img, EP, b, a, false, d);
            }
            sq = 2 * (long long)d * (long long)d;
        }
    }
    if (origin_do) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(kFull, sq, o);
        if (e == 0 && sq)
            atomicAdd(reinterpret_cast<unsigned long long *>(origin_do + layer), (unsigned long long)sq);
    }
}

template <int EP>
cudaError_t run_reduce(const uint32_t *partials, int P1, const Problem &p, int *D, int *counts,
                       unsigned char *bimg, bool big, long long *origin_do, cudaStream_t s) {
    constexpr int kWords = tri_words(EP);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((kWords + 31) / 32, (unsigned)p.L);
    cfg.blockDim = dim3(kRedThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const long long r_base = p.T * (long long)p.k;
    const int r_mult = p.E - 2 * p.k;
    return cudaLaunchKernelEx(&cfg, cooc_reduce_kernel<EP>, partials, P1, p.E, D, counts, bimg,
                              (int)big, origin_do, r_base, r_mult);
}

// The image of D' from a given matrix D (the split entry point's, or a matrix
// summed over ranks or micro-batches, Eq. global_do): off the diagonal D_ab, on
// it the marker, R_a = sum_{b != a} D_ab (D symmetric) in the image's tail.
// img_ok[layer] = 1, or 0 where the two fp16 pieces are not exact off the
// diagonal (0 <= D_ab < 2^22), D_aa != 0 or R_a does not fit int32: the loss
// kernel gathers that problem's rows from D.  Also Eq. origin_do and the loss kernels' done
// counters (each may be null).  One CTA per problem, 64 rows at a time; a
// thread builds one 16-byte chunk of row n of each piece (8 consecutive
// k = a) from D[n][a .. a + 7], the 16 threads of row n (a half warp) add R_n
// with shuffles, and the chunks are written whole (the 128-byte swizzle moves
// whole 16-byte chunks).
__global__ void __launch_bounds__(kImgThreads)
dprime_image_kernel(const int *__restrict__ D, int E, int EP, unsigned char *__restrict__ bimg,
                    int *__restrict__ img_ok, long long *__restrict__ origin_do, int *__restrict__ done) {
    __shared__ long long s_sq[kImgThreads / 32];
    const int layer = blockIdx.x;
    const int *Dl = D + (size_t)layer * E * E;
    unsigned char *img = bimg + (size_t)layer * bimg_bytes(EP);
    float *R = reinterpret_cast<float *>(img + bimg_r_offset(EP));
    pdl_wait();
    pdl_trigger();
    int ok = 1;
    long long sq = 0;
    const int a0 = 8 * ((int)threadIdx.x & 15);
#pragma unroll 2
    for (int n0 = 0; n0 < EP; n0 += kImgThreads / 16) {
        const int n = n0 + ((int)threadIdx.x >> 4);
        const int4 zero4 = make_int4(0, 0, 0, 0);
        const bool in = n < E;  // E a multiple of 4: whole int4s
        const int4 v0 = in && a0 < E ? __ldg(reinterpret_cast<const int4 *>(Dl + n * E + a0)) : zero4;
        const int4 v1 = in && a0 + 4 < E ? __ldg(reinterpret_cast<const int4 *>(Dl + n * E + a0 + 4)) : zero4;
        const int v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
        long long row = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (a0 + u == n) {
                ok &= v[u] == 0;
            } else {
                ok &= v[u] >= 0 && v[u] < (1 << 22);
                row += v[u];
                sq += (long long)v[u] * v[u];
            }
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) row += __shfl_xor_sync(kFull, row, o);
        ok &= row <= INT_MAX;
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            int h[2], l[2];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                dprime_pieces(false, v[u + x], &h[x], &l[x]);
                if (in && a0 + u + x == n) {
                    h[x] = -32768;
                    l[x] = 0;
                }
            }
            hw[u / 2] = (uint32_t)__half_as_ushort(half_piece(h[0])) |
                        ((uint32_t)__half_as_ushort(half_piece(h[1])) << 16);
            lw[u / 2] = (uint32_t)__half_as_ushort(half_piece(l[0])) |
                        ((uint32_t)__half_as_ushort(half_piece(l[1])) << 16);
        }
        if (n < EP && a0 < EP) {
            *reinterpret_cast<uint4 *>(img + sw128_k16_offset(n, a0, 2 * EP)) =
                make_uint4(hw[0], hw[1], hw[2], hw[3]);
            *reinterpret_cast<uint4 *>(img + sw128_k16_offset(EP + n, a0, 2 * EP)) =
                make_uint4(lw[0], lw[1], lw[2], lw[3]);
            if (a0 == 0) R[n] = (float)row;
        }
    }
    ok = __syncthreads_and(ok);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(kFull, sq, o);
    if ((threadIdx.x & 31) == 0) s_sq[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
        img_ok[layer] = ok;
        if (done) done[layer] = 0;
        if (origin_do) {
            long long sum = 0;
            for (int w = 0; w < kImgThreads / 32; ++w) sum += s_sq[w];
            origin_do[layer] = sum;
        }
    }
}

}  // namespace

cudaError_t launch_cooc_reduce(const uint32_t *partials, int P1, const Problem &p,
                               int *D, int *counts, unsigned char *bimg, bool big,
                               long long *origin_do, cudaStream_t s) {
    if (!cooc_sizes_ok(p.E, p.k) || (bimg && !bimg_sizes_ok(p.E, p.k))) return cudaErrorInvalidValue;
    switch (cooc_width(p.E)) {
        case 32: return run_reduce<32>(partials, P1, p, D, counts, bimg, big, origin_do, s);
        case 64: return run_reduce<64>(partials, P1, p, D, counts, bimg, big, origin_do, s);
        case 96: return run_reduce<96>(partials, P1, p, D, counts, bimg, big, origin_do, s);
        case 128: return run_reduce<128>(partials, P1, p, D, counts, bimg, big, origin_do, s);
        case 160: return run_reduce<160>(partials, P1, p, D, counts, bimg, big, origin_do, s);
        case 192: return run_reduce<192>(partials, P1, p, D, counts, bimg, big, origin_do, s);
        case 224: return run_reduce<224>(partials, P1, p, D, counts, bimg, big, origin_do, s);
        default: return run_reduce<256>(partials, P1, p, D, counts, bimg, big, origin_do, s);
    }
}

cudaError_t launch_dprime_image(const int *D, const Problem &p, unsigned char *bimg, int *img_ok,
                                long long *origin_do, int *done, cudaStream_t s) {
    if (!bimg_sizes_ok(p.E, p.k) || reinterpret_cast<uintptr_t>(D) % 16 != 0) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.L);
    cfg.blockDim = dim3(kImgThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, dprime_image_kernel, D, p.E, cooc_width(p.E), bimg, img_ok,
                              origin_do, done);
}

}  // namespace dol
