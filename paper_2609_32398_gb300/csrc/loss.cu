// Step 3: the surrogate DO-loss and its gradient to the router logits.
//
// Eq. do_loss (Sec. 3.1.3) with G = d_scale * D detached (Eq. global_do):
//   L = 1/(m^2 k) sum_i sum_j G_ij C_ij,   C_ij = sum_t p_it (f_it - f_jt).
// Summing over j first turns the double sum into one integer weight per
// token and expert:
//   sum_j G_ij (f_it - f_jt) = d_scale * w_it,
//   w_it = f_it R_i - sum_{j in S_t} D_ij,   R_i = sum_j D_ij,
// so L = d_scale/(m^2 k) sum_t A_t with A_t = sum_i p_it w_it, and
// dL/dp_it = d_scale w_it / (m^2 k).  Through the gate (S = sum_i s_it):
//   sigmoid-norm  dz_lt = c s_lt (1 - s_lt) / S (w_lt - A_t)
//   softmax       dz_lt = c p_lt (w_lt - A_t)
// with c = grad_scale * d_scale / (m^2 k).  w is exact in int32; A_t is
// accumulated in fp32 inside a token and in fp64 across tokens, in a fixed
// order.  The k-row gather of D reads rows of D, which relies on D being
// symmetric (every Hamming matrix, and every sum of them, is).
#include <climits>

#include "dol_internal.cuh"

namespace dol {
namespace {

constexpr size_t kSmemDLimit = 200 * 1024;

__device__ __forceinline__ float sigmoid_f(float z) {
    // exp of at most 80 keeps 1 + e finite, so the fast divide stays exact enough
    const float e = __expf(-fmaxf(z, -80.0f));
    return __fdividef(1.0f, 1.0f + e);
}

// Warps per CTA: fewer where a lane holds many experts (registers).
template <int R>
constexpr int loss_warps() { return R <= 8 ? 16 : 8; }
constexpr int kListMax = 64;  // chosen experts of a token listed in shared memory

// A warp per token: lanes hold experts i = lane + 32 r (r < R).  The tokens of a
// signature word are split over `split` warps (a power of two), so that a short
// window still fills the GPU: with 32 tokens in turn per warp the kernel took
// 170 of 202 us at E = 200, T = 2539.  The k chosen rows of D are read four at
// a time.
template <int R, bool kSmemD, int kGate>
__global__ void __launch_bounds__(loss_warps<R>() * 32)
loss_generic_kernel(const float *__restrict__ logits, const uint32_t *__restrict__ bits,
                    const int *__restrict__ Dg, const int *__restrict__ counts, int64_t T, int E, int k,
                    int64_t W, int split, float coef, float *__restrict__ dlogits,
                    double *__restrict__ partials, int P, int *__restrict__ status) {
    constexpr int kLossWarps = loss_warps<R>();
    extern __shared__ __align__(16) int smem[];
    __shared__ double s_part[kLossWarps];
    __shared__ int s_list[kLossWarps][kListMax];
    int *sD = smem;
    int *sR = smem + (kSmemD ? E * E : 0);

    const int layer = blockIdx.y;
    const int *Dl = Dg + (int64_t)layer * E * E;
    const float *z = logits + (int64_t)layer * T * E;
    float *dz = dlogits ? dlogits + (int64_t)layer * T * E : nullptr;
    const uint32_t *bl = bits + (int64_t)layer * E * W;

    if (kSmemD) {
        if ((E & 3) == 0 && (reinterpret_cast<uintptr_t>(Dl) & 15) == 0) {
#pragma unroll 4
            for (int q = threadIdx.x; q < E * E / 4; q += blockDim.x)
                reinterpret_cast<int4 *>(sD)[q] = __ldg(reinterpret_cast<const int4 *>(Dl) + q);
        } else {
            for (int q = threadIdx.x; q < E * E; q += blockDim.x) sD[q] = __ldg(Dl + q);
        }
        __syncthreads();
    }
    const int *Dsrc = kSmemD ? sD : Dl;
    for (int i = threadIdx.x; i < E; i += blockDim.x) {
        // R_i = (E - 2k) n_i + T k for the matrix of the same tokens, else a
        // column sum (D symmetric)
        long long acc = 0;
        if (counts) {
            acc = (long long)(E - 2 * k) * counts[(int64_t)layer * E + i] + (long long)T * k;
        } else {
#pragma unroll 8
            for (int j = 0; j < E; ++j) acc += Dsrc[(int64_t)j * E + i];
        }
        if (acc > INT_MAX || acc < 0) atomicOr(status, kDevOverflow);
        sR[i] = (int)acc;
    }
    __syncthreads();

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    int *list = s_list[warp];
    double tok_sum = 0.0;  // sum of A_t over this warp's tokens (meaningful in lane 0)
    const int per = 32 / split;

    for (int64_t item = (int64_t)blockIdx.x * kLossWarps + warp; item < W * split;
         item += (int64_t)P * kLossWarps) {
        const int64_t w = item / split;
        const int tt0 = (int)(item - w * split) * per;
        uint32_t bw[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r;
            bw[r] = (i < E) ? __ldg(bl + (int64_t)i * W + w) : 0u;
        }
        const int nt = (int)min64(tt0 + per, T - w * 32);
        for (int tt = tt0; tt < nt; ++tt) {
            const int64_t t = w * 32 + tt;
            const float *zt = z + t * E;
            float zr[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = lane + 32 * r;
                zr[r] = (i < E) ? __ldg(zt + i) : 0.0f;
            }
            int acc[R];
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = 0;
            // sum_{j in S_t} D_ji for this lane's experts i
            if (k <= kListMax) {
                int n = 0;
#pragma unroll
                for (int rr = 0; rr < R; ++rr) {
                    const unsigned m = __ballot_sync(kFull, (bw[rr] >> tt) & 1u);
                    const int at = n + __popc(m & ((1u << lane) - 1u));
                    if (((m >> lane) & 1u) && at < kListMax) list[at] = 32 * rr + lane;
                    n += __popc(m);
                }
                n = min(n, kListMax);
                __syncwarp();
                for (int q = 0; q < n; q += 4) {
                    const int *row[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) row[u] = Dsrc + (int64_t)list[min(q + u, n - 1)] * E;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int i = lane + 32 * r;
                        if (i < E) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int d = row[u][i];
                                acc[r] += q + u < n ? d : 0;
                            }
                        }
                    }
                }
                __syncwarp();
            } else {
#pragma unroll
                for (int rr = 0; rr < R; ++rr) {
                    unsigned m = __ballot_sync(kFull, (bw[rr] >> tt) & 1u);
                    while (m) {
                        const int j = 32 * rr + __ffs(m) - 1;
                        m &= m - 1;
                        const int *row = Dsrc + (int64_t)j * E;
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const int i = lane + 32 * r;
                            if (i < E) acc[r] += row[i];
                        }
                    }
                }
            }
            float wr[R], g[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = lane + 32 * r;
                const bool f = (bw[r] >> tt) & 1u;
                wr[r] = (float)(f ? sR[i] - acc[r] : -acc[r]);
            }
            float num = 0.0f, den = 0.0f;
            if (kGate == 0) {  // sigmoid-norm
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = lane + 32 * r;
                    g[r] = (i < E) ? sigmoid_f(zr[r]) : 0.0f;
                    den += g[r];
                    num += g[r] * wr[r];
                }
            } else {  // softmax
                float mx = -INFINITY;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (lane + 32 * r < E) mx = fmaxf(mx, zr[r]);
                mx = warp_max(mx);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = lane + 32 * r;
                    g[r] = (i < E) ? __expf(zr[r] - mx) : 0.0f;
                    den += g[r];
                    num += g[r] * wr[r];
                }
            }
            den = warp_sum(den);
            num = warp_sum(num);
            const float inv = 1.0f / den;
            const float A = num * inv;
            tok_sum += (double)A;
            if (dz) {
                const float cs = coef * inv;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = lane + 32 * r;
                    if (i < E) {
                        const float jac = (kGate == 0) ? g[r] * (1.0f - g[r]) : g[r];
                        dz[t * E + i] = cs * jac * (wr[r] - A);
                    }
                }
            }
        }
    }
    if (lane == 0) s_part[warp] = tok_sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int q = 0; q < kLossWarps; ++q) s += s_part[q];
        partials[(int64_t)layer * P + blockIdx.x] = s;
    }
}

// loss[l] = d_scale/(m^2 k) * sum of the partials in block order.
__global__ void __launch_bounds__(256)
loss_finalize_kernel(const double *__restrict__ partials, int P, double scale,
                     float *__restrict__ loss) {
    __shared__ double s_dred[256];
    const int layer = blockIdx.x;
    const double s = block_sum_fixed(partials + (int64_t)layer * P, P, s_dred, 256);
    if (threadIdx.x == 0) loss[layer] = (float)(s * scale);
}

// origin_do += sum_{i != j} D_ij^2 over kOriginRows rows of one problem (Eq.
// origin_do), exact in int64; origin_do zero on entry.  (One CTA for a whole
// problem, with a division per entry, took 23 us at E = 96.)
constexpr int kOriginRows = 8;
__global__ void __launch_bounds__(256)
origin_do_kernel(const int *__restrict__ Dg, int E, long long *__restrict__ origin_do) {
    __shared__ long long s_red[8];
    const int *Dl = Dg + (int64_t)blockIdx.y * E * E;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kOriginRows + warp;  // a row per warp
    long long acc = 0;
    if (i < E)
#pragma unroll 4
        for (int j = lane; j < E; j += 32) {
            const long long d = j == i ? 0 : __ldg(Dl + (int64_t)i * E + j);
            acc += d * d;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
    if (lane == 0) s_red[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long sum = 0;
        for (int q = 0; q < 8; ++q) sum += s_red[q];
        atomicAdd(reinterpret_cast<unsigned long long *>(origin_do + blockIdx.y), (unsigned long long)sum);
    }
}

// CTAs per problem and the split of a word over warps: one wave of the CTAs
// that fit (an SM holds one with a large D in shared memory), every warp with
// as few tokens as that allows.
template <int R>
void loss_generic_grid(const Problem &p, size_t smem, int P_max, int *P, int *split) {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int warps = loss_warps<R>();
    const int by_smem = (int)(220 * 1024 / (smem + 8 * 1024));
    const int occ = by_smem < 1 ? 1 : by_smem > 2 ? 2 : by_smem;
    int64_t ctas = (int64_t)sms * occ / p.L;
    if (ctas < 1) ctas = 1;
    int s = 1;
    while (s < 32 && p.W * s < ctas * warps) s *= 2;
    const int64_t need = (p.W * s + warps - 1) / warps;
    if (ctas > need) ctas = need;
    if (ctas > P_max) ctas = P_max;
    *P = (int)ctas;
    *split = s;
}

struct GenericArgs {
    const float *logits;
    const uint32_t *bits;
    const int *D, *counts;
    float coef;
    float *dlogits;
    double *partials;
    int P_max;
    int *status;
};

template <int R, bool kSmemD, int kGate>
cudaError_t run_loss(const GenericArgs &a, const Problem &p, int *P, cudaStream_t s) {
    const size_t smem = sizeof(int) * ((kSmemD ? (size_t)p.E * p.E : 0) + (size_t)p.E);
    auto kern = loss_generic_kernel<R, kSmemD, kGate>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    int split = 1;
    loss_generic_grid<R>(p, smem, a.P_max, P, &split);
    dim3 grid((unsigned)*P, (unsigned)p.L);
    kern<<<grid, loss_warps<R>() * 32, smem, s>>>(a.logits, a.bits, a.D, a.counts, p.T, p.E, p.k, p.W,
                                                 split, a.coef, a.dlogits, a.partials, *P, a.status);
    return cudaGetLastError();
}

template <int R>
cudaError_t dispatch_gate(const GenericArgs &a, const Problem &p, int gate, int *P, cudaStream_t s) {
    const bool smem_d = sizeof(int) * ((size_t)p.E * p.E + p.E) <= kSmemDLimit;
    if (gate == 0) return smem_d ? run_loss<R, true, 0>(a, p, P, s) : run_loss<R, false, 0>(a, p, P, s);
    return smem_d ? run_loss<R, true, 1>(a, p, P, s) : run_loss<R, false, 1>(a, p, P, s);
}

}  // namespace

int loss_blocks_per_problem(const Problem &p) {
    int64_t blocks = (p.W + 7) / 8;
    int64_t cap = 1024 / p.L;
    if (cap < 1) cap = 1;
    if (blocks > cap) blocks = cap;
    return (int)(blocks < 1 ? 1 : blocks);
}

WsLayout ws_layout(const Problem &p, bool wide) {
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    WsLayout w;
    const int64_t fast_parts = p.W;  // the fast kernel gives every CTA at least 32 tokens
    const int64_t gen_parts = loss_blocks_per_problem(p);
    w.max_parts = (int)(fast_parts > gen_parts ? fast_parts : gen_parts);
    const bool fast_k = p.k == 1 || p.k == 2 || p.k == 4 || p.k == 8;
    const bool fast_e = p.E == 32 || p.E == 64 || p.E == 128;
    w.cooc = (fast_k && fast_e) || (wide && cooc_sizes_ok(p.E, p.k));
    w.image = w.cooc && (wide ? bimg_sizes_ok(p.E, p.k) : p.E == 128);
    w.done = kWsHeader;
    w.partials = up(w.done + sizeof(int) * (size_t)p.L);
    w.idx = up(w.partials + sizeof(double) * (size_t)p.L * (size_t)w.max_parts);
    w.cooc_parts = up(w.idx + (fast_k ? (size_t)p.L * (size_t)p.T * (size_t)p.k : 0));
    const size_t parts = w.cooc ? sizeof(uint32_t) * (size_t)p.L *
                                                  (size_t)max_sig_ctas_per_problem(p) *
                                                  cooc_partial_words(p.E)
                                            : 0;
    w.bimg = up(w.cooc_parts + parts);
    // the dispatch order of a routed call may run beside the loss kernel: its
    // scratch has a region of its own
    w.img_ok = up(w.bimg + (w.image ? (size_t)bimg_bytes(cooc_width(p.E)) * (size_t)p.L : 0));
    w.route_base = up(w.img_ok + (w.image ? sizeof(int) * (size_t)p.L : 0));
    w.total = up(w.route_base + sizeof(int) * (size_t)route_scratch_ints(p));
    return w;
}

int max_sig_ctas_per_problem(const Problem &p) {
    int64_t gx = kMaxSigCtas / p.L;
    if (gx > p.W) gx = p.W;
    return (int)(gx < 1 ? 1 : gx);
}

cudaError_t launch_loss(const float *logits, const uint32_t *bits, const int *D, const Problem &p,
                        int gate, float d_scale, float grad_scale, float *loss,
                        long long *origin_do, float *dlogits, int *status, double *partials,
                        cudaStream_t s, const int *counts) {
    const double norm = 1.0 / ((double)p.T * (double)p.T * (double)p.k);
    const GenericArgs a = {logits, bits, D, counts, (float)((double)grad_scale * (double)d_scale * norm),
                           dlogits, partials, ws_layout(p, false).max_parts, status};
    const int r = (p.E + 31) / 32;
    int P = 1;
    cudaError_t e;
    if (r <= 1) e = dispatch_gate<1>(a, p, gate, &P, s);
    else if (r <= 2) e = dispatch_gate<2>(a, p, gate, &P, s);
    else if (r <= 4) e = dispatch_gate<4>(a, p, gate, &P, s);
    else if (r <= 8) e = dispatch_gate<8>(a, p, gate, &P, s);
    else if (r <= 16) e = dispatch_gate<16>(a, p, gate, &P, s);
    else e = dispatch_gate<32>(a, p, gate, &P, s);
    if (e != cudaSuccess) return e;
    loss_finalize_kernel<<<p.L, 256, 0, s>>>(partials, P, (double)d_scale * norm, loss);
    e = cudaGetLastError();
    if (e == cudaSuccess && origin_do) e = launch_origin_do(D, p, origin_do, s);
    return e;
}

// Variance of the E (E - 1) off-diagonal distances of a local window from
// Eq. origin_do (their sum of squares) and Eq. zero_sum (their sum is
// 2 T k (E - k)): var = origin_do / (E (E - 1)) - mean^2 (App. C.1).  One
// thread per problem, fp64.
__global__ void offdiag_variance_kernel(const long long *__restrict__ origin_do, int64_t T, int E,
                                        int k, int L, double *__restrict__ var) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= L) return;
    const double n = (double)E * (double)(E - 1);
    const double mean = 2.0 * (double)T * (double)k * (double)(E - k) / n;
    var[l] = (double)origin_do[l] / n - mean * mean;
}

cudaError_t launch_offdiag_variance(const long long *origin_do, const Problem &p, double *var,
                                    cudaStream_t s) {
    offdiag_variance_kernel<<<(p.L + 255) / 256, 256, 0, s>>>(origin_do, p.T, p.E, p.k, p.L, var);
    return cudaGetLastError();
}

cudaError_t launch_origin_do(const int *D, const Problem &p, long long *origin_do, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(origin_do, 0, sizeof(long long) * (size_t)p.L, s);
    if (e != cudaSuccess) return e;
    origin_do_kernel<<<dim3((unsigned)((p.E + kOriginRows - 1) / kOriginRows), (unsigned)p.L), 256, 0, s>>>(
        D, p.E, origin_do);
    return cudaGetLastError();
}

}  // namespace dol
