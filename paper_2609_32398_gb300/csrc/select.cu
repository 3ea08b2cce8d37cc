// Step 1: the launcher of the selection kernel (select.cuh).
#include "select.cuh"

namespace dol {
namespace {

int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 148;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 148;
    return n;
}

template <int KP, bool kCooc>
cudaError_t run_select(const CUtensorMap &map, const Problem &p, const SelArgs &args, int ctas,
                       cudaStream_t s) {
    cudaError_t e = ensure_smem_limit<select_kernel<KP, kCooc>>(kSelMaxSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas, (unsigned)p.L);
    cfg.blockDim = dim3((unsigned)(args.lay.consumers + 2) * 32);
    cfg.dynamicSmemBytes = args.lay.total;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, select_kernel<KP, kCooc>, map, args);
}

template <bool kCooc>
cudaError_t dispatch_select(const CUtensorMap &map, const Problem &p, const SelArgs &args, int ctas,
                            cudaStream_t s) {
    if (p.k <= 4) return run_select<4, kCooc>(map, p, args, ctas, s);
    if (p.k <= 8) return run_select<8, kCooc>(map, p, args, ctas, s);
    return run_select<16, kCooc>(map, p, args, ctas, s);
}

bool takes_sig_fast(const float *logits, const Problem &p, const RouteOut &route) {
    const uintptr_t al = reinterpret_cast<uintptr_t>(route.ids) | reinterpret_cast<uintptr_t>(route.combine);
    return signatures_fast_supported(logits, p) && (!route.ids || al % 16 == 0);
}

}  // namespace

// One CTA per SM over all problems, at most one per tile.
int sig_ctas_per_problem(const Problem &p) {
    int sms = sm_count();
    if (sms > kMaxSigCtas) sms = kMaxSigCtas;
    int64_t gx = sms / p.L;
    if (gx > p.W) gx = p.W;
    if (gx < 1) gx = 1;
    return (int)gx;
}

// E <= 512: at least three 32-token tiles fit in shared memory (E = 512 takes
// 64 KB each); above that and for k > 16 (register lists), E not a multiple of
// 4 and unaligned rows (TMA) the generic kernel is the one that runs.
bool select_supported(const float *logits, const Problem &p) {
    return p.E % 4 == 0 && p.E <= 512 && p.k <= 16 && reinterpret_cast<uintptr_t>(logits) % 16 == 0 &&
           (int64_t)p.L * p.T + 32 < (int64_t)INT_MAX;
}

bool cooc_counts_exact(int64_t W, int ctas) { return 32 * ((W + ctas - 1) / ctas) <= (int64_t)1 << 24; }

bool select_cooc_supported(const float *logits, const Problem &p, const RouteOut &route) {
    return select_supported(logits, p) && cooc_sizes_ok(p.E, p.k) &&
           (takes_sig_fast(logits, p, route) || cooc_counts_exact(p.W, sig_ctas_per_problem(p)));
}

cudaError_t launch_select(const float *logits, const Problem &p, const SelectOut &o, cudaStream_t s) {
    if (takes_sig_fast(logits, p, o.route))
        return o.route.ids ? launch_signatures_fast_routed(logits, p, o.bits, o.counts, o.idx, o.cooc, o.zero,
                                                           o.status, o.route, s)
                           : launch_signatures_fast(logits, p, o.bits, o.counts, o.idx, o.cooc, o.zero, o.status, s);
    CUtensorMap map;
    if (!select_supported(logits, p) || (o.cooc && !select_cooc_supported(logits, p, o.route)) || (o.idx && p.E > 256))
        return cudaErrorInvalidValue;
    // one copy per tile where the boxes of a row are whole and many (E = 256,
    // T = 2^20, 4 problems: the step 3,893 -> 3,808 us; at E = 128 a copy per
    // box was 0.9 us faster at T = 65536); else one per box, with zeros past E
    const bool whole = p.E % 32 == 0 && p.E > 128;
    if (whole ? !encode_tensor_map_boxes_f32(&map, logits, (uint64_t)p.L * p.T, (uint64_t)p.E, 32)
              : !encode_tensor_map_2d_f32(&map, logits, (uint64_t)p.L * p.T, (uint64_t)p.E, 32))
        return cudaErrorInvalidValue;
    const int ctas = sig_ctas_per_problem(p);
    SelArgs args;
    args.T = p.T;
    args.W = p.W;
    args.E = p.E;
    args.k = p.k;
    args.whole = whole;
    args.lay = sel_layout(p.E, p.k <= 4 ? 4 : p.k <= 8 ? 8 : 16, (p.W + ctas - 1) / ctas);
    args.bits = o.bits;
    args.counts = o.counts;
    args.cooc = o.cooc;
    args.zero = o.zero;
    args.status = o.status;
    args.idx = o.idx;
    args.route = o.route;
    return o.cooc ? dispatch_select<true>(map, p, args, ctas, s)
                  : dispatch_select<false>(map, p, args, ctas, s);
}

}  // namespace dol
