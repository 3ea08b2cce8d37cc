// Step 1, fast path: the launchers of the Top-K signature kernel (the kernel
// itself is in sig_fast.cuh) without routing outputs.
#include "sig_fast.cuh"

namespace dol {
// The sizes at which this kernel is the faster one: argmax rounds with the pairs
// counted in shared memory, 10.3 us of the E = 128, k = 8, T = 65536 step
// against 12.7 us of select.cuh's networks and tensor-core counts (28 against
// 38 us at T = 262144).
bool signatures_fast_supported(const float *logits, const Problem &p) {
    const bool e_ok = p.E == 32 || p.E == 64 || p.E == 128;
    const bool k_ok = p.k == 1 || p.k == 2 || p.k == 4 || p.k == 8;
    return e_ok && k_ok && (reinterpret_cast<uintptr_t>(logits) % 16 == 0) &&
           (int64_t)p.L * p.T + 32 < (int64_t)INT_MAX;
}

cudaError_t launch_signatures_fast(const float *logits, const Problem &p, uint32_t *bits,
                                   int *counts, uint8_t *idx, uint32_t *cooc, const ZeroSpans &zero,
                                   int *status, cudaStream_t s) {
    CUtensorMap map;
    if (!encode_tensor_map_2d_f32(&map, logits, (uint64_t)p.L * p.T, (uint64_t)p.E, 32))
        return cudaErrorInvalidValue;
    const RouteOut none = {nullptr, nullptr, 0};
    if (p.E == 32) return dispatch_mode<32, false>(map, p, bits, counts, idx, cooc, zero, status, none, s);
    if (p.E == 64) return dispatch_mode<64, false>(map, p, bits, counts, idx, cooc, zero, status, none, s);
    return dispatch_mode<128, false>(map, p, bits, counts, idx, cooc, zero, status, none, s);
}

}  // namespace dol
