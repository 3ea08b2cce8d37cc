// Launcher of the tensor-core loss kernel (loss_mma.cuh) and its routing-gradient
// instantiations.
#include "loss_mma.cuh"

namespace dol {

template <> cudaError_t run_loss_mma<1>(const CUtensorMap &, const CUtensorMap &, const MmaArgs &, int, bool, bool, bool, int, int, cudaStream_t);
template <> cudaError_t run_loss_mma<2>(const CUtensorMap &, const CUtensorMap &, const MmaArgs &, int, bool, bool, bool, int, int, cudaStream_t);
template <> cudaError_t run_loss_mma<3>(const CUtensorMap &, const CUtensorMap &, const MmaArgs &, int, bool, bool, bool, int, int, cudaStream_t);
template <> cudaError_t run_loss_mma<4>(const CUtensorMap &, const CUtensorMap &, const MmaArgs &, int, bool, bool, bool, int, int, cudaStream_t);

namespace {

int sms_now() {
    int dev = 0, n = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

}  // namespace

// Off-diagonal entries of D (at most T for one window) must stay below 2^22
// for the two fp16 pieces.
bool loss_mma_supported(const Problem &p, const float *logits, const float *dlogits) {
    auto al = [](const void *q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    return bimg_sizes_ok(p.E, p.k) && p.T < (int64_t)(1 << 22) && al(logits) && (!dlogits || al(dlogits));
}

// R_i <= (E - 1) T may reach 2^23: the marker diagonal.
bool loss_mma_big(const Problem &p) { return (int64_t)(p.E - 1) * p.T >= (int64_t)(1 << 23); }

// Where the ALU kernel of loss_fast.cu (E in {32, 64, 128}, k in {1, 2, 4, 8}) is
// the faster one: its gather of k rows a token costs by k T, the tensor-core
// kernel's set-up (TMEM, the operand image, a first MMA) once.  Measured, step
// with the ALU kernel against the tensor cores, us:
//   k T <= 512 E   E = 64,  k = 8, T = 4096:  10.8 / 11.4   (T = 8192: 11.9 / 11.5)
//                  E = 128, k = 8, T = 8192:  15.0 / 15.1   (T = 16384: 18.3 / 16.7)
//                  E = 32,  k = 2, T = 8192:   8.9 /  9.1   (T = 16384: 9.9 / 9.8)
//   k <= E / 64    E = 64,  k = 1, T = 200000: 30.9 / 32.6
//                  E = 128, k = 2, T = 93176:  30.6 / 33.9  (T = 200000: 61.3 / 60.3)
// At E = 128, sigmoid-norm, the tensor cores add the routing gradient as well, so
// the smaller sizes stay with them.
bool loss_alu_faster(const Problem &p, int gate) {
    const bool sizes = (p.E == 32 || p.E == 64 || p.E == 128) && (p.k == 1 || p.k == 2 || p.k == 4 || p.k == 8);
    if (!sizes || (p.E == 128 && gate == 0 && !loss_mma_big(p))) return false;
    const int64_t tokens = p.T * p.L;
    return tokens * p.k <= 512 * (int64_t)p.E || (p.k <= p.E / 64 && (p.E == 64 || tokens <= (1 << 17)));
}

// The routing gradient is added in the epilogue (else by its own kernel).
bool loss_mma_route_grad(const Problem &p, int gate, const int *ids, const float *g) {
    auto al = [](const void *q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    const bool k_ok = p.k == 1 || p.k == 2 || p.k == 4 || p.k == 8;
    return p.E == 128 && gate == 0 && k_ok && al(ids) && al(g);
}

cudaError_t launch_loss_mma(const float *logits, const uint32_t *bits, const uint8_t *idx,
                            const unsigned char *bimg, const Problem &p, int gate, float d_scale, float grad_scale,
                            float *loss, float *dlogits, double *partials, int *done, int *status,
                            int *status_out, cudaStream_t s, const int *rg_ids, const float *rg_g,
                            const int *img_ok, const int *D) {
    if (!bimg || (img_ok && !D) || (rg_ids && (!idx || !loss_mma_route_grad(p, gate, rg_ids, rg_g))))
        return cudaErrorInvalidValue;
    CUtensorMap zmap, dzmap;
    if (!encode_tensor_map_3d_f32(&zmap, logits, (uint64_t)p.L, (uint64_t)p.T, (uint64_t)p.E, 32))
        return cudaErrorInvalidValue;
    if (!dlogits) dzmap = zmap;  // forward only: never stored through
    else if (!encode_tensor_map_3d_f32(&dzmap, dlogits, (uint64_t)p.L, (uint64_t)p.T, (uint64_t)p.E, 32))
        return cudaErrorInvalidValue;
    const int64_t tiles = (p.T + kTileM - 1) / kTileM;
    int64_t gx = sms_now() / p.L;
    if (gx < 1) gx = 1;
    if (gx > tiles) gx = tiles;
    const double norm = 1.0 / ((double)p.T * (double)p.T * (double)p.k);
    MmaArgs args;
    args.bits = bits;
    args.idx = idx;
    args.k = p.k;
    args.bimg = bimg;
    args.T = p.T;
    args.W = p.W;
    args.E = p.E;
    args.has_dz = dlogits != nullptr;
    args.coef = (float)((double)grad_scale * (double)d_scale * norm);
    args.scale = (double)d_scale * norm;
    args.partials = partials;
    args.done = done;
    args.loss = loss;
    args.status = status;
    args.status_out = status_out;
    args.rg_ids = rg_ids;
    args.rg_g = rg_g;
    args.img_ok = img_ok;
    args.D = D;
    args.logits = logits;
    args.dlogits = dlogits;
    // a given matrix has the marker diagonal always
    const bool big = img_ok != nullptr || loss_mma_big(p);
    if (rg_ids && rg_g) {
#define DOL_RG_CASE(KK)                                                                       \
    return big ? run_mma<4, 0, true, false, true, KK>(zmap, dzmap, args, (int)gx, p.L, s)          \
               : run_mma<4, 0, false, false, true, KK>(zmap, dzmap, args, (int)gx, p.L, s)
        switch (p.k) {
            case 1: DOL_RG_CASE(1);
            case 2: DOL_RG_CASE(2);
            case 4: DOL_RG_CASE(4);
            default: DOL_RG_CASE(8);
        }
#undef DOL_RG_CASE
    }
    const bool pad = p.E % 32 != 0;
    switch (cooc_width(p.E) / 32) {
        case 1: return run_loss_mma<1>(zmap, dzmap, args, gate, big, pad, idx != nullptr, (int)gx, p.L, s);
        case 2: return run_loss_mma<2>(zmap, dzmap, args, gate, big, pad, idx != nullptr, (int)gx, p.L, s);
        case 3: return run_loss_mma<3>(zmap, dzmap, args, gate, big, pad, idx != nullptr, (int)gx, p.L, s);
        default: return run_loss_mma<4>(zmap, dzmap, args, gate, big, pad, idx != nullptr, (int)gx, p.L, s);
    }
}

}  // namespace dol
