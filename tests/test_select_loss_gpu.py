"""The selection kernel (topk_net.cuh, select.cuh), the co-occurrence reduction
and the loss kernels (loss_mma.cuh, loss.cu) at the sizes where their tiles,
paddings and splits end, against the CPU oracle.

Signatures, counts, D, origin_do and the routing integers are exact.

Loss and dlogits, per entry.  With p the gate's weights, w = dL/dp (fp64, from
the oracle) and M_t = sum_i p_it |w_it|, the kernels compute
dz_it = p_it (1 - s_it) (w_it - A_t) (softmax: p_it (w_it - A_t)), A_t = sum_i
p_it w_it.  The sums over E columns are fp32 (E u each, u = 2^-24); s comes from
one ex2.approx (2 ulp) of a product rounded at |z| <= 8 (12 u) and one rcp.approx
(1 ulp), so s, the sums and their quotient are within (E + 64) u; the integers
behind w are exact below 2^24 and rounded once above.  So
  |dz - ref| <= 2 (E + 64) u p (1 - s) (|w| + M_t),  |loss - ref| <= 2 (E + 64) u sum_t M_t,
the factor 2 for the two factors of the product (in the gather kernels 1 - s comes
as s - s^2, within u / (1 - s) <= 150 u at z <= 5, inside the same bound).  u p_max max|w| is added for
results rounded near zero.  Where |z| goes beyond 8 the rounded product z log2 e and
the rounded log2 e put up to 1.25 |z| u more into each s, and so on into every sum:
E + 64 + 1.25 (|z| - 8) in the place of E + 64.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_32398_gb300 import workloads
from test_routed_split_gpu import route_bound

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module")
def dl():
    import paper_2609_32398_gb300.doloss as m

    m.lib()
    return m


def check_loss(z, f, D, k, gate, loss, dz, d_scale=1.0, extra=0.0, extra_bound=0.0, zmax=8.0,
               near_zero=True):
    T, E = z.shape
    p = oracle.gate(z, gate)
    w = oracle.dloss_dp(D, f, T, k, d_scale)
    M = (p * np.abs(w)).sum(1, keepdims=True)
    ref = oracle.loss(D, oracle.direction(z, f, gate), T, k, d_scale)
    tol = 2.0 * (E + 64 + 1.25 * max(0.0, zmax - 8.0)) * U
    assert abs(loss - ref) <= tol * M.sum() + U * abs(ref), ("loss", loss, ref)
    if dz is None:
        return
    oms = 1.0 if gate == workloads.GATE_SOFTMAX else 1.0 / (1.0 + np.exp(z.astype(np.float64)))
    bound = tol * p * oms * (np.abs(w) + M) + near_zero * U * p.max() * np.abs(w).max()
    err = np.abs(dz.double().cpu().numpy() - oracle.gate_backward(z, w, gate) - extra)
    bound = bound + extra_bound
    assert (err <= bound).all(), ("dlogits", float((err / bound).max()))


# four experts, a width that is no multiple of 32, every number of 32-expert
# boxes, lists of 4, 8 and 16, one token, ragged and whole tiles, ties
@pytest.mark.parametrize("T,E,k,L,ties", [
    (1, 4, 1, 1, False), (33, 4, 4, 3, True), (31, 12, 3, 1, True), (257, 36, 9, 2, True),
    (500, 64, 5, 1, False), (1000, 96, 6, 2, True), (97, 100, 16, 1, True), (64, 128, 16, 1, True),
    (129, 160, 2, 1, True), (700, 200, 7, 1, False), (4801, 256, 8, 1, True), (333, 256, 16, 2, True),
    (65, 384, 12, 1, True), (2049, 512, 10, 1, True), (32, 512, 16, 2, False)])
def test_selection(dl, T, E, k, L, ties):
    z = workloads.random_logits(T, E, L=L, seed=31 * T + E + k, ties=ties)
    z[0, 0, : min(E, k + 1)] = -torch.inf            # ties of the lowest value
    if E >= 8:
        z[L - 1, T - 1, E // 2:] = torch.finfo(torch.float32).min
    zc = z.cuda()
    bits, counts = dl.signatures(zc, k)
    finite = z.clone()
    finite[0, 0] = torch.arange(E, dtype=torch.float32) % 3    # its combine weights are defined
    r = dl.routing(finite.cuda(), k, workloads.GATE_SOFTMAX)
    assert dl.device_status(r.workspace) == 0
    for l in range(L):
        f = oracle.select(z[l].numpy(), k)
        assert np.array_equal(bits[l].cpu().numpy().view(np.uint32), oracle.pack(f))
        assert np.array_equal(counts[l].cpu().numpy(), oracle.counts(f))
        ids, comb = oracle.route(finite[l].numpy(), k, workloads.GATE_SOFTMAX)
        assert np.array_equal(r.expert_ids[l].cpu().numpy(), ids)
        # k terms summed, exponentials of 2 ulp: (k + 12) u, doubled
        assert np.abs(r.combine[l].double().cpu().numpy() - comb).max() <= 2 * (k + 12) * U
        offsets, rows, pos = oracle.dispatch(ids, E)
        assert np.array_equal(r.offsets[l].cpu().numpy(), offsets)
        assert np.array_equal(r.rows[l].cpu().numpy(), rows)
        assert np.array_equal(r.pos[l].cpu().numpy(), pos)


# both sides of the line between the gather and the tensor-core kernel (k T L =
# 512 E; E = 128: two choices at the marker's sizes);
# one to four boxes of the tensor-core kernel, padded and whole; tiles of 128
# tokens and their remainders; both gates; the marker diagonal ((E - 1) T >=
# 2^23); counted widths above 128 and the generic kernel (k > 64, E > 256)
@pytest.mark.parametrize("T,E,k,L,gate", [
    (1, 4, 1, 1, 0), (127, 12, 3, 2, 1), (129, 32, 16, 1, 0), (1300, 36, 4, 1, 1), (128, 64, 5, 3, 0),
    (641, 68, 7, 1, 0), (255, 96, 6, 2, 1), (20011, 100, 8, 1, 0), (385, 128, 10, 2, 1),
    (2000, 128, 3, 1, 0), (66053, 128, 5, 1, 0), (84737, 100, 8, 1, 1),
    (4096, 64, 8, 1, 0), (4097, 64, 8, 1, 1), (16384, 32, 1, 1, 1), (16385, 32, 1, 1, 0),
    (2049, 128, 4, 2, 1), (66053, 128, 2, 1, 0),
    (300, 132, 8, 1, 0), (777, 160, 16, 2, 1), (1000, 252, 3, 1, 0),
    (130, 100, 70, 2, 1), (99, 300, 5, 1, 0), (4099, 320, 9, 2, 1), (33, 1000, 12, 1, 0)])
def test_step(dl, T, E, k, L, gate):
    z = workloads.random_logits(T, E, L=L, seed=T + 7 * E + k)
    zc = z.cuda()
    out = dl.forward_backward(zc, k, gate)
    fwd = dl.forward_backward(zc, k, gate, with_grad=False)
    again = dl.forward_backward(zc, k, gate, out=dl.Buffers(L, T, E, k))
    torch.cuda.synchronize()
    assert dl.device_status(out.workspace) == 0 and dl.device_status(fwd.workspace) == 0
    assert torch.equal(out.dlogits, again.dlogits) and torch.equal(out.loss, again.loss)
    for l in range(L):
        zl = z[l].numpy()
        f = oracle.select(zl, k)
        D = oracle.hamming(f)
        for o in (out, fwd):
            assert np.array_equal(o.bits[l].cpu().numpy().view(np.uint32), oracle.pack(f))
            assert np.array_equal(o.counts[l].cpu().numpy(), oracle.counts(f))
            assert np.array_equal(o.D[l].cpu().numpy(), D)
            assert int(o.origin_do[l]) == oracle.origin_do(D)
        check_loss(zl, f, D, k, gate, float(out.loss[l]), out.dlogits[l])
        check_loss(zl, f, D, k, gate, float(fwd.loss[l]), None)


# the sigmoid gate on rows of low logits: p = s / sum of s is relative to the row,
# so that every s keeps its relative accuracy; both sides of T = 66052 (the marker
# diagonal), one to four boxes, the fused call and the given matrix
@pytest.mark.parametrize("T,E,k,shift", [
    (515, 32, 3, -60.0), (515, 64, 5, -30.0), (515, 96, 6, -12.0), (515, 96, 6, -20.0), (515, 100, 8, -30.0),
    (515, 124, 4, -60.0), (515, 128, 8, -18.0), (4100, 128, 8, -30.0), (515, 128, 3, -60.0),
    (66053, 96, 6, -20.0), (66053, 128, 8, -30.0)])
def test_low_logits(dl, T, E, k, shift):
    z = workloads.random_logits(T, E, seed=T + E + k) + shift
    z[0, : T // 2, :: 5] += -shift                   # rows that mix low logits with ordinary ones
    zc = z.cuda()
    out = dl.forward_backward(zc, k)
    loss, _, dz = dl.loss_fwd_bwd(zc, out.bits, out.D, k)
    torch.cuda.synchronize()
    assert dl.device_status(out.workspace) == 0
    f = oracle.select(z[0].numpy(), k)
    D = oracle.hamming(f)
    zmax = float(z.abs().max())
    check_loss(z[0].numpy(), f, D, k, 0, float(out.loss[0]), out.dlogits[0], zmax=zmax)
    check_loss(z[0].numpy(), f, D, k, 0, float(loss[0]), dz[0], zmax=zmax)


# saturated experts: 1 - s keeps its relative accuracy where s is one to rounding, at
# every number of boxes (the bound without its term for results near zero)
@pytest.mark.parametrize("T,E,k", [(515, 32, 3), (515, 64, 5), (5000, 64, 8), (515, 96, 6), (515, 128, 8)])
def test_saturated_experts(dl, T, E, k):
    z = workloads.random_logits(T, E, seed=T + E)
    z[0, :, : E // 2] += 20.0
    out = dl.forward_backward(z.cuda(), k)
    torch.cuda.synchronize()
    assert dl.device_status(out.workspace) == 0
    f = oracle.select(z[0].numpy(), k)
    check_loss(z[0].numpy(), f, oracle.hamming(f), k, 0, float(out.loss[0]), out.dlogits[0],
               zmax=float(z.abs().max()), near_zero=False)


# the softmax gate far from zero: rows of the lowest value (uniform weights), rows and
# whole boxes of masks of several sizes, large rows of either sign, ordinary rows
# beside them; one to four boxes and the gather kernels
@pytest.mark.parametrize("T,E,k", [(300, 24, 3), (300, 64, 5), (2300, 64, 8), (515, 96, 6), (515, 100, 8), (4100, 128, 8),
                                   (300, 32, 4), (300, 200, 5), (300, 256, 8)])
def test_softmax_far_from_zero(dl, T, E, k):
    low = torch.finfo(torch.float32).min
    z = workloads.random_logits(T, E, seed=T + E)
    z[0, 1] = low
    z[0, 2] = -1e9
    z[0, 3, : E // 2] = 1e9
    z[0, 4, E // 2:] = -1e10
    z[0, 5, : E // 2] = -1e29
    z[0, 6] += 2.9e6                                  # around the line where the form changes
    z[0, 7] -= 4.3e6
    z[0, 8, E // 2:] = low
    z[0, 9, :] = low
    z[0, 9, E - 1] = 0.0
    z[0, 10] *= 1e12
    z[0, 11, : E // 2] += 4194304.0
    z[0, 12, E // 2:] -= 4194304.0
    z[0, T - 1, 1:] = -3e38
    zc = z.cuda()
    out = dl.forward_backward(zc, k, workloads.GATE_SOFTMAX)
    loss, _, dz = dl.loss_fwd_bwd(zc, out.bits, out.D, k, workloads.GATE_SOFTMAX)
    torch.cuda.synchronize()
    assert dl.device_status(out.workspace) == 0
    zl = z[0].numpy()
    f = oracle.select(zl, k)
    D = oracle.hamming(f)
    # logits that weigh anything are within 8 of their row's maximum, or at least 0.25
    # apart and exact there: the arguments of the exponentials are as in the note above
    check_loss(zl, f, D, k, workloads.GATE_SOFTMAX, float(out.loss[0]), out.dlogits[0])
    check_loss(zl, f, D, k, workloads.GATE_SOFTMAX, float(loss[0]), dz[0])


# one zeroed workspace for two shapes in turn, both orders, each also twice running:
# nothing that a call leaves in it may reach the next one
@pytest.mark.parametrize("one,two", [
    ((1, 40000, 256, 8), (1, 1000, 256, 8)), ((1, 30000, 96, 6), (3, 700, 96, 6)),
    ((1, 65536, 128, 8), (1, 9000, 64, 8)), ((2, 9000, 160, 3), (1, 500, 8, 2)), ((4, 3000, 32, 2), (1, 20000, 128, 5))])
def test_workspace_of_two_shapes(dl, one, two):
    n = max(int(dl.lib().do_routed_workspace_size(T, E, k, L)) for L, T, E, k in (one, two))
    ws = torch.zeros(n, dtype=torch.uint8, device="cuda")

    def run(shape, z, routed, ws=None):
        out = dl.Buffers(*shape)
        if ws is not None:
            out.workspace = ws
        if not routed:
            return dl.forward_backward(z, shape[3], out=out)
        dl.routed_forward(z, shape[3], out=out)
        return dl.routed_backward(z, None, None, shape[3], out=out)

    z = {s: workloads.random_logits(s[1], s[2], L=s[0], seed=s[2] + s[3]).cuda() for s in (one, two)}
    want = {(s, r): run(s, z[s], r) for s in (one, two) for r in (False, True)}
    for shape in (one, two, two, one, one):
        for routed in (False, True):
            out = run(shape, z[shape], routed, ws)
            for name in ("counts", "D", "origin_do", "loss", "dlogits"):
                assert torch.equal(getattr(out, name), getattr(want[shape, routed], name)), (shape, routed, name)
    assert dl.device_status(ws) == 0


# a given matrix: its image (the first problem), and one that no image holds (an
# entry of 2^22, or a non-zero diagonal), gathered from D in the same launch.  A
# non-zero diagonal, which no matrix of distances has, only at sizes of the
# tensor-core kernel: the ALU kernel's column sums R take it in.
@pytest.mark.parametrize("T,E,k,gate,fault", [
    (200, 36, 5, 0, "large"), (515, 128, 5, 1, "diagonal"), (260, 96, 3, 0, "diagonal"),
    (129, 64, 8, 1, "large")])
def test_given_matrix(dl, T, E, k, gate, fault):
    z = workloads.random_logits(T, E, L=2, seed=T + E)
    f = [oracle.select(z[l].numpy(), k) for l in range(2)]
    D = np.stack([3 * oracle.hamming(x) for x in f])
    if fault == "large":
        D[1, 1, 3] = D[1, 3, 1] = 1 << 22
    else:
        D[1, 2, 2] = 5
    bits = torch.from_numpy(np.stack([oracle.pack(x) for x in f]).view(np.int32)).cuda()
    loss, origin, dz = dl.loss_fwd_bwd(z.cuda(), bits, torch.from_numpy(D).cuda(), k, gate, d_scale=0.5)
    for l in range(2):
        off = D[l].astype(np.int64) ** 2
        assert int(origin[l]) == int(off.sum() - np.trace(off))
        check_loss(z[l].numpy(), f[l], D[l], k, gate, float(loss[l]), dz[l], d_scale=0.5)


# the routing gradient: the choices of a token split over four warps (k = 2: two
# of them idle), with the marker diagonal and without
@pytest.mark.parametrize("T,k", [(1, 8), (129, 2), (500, 4), (66053, 8)])
def test_routing_gradient(dl, T, k):
    E = 128
    z = workloads.random_logits(T, E, seed=T + k)
    g = 1e-3 * torch.randn(1, T, k, generator=torch.Generator().manual_seed(T))
    out, r = dl.routed_forward(z.cuda(), k)
    dl.routed_backward(z.cuda(), r.expert_ids, g.cuda(), k, out=out)
    torch.cuda.synchronize()
    assert dl.device_status(out.workspace) == 0
    zl, gl = z[0].numpy(), g[0].numpy()
    f = oracle.select(zl, k)
    ids, _ = oracle.route(zl, k)
    check_loss(zl, f, oracle.hamming(f), k, 0, float(out.loss[0]), out.dlogits[0],
               extra=oracle.route_backward(zl, ids, gl), extra_bound=route_bound(zl, ids, gl, 0))


# E = 256: 13-bit and (from T = 2^21 on) 16-bit fields of D in shared memory,
# against the general kernels, which take logits that are not 16-byte aligned.
# Both sides are within the bound above; an entry of dz is at most p_max (|w| + M).
@pytest.mark.parametrize("T,k,gate", [(1, 8, 0), (4097, 8, 1), (70001, 4, 0), (1 << 21, 8, 0)])
def test_planes_against_general_path(dl, T, k, gate):
    E = 256
    z = workloads.random_logits(T, E, seed=T, device="cuda")
    z[:, :, :4] += 6.0                               # crowded experts: large counts
    shifted = torch.empty(T * E + 1, device="cuda")[1:].view(1, T, E)
    shifted.copy_(z)
    a, b = dl.forward_backward(z, k, gate), dl.forward_backward(shifted, k, gate)
    torch.cuda.synchronize()
    assert dl.device_status(a.workspace) == 0 and dl.device_status(b.workspace) == 0
    assert torch.equal(a.bits, b.bits) and torch.equal(a.D, b.D) and torch.equal(a.counts, b.counts)
    tol = 4.0 * (E + 64) * U
    assert float(a.loss) == pytest.approx(float(b.loss), rel=tol, abs=tol)
    assert (a.dlogits - b.dlogits).abs().max() <= 2 * tol * b.dlogits.abs().max()


# the narrow workspace layout: E = 256 in the library's fixed 16 MiB array where
# the layout with counts does not fit any more
@pytest.mark.parametrize("T", [1 << 16, 500000])
def test_static_scratch_narrow_layout(dl, T):
    E, k = 256, 8
    z = workloads.random_logits(T, E, seed=T, device="cuda")
    out, ref = dl.Buffers(1, T, E, k), dl.Buffers(1, T, E, k)
    dl.forward_backward_static(z, k, out)
    dl.forward_backward(z, k, out=ref)
    torch.cuda.synchronize()
    for a, b in ((out.bits, ref.bits), (out.counts, ref.counts), (out.D, ref.D), (out.origin_do, ref.origin_do)):
        assert torch.equal(a, b)
    assert float(out.loss) == pytest.approx(float(ref.loss), rel=1e-5)
    assert (out.dlogits - ref.dlogits).abs().max() <= 1e-4 * ref.dlogits.abs().max()
