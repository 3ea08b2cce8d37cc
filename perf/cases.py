"""The measured workloads of the DO-loss library, through its Python entry points.

Each case is one call, or one training step's calls, that a user's program
makes: the loss step on router logits (`forward_backward`, or `do_loss` under
autograd), the router's dispatch (`routing`), the routed training step in its
two halves, the router's linear map with its backward, and the three split
calls.  The sizes are those of the library's workloads (tiny, c2, c3,
collapse, long) and generic ones around them: expert counts and k off the
powers of two, ragged token counts, both gates, one or several layers.
"""
from __future__ import annotations

import math
from dataclasses import replace

import torch

from paper_2609_32398_gb300 import doloss as dl
from paper_2609_32398_gb300 import workloads

SIGMOID, SOFTMAX = dl.GATE_SIGMOID_NORM, dl.GATE_SOFTMAX
LOSS_WEIGHT = 1e-2


def _case(name, kind, recipe, E, k, T, L=1, gate=SIGMOID, H=0):
    c = {"kind": kind, "recipe": recipe, "E": E, "k": k, "T": T, "L": L, "gate": gate}
    if H:
        c["H"] = H
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest step: a toy router, softmax gate; launches and host time are all of it
        _case("tiny_step", "step", "tiny", 8, 2, 1024, gate=SOFTMAX),
        # one micro-batch (4 x 4096 tokens) of a 64-expert layer
        _case("c2_step", "step", "c2", 64, 8, 16384),
        # one micro-batch (16 x 4096 tokens) of a 128-expert layer: the library's headline step
        _case("c3_step", "step", "c3", 128, 8, 65536),
        # a collapsing router over a long window, with exact ties in 5% of the rows
        _case("collapse_step", "step", "collapse", 128, 8, 262144),
        # a long signature window for several 256-expert layers in one call (the largest)
        _case("long_step", "step", "long", 256, 8, 1 << 20, L=4),
        # an expert count and k that are no powers of two, a ragged token count
        _case("odd_step", "step", "plain", 96, 6, 20011),
        # the loss term in a training loop with a softmax router, through autograd; ragged
        _case("softmax_autograd", "autograd", "plain", 128, 8, 30001, gate=SOFTMAX),
        # a routed layer's training step: routing forward, then loss and both gradients
        _case("routed_train", "routed", "c3", 128, 8, 65536),
        # the dispatch of one decode batch: latency
        _case("decode_route", "routing", "plain", 128, 8, 64),
        # the dispatch of a prefill batch, 256 experts, softmax router
        _case("prefill_route", "routing", "plain", 256, 8, 32768, gate=SOFTMAX),
        # the router's linear map, the loss step on its logits and its backward to W and X
        _case("router_train", "router", "hidden", 128, 8, 32768, H=2048),
        # the three calls of the split interface on four layers at once
        _case("split_layers", "split", "plain", 64, 8, 16384, L=4),
    ]


EXPERTS = (8, 16, 24, 32, 48, 60, 64, 72, 96, 100, 128, 128, 160, 192, 200, 256, 256, 320, 384, 512)


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "autograd", "routed", "routing", "routing", "split", "router"))
    gate = rng.choice((SIGMOID, SIGMOID, SOFTMAX))
    recipe = rng.choice(("plain", "plain", "collapse"))
    if kind == "router":  # the router calls take 128 experts and k a power of two
        return _case("", kind, "hidden", 128, rng.choice((1, 2, 4, 8, 8)), _log_uniform(rng, 512, 65536),
                     gate=gate, H=64 * rng.randint(4, 48))
    E = rng.choice(EXPERTS)
    k = rng.choice([q for q in (1, 2, 3, 4, 5, 6, 8, 8, 8, 10) if 4 * q <= E])
    L = rng.choice((1, 1, 1, 2, 4, 7))
    lo = 1 if kind == "routing" else 128
    hi = max(lo + 1, min(1 << 18, (1 << 25) // (E * L)))
    return _case("", kind, recipe, E, k, _log_uniform(rng, lo, hi), L=L, gate=gate)


# ------------------------------------------------------------------ inputs

def _logits(case, seed):
    L, T, E = case["L"], case["T"], case["E"]
    if case["recipe"] in ("tiny", "c2", "c3", "collapse", "long"):
        w = workloads.get(case["recipe"], T=T, L=L)
        w = replace(w, E=E, seed=w.seed + 100003 * (seed + 1))
        if case["recipe"] == "collapse" and E < 64:  # the recipe biases 48 experts
            w = replace(w, name="long")
        return workloads.logits(w, device="cuda")
    # plain: N(0,1) scores with a bias of its own for each expert
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    z = torch.randn(L, T, E, generator=g, device="cuda")
    z += 0.3 * torch.randn(L, 1, E, generator=g, device="cuda")
    return z


def prepare(case, seed):
    L, T, E, k = case["L"], case["T"], case["E"], case["k"]
    s = {"case": dict(case)}
    if case["kind"] == "router":
        s["X"], s["W"] = workloads.router_inputs(T, case["H"], E, L, seed=seed + 11, device="cuda")
        s["out"] = dl.Buffers(L, T, E, k)
        s["logits"] = torch.empty(L, T, E, device="cuda")
        s["ws"] = torch.zeros(int(dl.lib().do_router_backward_workspace_size(T, E, case["H"], L)),
                              dtype=torch.uint8, device="cuda")
        return s
    z = _logits(case, seed)
    s["z"] = z
    if case["kind"] == "autograd":
        s["z"] = z.requires_grad_(True)
    elif case["kind"] == "routing":
        s["route"] = dl.Routing(L, T, E, k)
    elif case["kind"] == "split":
        s["bits"] = torch.empty(L, E, dl.words(T), dtype=torch.int32, device="cuda")
        s["counts"] = torch.empty(L, E, dtype=torch.int32, device="cuda")
        s["D"] = torch.empty(L, E, E, dtype=torch.int32, device="cuda")
        s["dz"] = torch.empty_like(z)
        s["ws"] = dl.new_workspace(T, E, k, L)
    else:
        s["out"] = dl.Buffers(L, T, E, k)
        if case["kind"] == "routed":
            s["route"] = dl.Routing(L, T, E, k)
            s["g"] = _combine_grad(case, seed)
    return s


def _combine_grad(case, seed):
    """The gradient that comes back for the combine weights, the size of the loss's own."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 31 + 5)
    return torch.randn(case["L"], case["T"], case["k"], generator=g, device="cuda") / case["T"]


def _step_outputs(out):
    return {"bits": out.bits, "counts": out.counts, "D": out.D, "loss": out.loss,
            "origin_do": out.origin_do, "dlogits": out.dlogits}


def _route_outputs(r):
    return {"ids": r.expert_ids, "combine": r.combine, "offsets": r.offsets, "rows": r.rows, "pos": r.pos}


def run(state):
    c = state["case"]
    k, gate, kind = c["k"], c["gate"], c["kind"]
    if kind == "step":
        return _step_outputs(dl.forward_backward(state["z"], k, gate, out=state["out"]))
    if kind == "autograd":
        loss = dl.do_loss(state["z"], k, gate)
        (dz,) = torch.autograd.grad((LOSS_WEIGHT * loss).sum(), state["z"])
        return {"loss": loss, "dlogits": dz}
    if kind == "routing":
        r = dl.routing(state["z"], k, gate, out=state["route"])
        return dict(_route_outputs(r), counts=r.counts)
    if kind == "routed":
        out, r = dl.routed_forward(state["z"], k, gate, out=state["out"], route=state["route"])
        dl.routed_backward(state["z"], r.expert_ids, state["g"], k, gate, out=out)
        return dict(_step_outputs(out), **_route_outputs(r))
    if kind == "split":
        bits, counts = dl.signatures(state["z"], k, state["bits"], state["counts"])
        D = dl.pairwise_hamming(bits, c["T"], state["D"])
        loss, origin, dz = dl.loss_fwd_bwd(state["z"], bits, D, k, gate, workspace=state["ws"],
                                           dlogits=state["dz"])
        return {"bits": bits, "counts": counts, "D": D, "loss": loss, "origin_do": origin, "dlogits": dz}
    logits, out = dl.router_forward_backward(state["X"], state["W"], k, gate, out=state["out"],
                                             logits=state["logits"])
    dW, dX = dl.router_backward(state["X"], state["W"], out.dlogits, workspace=state["ws"])
    return dict(_step_outputs(out), logits=logits, dW=dW, dX=dX)


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    L, T, E, k, kind = case["L"], case["T"], case["E"], case["k"], case["kind"]
    n = L * T * E
    logits, bits, D = 4 * n, L * E * ((T + 31) // 32) * 4, 4 * L * E * E
    route = L * (8 * T * k + 8 * T * k + 4 * (E + 1))  # ids and weights, rows and positions, offsets
    # one pass of the gate, the weights' k-row sums, the loss and its gradient: about 20 operations an
    # element besides the k additions; the selection at least a comparison an element
    step_flops = (20 + k + 1) * n
    small = L * (4 * E + 12)
    if kind == "step":
        return {"bytes": 2 * logits + bits + D + small, "flops": step_flops}
    if kind == "autograd":
        return {"bytes": 2 * logits + small, "flops": step_flops}
    if kind == "routing":
        return {"bytes": logits + route + 4 * L * E, "flops": n + 10 * L * T * k}
    if kind == "routed":
        return {"bytes": 2 * logits + bits + D + small + route + 4 * L * T * k,
                "flops": step_flops + 20 * L * T * k}
    if kind == "split":  # the bits and D are one call's outputs and the next one's inputs: written once
        return {"bytes": 2 * logits + bits + D + small, "flops": step_flops}
    H = case["H"]
    X, W = 2 * L * T * H, 2 * L * E * H
    return {"bytes": 2 * X + W + 2 * W + 2 * logits + bits + D + small,
            "flops": step_flops + 6 * L * T * H * E}


def tolerance(case):
    if case["kind"] == "router":
        # bf16 dX, and dz rounded to bf16 for both products; another order of the logits' fp32 sums
        # moves a handful of near-ties between experts, and with them a few entries of D
        return {"rel": 1e-2, "max": 0.9, "differ": 1e-2}
    # fp32 gate, weights and sums; whole numbers stay the same
    return {"rel": 2e-6, "max": 1e-4}


# ------------------------------------------------------------------ the same in 64 bits

def _select(z, k):
    """The k largest of each row of z [T,E], largest first, equal values lower index first."""
    return torch.sort(z, dim=1, descending=True, stable=True).indices[:, :k].contiguous()


def _gate(z, gate):
    return torch.softmax(z, dim=1) if gate == SOFTMAX else torch.sigmoid(z)


def _layer(z, k, gate):
    """One problem [T,E] in fp64: the step's outputs and the selection."""
    T, E = z.shape
    chunk = 1 << 16
    ids = torch.cat([_select(z[a:a + chunk], k) for a in range(0, T, chunk)])
    D = torch.zeros(E, E, dtype=torch.float64, device=z.device)
    counts = torch.zeros(E, dtype=torch.float64, device=z.device)
    bits = torch.zeros(E, (T + 31) // 32, dtype=torch.int32, device=z.device)
    place = torch.arange(32, device=z.device)
    for a in range(0, T, chunk):
        i = ids[a:a + chunk]
        F = torch.zeros(i.shape[0], E, dtype=torch.float64, device=z.device).scatter_(1, i, 1.0)
        D += F.T @ F
        counts += F.sum(0)
        pad = (-F.shape[0]) % 32
        B = torch.cat([F, F.new_zeros(pad, E)]).to(torch.int64).view(-1, 32, E)
        word = (B << place[None, :, None]).sum(1)
        word = torch.where(word >= 1 << 31, word - (1 << 32), word)
        bits[:, a // 32:a // 32 + word.shape[0]] = word.to(torch.int32).T
    D = counts[:, None] + counts[None, :] - 2 * D
    R = D.sum(1)
    scale = 1.0 / (float(T) * float(T) * k)
    dz = torch.empty(T, E, dtype=torch.float64, device=z.device)
    total = torch.zeros((), dtype=torch.float64, device=z.device)
    for a in range(0, T, chunk):
        i, zc = ids[a:a + chunk], z[a:a + chunk].double()
        F = torch.zeros(i.shape[0], E, dtype=torch.float64, device=z.device).scatter_(1, i, 1.0)
        w = F * R - F @ D
        s = _gate(zc, gate)
        S = s.sum(1, keepdim=True)
        p = s / S
        A = (p * w).sum(1, keepdim=True)
        total += A.sum()
        jac = p if gate == SOFTMAX else p * torch.sigmoid(-zc)
        dz[a:a + chunk] = scale * jac * (w - A)
    origin = (D * D).sum()  # below 2^53 times a few: exact enough for a diagnostic
    return {"bits": bits, "counts": counts.to(torch.int32), "D": D.to(torch.int32),
            "loss": (total * scale), "origin_do": origin.to(torch.int64), "dlogits": dz}, ids


def _combine(z, ids, gate):
    v = z.double().gather(1, ids)
    if gate == SOFTMAX:
        return torch.softmax(v, dim=1)
    s = torch.sigmoid(v)
    return s / s.sum(1, keepdim=True)


def _dispatch(ids, E):
    """Offsets, rows and positions of the (token, choice) pairs grouped by expert, tokens ascending."""
    T, k = ids.shape
    flat = ids.reshape(-1)
    order = torch.sort(flat, stable=True).indices
    pos = torch.empty_like(order)
    pos[order] = torch.arange(order.numel(), device=ids.device)
    offsets = torch.zeros(E + 1, dtype=torch.int64, device=ids.device)
    offsets[1:] = torch.cumsum(torch.bincount(flat, minlength=E), 0)
    return offsets.to(torch.int32), (order // k).to(torch.int32), pos.view(T, k).to(torch.int32)


def exact(case, seed):
    if case["L"] * case["T"] * case["E"] > 1 << 31:
        return None
    k, gate, kind, L, E = case["k"], case["gate"], case["kind"], case["L"], case["E"]
    got = {}

    def add(**kw):
        for name, v in kw.items():
            got.setdefault(name, []).append(v)

    s = prepare(case, seed)
    for l in range(L):
        if kind == "router":
            X, W = s["X"][l], s["W"][l].double()
            z = torch.cat([X[a:a + 8192].double() @ W.T for a in range(0, X.shape[0], 8192)])
        else:
            z = s["z"].detach()[l]
        if kind == "routing":
            ids = torch.cat([_select(z[a:a + 65536], k) for a in range(0, z.shape[0], 65536)])
            out = {"counts": torch.bincount(ids.reshape(-1), minlength=E).to(torch.int32)}
        else:
            out, ids = _layer(z, k, gate)
        if kind in ("routing", "routed"):
            offsets, rows, pos = _dispatch(ids, E)
            w = _combine(z, ids, gate)
            out.update(ids=ids.to(torch.int32), combine=w, offsets=offsets, rows=rows, pos=pos)
        if kind == "routed":
            g = s["g"][l].double()
            d = w * (g - (g * w).sum(1, keepdim=True))
            if gate != SOFTMAX:
                d = d * torch.sigmoid(-z.double().gather(1, ids))
            out["dlogits"].scatter_add_(1, ids, d)
        if kind == "router":
            dz = out["dlogits"]
            dW = torch.zeros(E, W.shape[1], dtype=torch.float64, device=z.device)
            dX = torch.empty(X.shape, dtype=torch.float64, device=z.device)
            for a in range(0, X.shape[0], 8192):
                dW += dz[a:a + 8192].T @ X[a:a + 8192].double()
                dX[a:a + 8192] = dz[a:a + 8192] @ W
            # a near-tie that fp32 sums decide otherwise changes whole numbers: no such value there
            out = {"loss": out["loss"], "dlogits": dz, "logits": z, "dW": dW, "dX": dX}
        if kind == "autograd":
            out = {"loss": out["loss"], "dlogits": LOSS_WEIGHT * out["dlogits"]}
        add(**out)
    full = {name: torch.stack(v) for name, v in got.items()}
    if kind == "router":
        full.update(bits=None, counts=None, D=None, origin_do=None)
    return full
