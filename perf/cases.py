"""The workloads this library is timed on: one verification block (or a batch of blocks) through a stack of MoE layers.

A case is a plain dict: the layer's shape (hidden, experts, top_k, inter, shared, dtype), the number of stacked layers,
the sizes of the verification blocks, and how the library is called (`call`).  Shapes are those of the
configurations in `workloads.py`; `draw` spreads over the same ranges, odd sizes included.  Every layer of a stack has
weights and hidden states of its own, so that experts stream cold, as they do in a model.
"""
import math
from dataclasses import replace

import torch

from paper_2608_02989_b200 import acm, workloads as wl

DEVICE = "cuda:0"
# call:
#   verify    acm_moe_verify per layer, tensors on the device (what a serving loop runs)
#   natural   the same with every expert eligible (the target model's own routing)
#   host      acm_moe_verify_host per layer: pinned host buffers in and out
#   batch     acm_moe_verify_batch per layer: several blocks share one pass over the experts
#   stages    acm_router, acm_select_eligible, acm_route_restricted, acm_expert_ffn one by one
#   offload   acm_moe_verify on layers of which a part of the experts is resident, the others in pinned host memory
# weights: "bf16", "f32" or "mxfp4" (routed experts in MXFP4, the rest bf16)


def _case(config, call, blocks, layers, weights=None, zipf=None, **kw):
    c = wl.CONFIGS[config]
    case = {"call": call, "weights": weights or c.dtype, "hidden": c.hidden, "experts": c.n_experts, "top_k": c.top_k,
            "inter": c.inter, "shared": c.n_shared, "weighting": c.weighting, "depth": c.max_depth, "layers": layers,
            "zipf": c.zipf_bias if zipf is None else zipf, "p_scale": c.p_scale, "p_decay": c.p_decay,
            "blocks": "+".join(str(b) for b in blocks), "resident": 1.0, "residency": 0}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest block there is: the fp32 toy layer, 8 nodes -- launches and latency are all that counts
        {"name": "toy-f32", **_case(1, "verify", [8], 1)},
        # no draft at all (a plain decode step): the root alone, top-k experts per layer
        {"name": "qwen30b-root", **_case(3, "verify", [1], 8)},
        # the headline: full 64-node blocks, skewed routing, about 22 of 128 experts a layer
        {"name": "qwen30b-block", **_case(3, "verify", [64], 12)},
        # diffuse routing over 64 experts, 32-node blocks, raw softmax weights
        {"name": "olmoe-block", **_case(2, "verify", [32], 8)},
        # an odd block on layers with always-on shared experts
        {"name": "deepseek-block", **_case(4, "verify", [47], 6)},
        # the largest: about a hundred 38 MB experts a layer
        {"name": "qwen235b-block", **_case(5, "verify", [64], 2)},
        # the same blocks as the headline through host buffers: upload, layer, download
        {"name": "qwen30b-host", **_case(3, "host", [64], 8)},
        # four ragged requests verified together (64-row accumulators)
        {"name": "qwen30b-batch", **_case(3, "batch", [23, 9, 17, 6], 6)},
        # two full blocks together (128-row accumulators)
        {"name": "qwen30b-batch-wide", **_case(3, "batch", [64, 61], 6)},
        # the headline with the routed experts stored in MXFP4
        {"name": "qwen30b-mxfp4", **_case(3, "verify", [64], 8, weights="mxfp4")},
        # a caller that drives the stages itself (its own anchors, its own set), every result returned
        {"name": "olmoe-stages", **_case(2, "stages", [29], 4)},
        # 40 % of the experts on the GPU; non-resident anchors are copied in on demand
        {"name": "qwen30b-offload", **_case(3, "offload", [64], 1, resident=0.4, residency=2)},
    ]


def draw(rng):
    """One more case: a call, a layer shape and block sizes from the ranges that the listed cases stand for."""
    call = rng.choice(["verify", "verify", "verify", "natural", "host", "batch", "batch", "stages", "mxfp4", "mxfp4", "f32",
                       "offload"])
    log_int = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if call == "f32":           # toy-sized layers: any hidden that is a multiple of 32
        experts = rng.randint(5, 40)
        return _case(1, rng.choice(["verify", "stages"]), [log_int(1, 40)], 1, hidden=32 * rng.randint(3, 16),
                     inter=32 * rng.randint(2, 20), experts=experts, top_k=rng.randint(1, min(8, experts)), depth=rng.randint(1, 6))
    weights = "mxfp4" if call == "mxfp4" else "bf16"
    base = rng.choice([2, 3, 3, 4, 5])
    c = wl.CONFIGS[base]
    kw = {"hidden": c.hidden, "inter": c.inter, "experts": c.n_experts, "top_k": c.top_k, "shared": c.n_shared,
          "weighting": rng.randint(0, 2), "depth": rng.randint(3, 8)}
    if rng.random() < 0.5:      # a shape between the configurations' own
        kw.update(hidden=128 * rng.randint(8, 32), inter=64 * rng.randint(8, 24), experts=rng.randint(24, 128),
                  top_k=rng.randint(2, 8), shared=rng.choice([0, 0, 0, 1, 2]))
    if weights == "mxfp4":
        kw.update(shared=0, inter=128 * max(4, kw["inter"] // 128))
        call = rng.choice(["verify", "verify", "natural", "batch"])
    elif call in ("offload", "stages"):
        kw["shared"] = 0 if call == "offload" else kw["shared"]
    if call == "offload":
        kw.update(resident=rng.uniform(0.25, 0.75), residency=rng.choice([1, 2]), experts=min(kw["experts"], 64),
                  hidden=min(kw["hidden"], 2048), inter=min(kw["inter"], 1024))
        kw["top_k"] = min(kw["top_k"], kw["experts"])
    if call == "batch":
        total = log_int(6, 64 if weights == "mxfp4" else 128)
        n = rng.randint(2, min(8, total))
        cuts = sorted(rng.sample(range(1, total), n - 1))
        blocks = [b - a for a, b in zip([0] + cuts, cuts + [total])]
        if max(blocks) > 64:
            blocks = [x for b in blocks for x in ([b // 2, b - b // 2] if b > 64 else [b])]
    else:
        blocks = [log_int(1, 64)]
    case = _case(base, call, blocks, 1, weights=weights, zipf=rng.random() < 0.6, **kw)
    if call not in ("offload", "natural"):      # as many layers as stay well below the largest listed case
        case["layers"] = max(1, min(8, int(4e9 / work(case)["bytes"]), int(8e9 / _layer_bytes(case))))
    return case


# ------------------------------------------------------------------------------------------------------------------
def _blocks(case):
    return [int(b) for b in case["blocks"].split("+")]


def _config(case, seed):
    return wl.BlockConfig(index=100 + seed, name="case", dtype="f32" if case["weights"] == "f32" else "bf16",
                          hidden=case["hidden"], n_experts=case["experts"], top_k=case["top_k"], inter=case["inter"],
                          n_shared=case["shared"], n_nodes=sum(_blocks(case)), max_depth=case["depth"],
                          n_layers=case["layers"], p_scale=case["p_scale"], p_decay=case["p_decay"],
                          weighting=case["weighting"], zipf_bias=case["zipf"], resident_frac=case["resident"])


def _pinned(t):
    host = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    host.copy_(t)
    return host


def prepare(case, seed):
    """The context with its layers' weights, and per layer a block: hidden states, node weights, output buffers."""
    cfg = _config(case, seed)
    sizes = _blocks(case)
    T, L, dev = cfg.n_nodes, cfg.n_layers, torch.device(DEVICE)
    ctx = acm.Context.for_config(cfg, max_nodes=max(sizes))
    table = wl.commitment_table(cfg)
    offsets, alpha = [0], []
    for i, n in enumerate(sizes):                       # every block is a draft tree of its own
        depth = wl.tree_depths(replace(cfg, n_nodes=n, index=cfg.index + 7919 * i))
        alpha.append(acm.node_weights(depth, table))
        offsets.append(offsets[-1] + n)
    alpha = torch.cat(alpha)
    state = {"call": case["call"], "ctx": ctx, "layers": L, "offsets": offsets, "alpha": alpha.to(dev),
             "params": acm.SelectParams(residency=case["residency"])}
    for layer in range(L):
        if case["weights"] == "mxfp4":
            w = wl.layer_weights_mxfp4(cfg, layer, dev)
            ctx.set_layer_weights_mxfp4(layer, w["w_router"], w["router_bias"],
                                        acm.pack_mxfp4_gate_up(w["gate_up_codes"], w["gate_up_scales"]),
                                        acm.pack_mxfp4_down(w["down_codes"], w["down_scales"]))
            continue
        w = wl.layer_weights(cfg, layer, dev)
        if case["call"] == "offload":
            gate_up_host, down_host = _pinned(w["gate_up"]), _pinned(w["down"])
            mask = wl.resident_mask(cfg, layer)
            absent = [e for e in range(cfg.n_experts) if not (int(mask[e // 32]) >> (e % 32)) & 1]
            w["gate_up"][absent] = float("nan")         # the device tensors hold the resident experts only
            w["down"][absent] = float("nan")
        ctx.set_layer_weights(layer, w["w_router"], w["router_bias"], w["gate_up"], w["down"], w["shared_gate_up"],
                              w["shared_down"])
        if case["call"] == "offload":
            ctx.set_resident(layer, mask, gate_up_host, down_host)
    x = [wl.hidden_states(cfg, layer, dev) for layer in range(L)]
    if case["call"] == "host":
        state["alpha"] = _pinned(alpha)
        state["x"] = [_pinned(t) for t in x]
        state["out"] = [torch.empty(T, cfg.hidden, dtype=torch.float32, pin_memory=True) for _ in range(L)]
    else:
        state["x"] = x
        state["out"] = [torch.empty(T, cfg.hidden, dtype=torch.float32, device=dev) for _ in range(L)]
    if case["call"] == "natural":
        state["every"] = torch.full((ctx.words,), -1, dtype=torch.int32, device=dev)
    return state


def run(state):
    ctx, x, alpha, out, params = state["ctx"], state["x"], state["alpha"], state["out"], state["params"]
    call, layers = state["call"], range(state["layers"])
    if call in ("verify", "offload"):
        for l in layers:
            ctx.moe_verify(l, x[l], alpha, params, out=out[l])
        return out
    if call == "natural":
        for l in layers:
            ctx.moe_verify(l, x[l], alpha, mask_override=state["every"], out=out[l])
        return out
    if call == "host":
        for l in layers:
            ctx.moe_verify_host(l, x[l], alpha, out[l], params)
        ctx.host_synchronize()
        return out
    if call == "batch":
        for l in layers:
            ctx.moe_verify_batch(l, x[l], state["offsets"], alpha, params, out=out[l])
        return out
    results = []
    for l in layers:
        logits, probs, natural = ctx.router(l, x[l])
        sel = ctx.select_eligible(probs, natural, alpha, params)
        idx, w = ctx.route_restricted(logits, sel["mask"])
        ctx.expert_ffn(l, x[l], idx, w, out=out[l])
        results.append({"logits": logits, "natural": natural, "mask": sel["mask"], "demand": sel["demand"], "idx": idx, "w": w,
                        "out": out[l]})
    return results


# ------------------------------------------------------------------------------------------------------------------
def _expert_bytes(case):
    n = 3 * case["hidden"] * case["inter"]
    return n * 4 if case["weights"] == "f32" else n * 2 if case["weights"] == "bf16" else n * 17 // 32


def _layer_bytes(case):
    return (case["experts"] + case["shared"]) * _expert_bytes(case)


def _expected_experts(case):
    """(activated experts a layer, those of them loaded from the host): the mean over a few draws of the logits'
    distribution -- N(0, 0.02^2 hidden) plus the popularity bias -- of natural top-k, demand and self-sizing."""
    E, k = case["experts"], case["top_k"]
    g = torch.Generator().manual_seed(1)
    total = loaded = 0.0
    draws = 8
    for _ in range(draws):
        bias = torch.zeros(E)
        if case["zipf"]:
            bias = -1.1 * torch.log(torch.arange(1, E + 1, dtype=torch.float32))
        union = torch.zeros(E, dtype=torch.bool)
        fetched = 0
        for n in _blocks(case):
            z = torch.randn(n, E, generator=g) * 0.02 * math.sqrt(case["hidden"]) + bias
            r, nat = torch.softmax(z, 1), torch.zeros(n, E).scatter_(1, z.topk(k, 1).indices, 1.0)
            chosen = nat.any(0)
            if case["call"] != "natural":
                anchor = nat[0] > 0
                level = torch.linspace(0, case["depth"], n).round()
                u = ((case["p_decay"] ** level).sqrt()[:, None] * r * nat).sum(0).masked_fill(anchor, 0.0)
                keep = anchor.clone()
                if float(u.sum()) > 0:
                    p = u[u > 0] / u.sum()
                    n_er = max(int(math.ceil(math.exp(float(-(p * p.log()).sum())))), k - int(anchor.sum()))
                    keep[u.topk(min(n_er, int((u > 0).sum()))).indices] = True
                chosen = keep
                if case["call"] == "offload":
                    resident = torch.rand(E, generator=g) < case["resident"]
                    if case["residency"] == 2:
                        chosen = (keep & resident) | anchor
                    fetched += int((chosen & ~resident).sum())
            union |= chosen
        total += float(union.sum())
        loaded += fetched
    return total / draws, loaded / draws


def work(case):
    """Per layer: router rows, hidden states, every activated (and shared) expert's weights once, the output once.  An
    expert loaded on demand is read from the host tensor once and counts once."""
    T, H, I, E, L = sum(_blocks(case)), case["hidden"], case["inter"], case["experts"], case["layers"]
    elt = 4 if case["weights"] == "f32" else 2
    activated, _ = _expected_experts(case)
    layer_bytes = (E * H + T * H) * elt + (activated + case["shared"]) * _expert_bytes(case) + T * H * 4
    layer_flops = 2.0 * T * H * E + 6.0 * T * (case["top_k"] + case["shared"]) * H * I
    return {"bytes": L * layer_bytes, "flops": L * layer_flops}


def tolerance(case):
    # Four times what the layer's output differs from the expert FFN in 64 bits on the routes the library returned:
    # fp32 layers 1.6e-7 (2-norm) and 7.4e-7 (largest, over the RMS); bf16 layers 1.66e-3 (1.56e-3 to 1.73e-3 over eleven
    # shapes) and 9.8e-3 -- the activation between the two products is rounded to bf16.  Whole numbers are the same.
    if case["weights"] == "f32":
        return {"rel": 7e-7, "max": 4e-6}
    return {"rel": 7e-3, "max": 4e-2}


# ------------------------------------------------------------------------------------------------------------------
def _exact_select(p, taken, alpha, params, k, resident):
    """The eligible set of one block in 64 bits: Eq. 4 to 7 on probabilities `p` [n, E] and natural membership `taken`."""
    E = p.shape[1]
    u = (alpha[:, None] * p * taken).sum(0)
    votes, anchor = taken.sum(0), taken[0]
    rest = torch.where(anchor, 0.0, u)
    positive = int((rest > 0).sum())
    keep = max(0, k - int(anchor.sum()))
    if positive:
        q = rest[rest > 0] / rest.sum()
        keep = max(keep, min(max(math.ceil(math.exp(float(-(q * q.log()).sum())) - params.ceil_guard), 1), positive))
    order = sorted((e for e in range(E) if not anchor[e]), key=lambda e: (-float(u[e]), e))
    S = anchor.clone()
    S[order[:keep]] = True
    if params.residency == 2:
        S = (S & resident) | anchor
    elif params.residency == 1:
        budget, moved, size, removed = int(votes[~S].sum()), 0, int(S.sum()), []
        for e in sorted((e for e in range(E) if S[e] and not resident[e]), key=lambda e: (float(u[e]), e)):
            moved += int(votes[e])
            if moved > budget or size - len(removed) - 1 < k or len(removed) == params.max_remove:
                break
            removed.append(e)
        S[removed] = False
    return S, u


def _exact_weights(w, experts):
    """expert -> (gate_up [2I, H], down [H, I]) in 64 bits"""
    def mxfp4(codes, scales):
        grid = torch.tensor(wl.E2M1_VALUES, dtype=torch.float64, device=codes.device)
        value = grid[(codes & 7).long()] * torch.where(codes >= 8, -1.0, 1.0)
        return value * torch.exp2(scales.double() - 127).repeat_interleave(32, -1)
    if w["gate_up"] is None:
        return lambda e: (mxfp4(w["gate_up_codes"][e], w["gate_up_scales"][e]), mxfp4(w["down_codes"][e], w["down_scales"][e]))
    return lambda e: (w["gate_up"][e].double(), w["down"][e].double()) if e < experts else \
        (w["shared_gate_up"][e - experts].double(), w["shared_down"][e - experts].double())


def exact(case, seed):
    """What `run` returns, in 64 bits throughout: routes are ranked on 64-bit logits, and the activation between the two
    products is not rounded."""
    cfg, dev, sizes = _config(case, seed), torch.device(DEVICE), _blocks(case)
    E, k, T, params = cfg.n_experts, cfg.top_k, cfg.n_nodes, acm.SelectParams(residency=case["residency"])
    table, alpha = wl.commitment_table(cfg).double(), []
    for i, n in enumerate(sizes):
        depth = wl.tree_depths(replace(cfg, n_nodes=n, index=cfg.index + 7919 * i)).long()
        alpha.append((table[depth].sqrt() / torch.bincount(depth)[depth].double().sqrt()).float().double().to(dev))
    results = []
    for layer in range(cfg.n_layers):
        w = wl.layer_weights_mxfp4(cfg, layer, dev) if case["weights"] == "mxfp4" else wl.layer_weights(cfg, layer, dev)
        mask = wl.resident_mask(cfg, layer).tolist()
        resident = torch.tensor([bool((mask[e // 32] >> (e % 32)) & 1) for e in range(E)])
        x = wl.hidden_states(cfg, layer, dev).double()
        z = x @ w["w_router"].double().T + (0 if w["router_bias"] is None else w["router_bias"].double())
        p, natural = torch.softmax(z, 1), z.sort(dim=1, descending=True, stable=True).indices[:, :k]
        taken = torch.zeros(T, E, dtype=torch.bool, device=dev).scatter_(1, natural, True)
        eligible, demand, row = torch.ones(T, E, dtype=torch.bool, device=dev), None, 0
        for n, a in zip(sizes, alpha) if case["call"] != "natural" else ():
            S, demand = _exact_select(p[row:row + n].cpu(), taken[row:row + n].cpu(), a.cpu(), params, k, resident)
            eligible[row:row + n] = S.to(dev)
            row += n
        zr = z.masked_fill(~eligible, float("-inf"))
        top = zr.sort(dim=1, descending=True, stable=True)
        zk, idx = top.values[:, :k], top.indices[:, :k]
        wk = torch.softmax(zk, 1) if cfg.weighting == 0 else p.gather(1, idx) if cfg.weighting == 1 else torch.softmax(zr, 1).gather(1, idx)
        wk = wk.masked_fill(zk == float("-inf"), 0.0)
        weight = torch.zeros(T, E + cfg.n_shared, dtype=torch.float64, device=dev).scatter_(1, idx, wk)
        weight[:, E:] = 1.0
        out, expert = torch.zeros(T, cfg.hidden, dtype=torch.float64, device=dev), _exact_weights(w, E)
        for e in weight.any(0).nonzero().flatten().tolist():
            rows = weight[:, e].nonzero().flatten()
            gate_up, down = expert(e)
            g, up = (x[rows] @ gate_up.T).chunk(2, 1)
            out[rows] += weight[rows, e, None] * ((torch.nn.functional.silu(g) * up) @ down.T)
        results.append(out if case["call"] != "stages" else
                       {"logits": z, "natural": None, "mask": None, "demand": demand.to(dev), "idx": None, "w": wk, "out": out})
    return results
