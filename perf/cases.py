"""Workloads of the masked MoE layer that users of libmcft run, as cases to be timed and checked.

A case is one pass of a user's program through the public entry points of
``paper_2609_34077_gb300.mcft``: routing, the layer forward and what belongs to it, on inputs that
are already on the GPU and with the weights, workspaces, caches and stacks such a program keeps.
Kinds of passes (``kind``):

* ``decode``   soft-prior routing and the forward of a layer whose experts are all resident, for the
               1 to 64 tokens of one decode step;
* ``prefill``  the same two calls for a prompt, a chunk of a prompt or a fine-tuning batch of 65 to
               4096 tokens, routed under a hard mask or a soft prior;
* ``cached``   a few decode steps of a layer whose experts come from the cache: routing, cache step
               and the forward that fetches the misses from pinned host memory;
* ``stack``    one decode step of a chained stack of layers with next-layer prefetch;
* ``lora``     the Stage-2 forward: hard-mask routing and the layer with LoRA adapters (rank 8 / 16);
* ``mask``     the Stage-1 step: mask sampling, hard-mask routing, the forward, dL/dgate and the
               straight-through mask gradient.

Ranges (``draw``): hidden sizes and widths of 128 to 4096 (and the two model shapes of
``inputs.py``) in multiples of 64, 4 to 64 experts, 1 to 8 of them active, 0 to 3 shared experts,
bf16 and, for small layers, fp32; batches as above.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_34077_gb300 import inputs as I
from paper_2609_34077_gb300 import mcft as M

DEV = "cuda"


def _case(kind, shape, T, name=None, **kw):
    c = dict(kind=kind, T=int(T), d=shape.d, E=shape.E, K=shape.K, w=shape.w, S=shape.n_shared,
             gate=shape.gate, dtype="bf16" if shape.dtype == I.BF16 else "f32",
             mode="soft", keep=shape.keep)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    mix, ds, tiny = I.MIXTRAL, I.DSV2_LITE, I.TINY
    odd = I.LayerShape("odd", d=960, E=16, K=4, w=704, n_shared=1, gate=I.GATE_RENORM, dtype=I.BF16,
                       cache_slots=4, keep=12)
    return [
        # one user's next token: the smallest call, where launches and latency count
        _case("decode", ds, 1, "decode-ds-b1"),
        # a small serving batch of the layer with few wide experts: every expert's weights stream
        _case("decode", mix, 16, "decode-mix-b16"),
        # a ragged serving batch of the layer with many narrow experts
        _case("decode", ds, 50, "decode-ds-b50"),
        # offloaded decoding: four steps of a batch whose misses come over the host link
        _case("cached", ds, 8, "cached-ds-b8", steps=4, slots=ds.cache_slots, policy="LRU"),
        # offloaded decoding of a chained stack at batch 1, with prefetch of the next layer
        _case("stack", ds, 1, "stack-ds-b1", layers=3, slots=ds.cache_slots, policy="LRU",
              prefetch=2),
        # the tail chunk of a prompt: few tokens per expert, more than a decode batch
        _case("prefill", ds, 200, "chunk-ds-200"),
        # prompts / fine-tuning batches of 8 x 512 tokens under the hard mask, both model shapes
        _case("prefill", ds, 4096, "prefill-ds-4096", mode="hard", keep=48),
        _case("prefill", mix, 4096, "prefill-mix-4096", mode="hard"),
        # a layer whose sizes are no multiples of the tensor-core tiles
        _case("prefill", odd, 1023, "prefill-odd-1023"),
        # Stage-2 fine-tuning forward with adapters on every expert
        _case("lora", mix, 1000, "lora-mix-1000", mode="hard", rank=8),
        # Stage-1 mask optimisation step
        _case("mask", mix, 2048, "mask-mix-2048", mode="hard", keep=6, layers=32),
        # the fp32 layer of the parity configuration, at a prompt's length
        _case("prefill", tiny, 512, "prefill-f32-512", mode="hard"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _generic(rng, dmax, wmax, dtype):
    E = rng.randint(4, 64)
    K = rng.randint(1, min(8, E // 2))
    return I.LayerShape("generic", d=64 * _log_int(rng, 2, dmax // 64), E=E, K=K,
                        w=64 * _log_int(rng, 2, wmax // 64), n_shared=rng.choice([0, 0, 1, 2, 3]),
                        gate=rng.choice([I.GATE_RENORM, I.GATE_PLAIN]), dtype=dtype, cache_slots=max(K, E // 4),
                        keep=max(K, (3 * E) // 4))


def draw(rng):
    kind = rng.choice(["decode", "decode", "prefill", "prefill", "prefill", "cached", "stack", "lora",
                       "mask", "f32"])
    dtype = I.BF16
    if kind == "f32":
        kind, dtype = rng.choice(["decode", "prefill"]), I.F32
    if dtype == I.F32:
        shape = _generic(rng, 512, 1024, dtype)
    else:
        shape = rng.choice([I.MIXTRAL, I.DSV2_LITE, "generic", "generic"])
        if kind in ("cached", "stack") and shape is I.MIXTRAL:
            shape = I.DSV2_LITE  # (host blocks of 2.8 GB a layer take too long to lay out)
        if shape == "generic":
            d, w = {"decode": (4096, 4096), "cached": (1024, 1024), "stack": (1024, 1024)}.get(kind, (4096, 2048))
            shape = _generic(rng, d, w, dtype)
    mode = rng.choice(["soft", "hard"])
    if kind in ("decode", "cached", "stack"):
        mode = "soft"
    if kind in ("lora", "mask"):
        mode = "hard"
    kw = dict(mode=mode)
    if mode == "hard" and shape is I.DSV2_LITE:
        kw["keep"] = 48
    if kind == "decode":
        T = _log_int(rng, 1, 64)
    elif kind == "cached":
        T = _log_int(rng, 1, 16)
        kw.update(steps=rng.randint(1, 2) if T > 8 else rng.randint(2, 4), slots=shape.cache_slots,
                  policy=rng.choice(["LRU", "LFU", "FIFO"]))
    elif kind == "stack":
        T = rng.choice([1, 1, 2, 3, 4])
        kw.update(layers=rng.randint(2, 3), slots=shape.cache_slots,
                  policy=rng.choice(["LRU", "LFU", "FIFO"]),
                  prefetch=rng.choice([0, min(2, shape.cache_slots)]))
    elif dtype == I.F32:
        T = _log_int(rng, 65, 512)
    else:
        T = _log_int(rng, 65, 4096 if shape.n_shared < 3 and shape.K < 7 else 2048)
    if kind == "lora":
        T = min(T, 3000)  # the adapters' share comes on top
        kw["rank"] = rng.choice([8, 16])
    if kind == "mask":
        T = min(T, 3000)
        kw["layers"] = rng.choice([26, 32])
    return _case(kind, shape, T, **kw)


def _dt(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _desc(case):
    return M.LayerDesc(case["d"], case["E"], case["K"], case["w"], case["S"], case["gate"],
                       M.MCFT_BF16 if case["dtype"] == "bf16" else M.MCFT_F32)


def _normal(g, dtype, *shape, std=1.0, mean=0.0):
    return (torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32) * std + mean).to(dtype)


def _blocks(g, case, n):
    """n packed expert blocks [W1 | W3 | W2], N(0, 0.02^2)."""
    return [_normal(g, _dt(case), 3 * case["w"] * case["d"], std=0.02) for _ in range(n)]


def _pinned(blocks):
    """The blocks in one pinned host allocation (as an offloading server keeps them)."""
    n = blocks[0].numel()
    host = torch.empty(len(blocks), n, dtype=blocks[0].dtype, pin_memory=True)
    for h, b in zip(host, blocks):
        h.copy_(b, non_blocking=True)
    return [host[i] for i in range(len(blocks))]


def _ar1(g, case, steps):
    """Decode hidden states [steps, T, d]: one stationary AR(1) stream per row, rho = 0.8."""
    eps = torch.randn(steps, case["T"], case["d"], generator=g, device=DEV)
    x = torch.empty_like(eps)
    x[0] = eps[0] / 0.6
    for t in range(1, steps):
        x[t] = 0.8 * x[t - 1] + eps[t]
    return x


def _lora_sizes(case):
    d, w, r = case["d"], case["w"], case["rank"]
    return [(r, d), (w, r), (r, d), (w, r), (r, w), (d, r)]  # A1 B1 A3 B3 A2 B2


def _adapter(g, case):
    """Packed trained adapter: A ~ N(0, 0.02^2), B ~ N(0, 0.05^2)."""
    parts = [_normal(g, _dt(case), a * b, std=0.02 if i % 2 == 0 else 0.05)
             for i, (a, b) in enumerate(_lora_sizes(case))]
    return torch.cat(parts)


def _inputs(case, seed):
    """Everything that is drawn for a case: the same for run() and exact()."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + 17)
    kind, E, d = case["kind"], case["E"], case["d"]
    layers = case["layers"] if kind == "stack" else 1
    keep = [I.keep_mask(int(seed), E, case["keep"], layer=l) for l in range(layers)]
    s = dict(case=case, desc=_desc(case), keep=keep, prior=[I.prior_from_mask(k) for k in keep],
             mode=M.MCFT_ROUTE_HARD_MASK if case["mode"] == "hard" else M.MCFT_ROUTE_SOFT_PRIOR)
    s["routers"] = [_normal(g, _dt(case), E, d, std=0.02) for _ in range(layers)]
    s["experts"] = [_blocks(g, case, E) for _ in range(layers)]
    s["shared"] = [_blocks(g, case, case["S"]) for _ in range(layers)]
    if kind == "stack":
        s["gammas"] = [_normal(g, _dt(case), d, std=0.1, mean=1.0) for _ in range(layers)]
        s["x0"] = _ar1(g, case, 1)[0].to(_dt(case)).float()
    elif kind in ("decode", "cached"):
        s["x"] = _ar1(g, case, case.get("steps", 1)).to(_dt(case))
    else:
        s["x"] = _normal(g, _dt(case), 1, case["T"], d)
    if kind == "lora":
        s["lora"] = [_adapter(g, case) for _ in range(E)]
        s["shared_lora"] = [_adapter(g, case) for _ in range(case["S"])]
        s["scale"] = 16.0 / case["rank"]
    if kind == "mask":
        s["dy"] = _normal(g, _dt(case), case["T"], d)
        s["m_tilde"] = 2.0 * torch.rand(case["layers"], E, generator=g, device=DEV)
        s["u"] = torch.rand(case["layers"], E, generator=g, device=DEV).clamp(2.0 ** -24, 1 - 2.0 ** -24)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind, T, desc = case["kind"], case["T"], s["desc"]
    if kind in ("cached", "stack"):
        s["host"] = _pinned([b for layer in s["experts"] for b in layer])
        del s["experts"]
        s["cache"] = M.mcft_cache_create(len(s["routers"]), case["E"], case["slots"],
                                         s["host"][0].numel() * s["host"][0].element_size(), s["host"],
                                         max_assign=T * case["K"], policy=case["policy"])
        s["copy"] = torch.cuda.Stream()
    if kind == "stack":
        s["stack"] = M.mcft_stack_create(desc, s["routers"], np.stack(s["prior"]), s["gammas"],
                                         s["shared"] if case["S"] else None, 1e-6, s["cache"],
                                         n_prefetch=case["prefetch"], T_max=T)
        s["xs"] = torch.empty_like(s["x0"])
        return s
    steps = s["x"].shape[0]
    s["idx"] = torch.empty(steps, T, case["K"], dtype=torch.int32, device=DEV)
    s["gates"] = torch.empty(steps, T, case["K"], dtype=torch.float32, device=DEV)
    s["y"] = torch.empty_like(s["x"])
    nbytes = (M.mcft_moe_workspace_size_lora(desc, case["rank"], T) if kind == "lora"
              else M.mcft_moe_workspace_size(desc, T))
    s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
    if kind == "mask":
        s["dgate"] = torch.empty(T, case["K"], dtype=torch.float32, device=DEV)
    return s


def run(s):
    case, desc = s["case"], s["desc"]
    kind = case["kind"]
    if kind == "stack":
        s["xs"].copy_(s["x0"])
        M.mcft_stack_step(s["stack"], s["xs"], copy_stream=s["copy"])
        return {"x": s["xs"]}
    extra = dict(mask=s["keep"][0]) if case["mode"] == "hard" else dict(prior=s["prior"][0])
    out = {"y": s["y"], "idx": s["idx"], "gate": s["gates"]}
    if kind == "mask":
        mask, pi = M.mcft_mask_sample(s["m_tilde"], s["u"], case["keep"])
    for t in range(s["x"].shape[0]):
        x, y = s["x"][t], s["y"][t]
        idx, gate = M.mcft_route(desc, x, s["routers"][0], s["mode"], idx=s["idx"][t], gate=s["gates"][t],
                                 **extra)
        if kind == "cached":
            M.mcft_cache_step(s["cache"], 0, idx)
            M.mcft_moe_forward_cached(desc, x, idx, gate, s["cache"], 0, s["shared"][0], y=y,
                                      workspace=s["ws"], copy_stream=s["copy"])
        elif kind == "lora":
            M.mcft_moe_forward_lora(desc, x, idx, gate, s["experts"][0], s["shared"][0], s["lora"],
                                    s["shared_lora"], rank=case["rank"], scale=s["scale"], y=y,
                                    workspace=s["ws"])
        else:
            M.mcft_moe_forward(desc, x, idx, gate, s["experts"][0], s["shared"][0], y=y,
                               workspace=s["ws"])
    if kind == "mask":
        dgate = M.mcft_gate_grad(desc, s["dy"], s["ws"], dgate=s["dgate"])
        dm, dmt = M.mcft_mask_grad(desc, idx, gate, dgate, pi[0])
        out.update(mask=mask, pi=pi, dgate=dgate, dm=dm, dm_tilde=dmt)
    return out


def _routed(case):
    """Distinct experts of a typical batch: routing of T tokens with logits as the inputs give."""
    g = np.random.default_rng(1)
    E, K, T = case["E"], case["K"], case["T"]
    scale = 0.02 * math.sqrt(case["d"]) * (1 / 0.6 if case["kind"] in ("decode", "cached") else 1.0)
    z = scale * g.standard_normal((T, E))
    kept = np.arange(E) < case["keep"]
    z += np.where(kept, 2.0, 0.0) if case["mode"] == "soft" else np.where(kept, 0.0, -1e9)
    return len(np.unique(np.argpartition(-z, K - 1, axis=1)[:, :K]))


def work(case):
    """Weights of the experts a pass uses, its inputs and outputs, once each; the layer's products."""
    b = 2 if case["dtype"] == "bf16" else 4
    d, w, E, K, T, S = (case[k] for k in ("d", "w", "E", "K", "T", "S"))
    n = _routed(case)
    layers = case["layers"] if case["kind"] == "stack" else case.get("steps", 1)
    nbytes = (n + S) * 3 * w * d * b + E * d * b + 2 * T * d * b + T * K * 8
    rows = T * (K + S)
    flops = 6.0 * rows * w * d + 2.0 * T * E * d
    if case["kind"] == "lora":
        r = case["rank"]
        nbytes += (n + S) * 3 * r * (d + w) * b
        flops += 6.0 * rows * r * (d + w)
    if case["kind"] == "mask":
        nbytes += T * d * b + T * K * 4 + case["layers"] * E * 13
        flops += 2.0 * T * K * d
    return {"bytes": float(layers * nbytes), "flops": float(layers * flops)}


def tolerance(case):
    """Relative 2-norm of the difference; share of routing decisions that may differ (near ties)."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 2e-4, "differ": 1e-3}
    return {"rel": 1e-2, "max": 0.1, "differ": 2e-3}


# ---- the same passes in 64-bit torch, from the formulas ----
def _route64(case, x, router, keep, prior):
    z = x.double() @ router.double().t()
    p = torch.softmax(z, dim=-1)
    if case["mode"] == "hard":
        score = p.masked_fill(torch.from_numpy(keep == 0).to(DEV), -1.0)
    else:
        score = p * torch.from_numpy(prior).to(DEV).double()
    order = torch.sort(score, dim=-1, descending=True, stable=True).indices[:, :case["K"]]
    g = torch.gather(p, 1, order)
    if case["gate"] == I.GATE_RENORM:
        g = g / g.sum(-1, keepdim=True)
    return order, g


def _expert64(case, v, block, lora=None, scale=0.0):
    d, w = case["d"], case["w"]
    w1, w3, w2 = block[:w * d].view(w, d), block[w * d:2 * w * d].view(w, d), block[2 * w * d:].view(d, w)
    a1 = b1 = a3 = b3 = a2 = b2 = None
    if lora is not None:
        parts = torch.split(lora, [a * b for a, b in _lora_sizes(case)])
        a1, b1, a3, b3, a2, b2 = (q.view(*sz).double() for q, sz in zip(parts, _lora_sizes(case)))

    def lin(m, u, a, bb):
        o = u @ m.double().t()
        return o if a is None else o + scale * ((u @ a.t()) @ bb.t())

    gate, up = lin(w1, v, a1, b1), lin(w3, v, a3, b3)
    return lin(w2, torch.nn.functional.silu(gate) * up, a2, b2)


def _layer64(case, s, layer, v, idx, g, want_dgate=None):
    y = torch.zeros_like(v)
    dgate = torch.zeros(v.shape[0], case["K"], dtype=torch.float64, device=DEV)
    lora = s.get("lora")
    for e in range(case["E"]):
        t, k = torch.nonzero(idx == e, as_tuple=True)
        if t.numel() == 0:
            continue
        f = _expert64(case, v[t], s["experts"][layer][e], lora[e] if lora else None, s.get("scale", 0.0))
        y.index_add_(0, t, g[t, k, None] * f)
        if want_dgate is not None:
            dgate[t, k] = (want_dgate[t] * f).sum(-1)
    for i, b in enumerate(s["shared"][layer]):
        y += _expert64(case, v, b, s["shared_lora"][i] if lora else None, s.get("scale", 0.0))
    return y, dgate


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "stack":
        x = s["x0"].double()
        for l in range(case["layers"]):
            u = s["gammas"][l].double() * x / torch.sqrt((x * x).mean(-1, keepdim=True) + 1e-6)
            idx, g = _route64(case, u, s["routers"][l], s["keep"][l], s["prior"][l])
            x = x + _layer64(case, s, l, u, idx, g)[0]
        return {"x": x}
    ys, ids, gs = [], [], []
    for t in range(s["x"].shape[0]):
        v = s["x"][t].double()
        idx, g = _route64(case, v, s["routers"][0], s["keep"][0], s["prior"][0])
        y, dgate = _layer64(case, s, 0, v, idx, g, s["dy"].double() if kind == "mask" else None)
        ys.append(y)
        ids.append(idx.int())
        gs.append(g)
    out = {"y": torch.stack(ys), "idx": torch.stack(ids), "gate": torch.stack(gs)}
    if kind == "mask":
        lp = torch.log_softmax(s["m_tilde"].double(), dim=-1)
        keys = lp - torch.log(-torch.log(s["u"].double()))
        top = torch.topk(keys, case["keep"], dim=-1).indices
        mask = torch.zeros_like(keys).scatter_(1, top, 1.0).to(torch.uint8)
        c = g * (dgate - (g * dgate).sum(-1, keepdim=True)) if case["gate"] == I.GATE_RENORM else g * dgate
        dm = torch.zeros(case["E"], dtype=torch.float64, device=DEV)
        dm.index_add_(0, idx.reshape(-1), c.reshape(-1))
        pi = lp.exp()
        out.update(mask=mask, pi=pi, dgate=dgate, dm=dm, dm_tilde=pi[0] * (dm - (pi[0] * dm).sum()))
    return out
