"""The work that a user of the library has it do, as cases that can be timed and compared.

The library verifies the MoE layers of a target model on a batch or tree of draft tokens.  Its
users call it for a whole stack of layers (directly, from a captured graph, or with host buffers),
for single layers between their own attention kernels, with one token (plain decoding) up to 64,
and call the expansion step that picks the draft tokens.  The shapes are those of
``paper_2608_15018_b200.workloads`` (the model families of the paper's Table 1) with fewer layers,
every layer with weights of its own, so that no stack fits the L2 cache.

A case is a dict of plain values: ``path`` names the entry point ("stack", "graph", "layer",
"host", "expand"), ``shape`` an entry of ``workloads.CONFIGS`` whose fields the other values
replace.
"""
import math

import torch

from paper_2608_15018_b200 import binding, workloads

GB = 1e9
LARGEST = 5.2 * GB           # bytes that a pass of a drawn case may need at most (the largest listed case)
STATE = 14.0 * GB            # bytes of weights that a drawn case may hold


def listed():
    return [
        # one small fp32 layer: the smallest call, every microsecond of it latency and launches
        dict(name="tiny-f32", path="layer", shape="cfg1", layers=1, tokens=4, sigma=0.3),
        # plain decoding: one token, layer by layer between the caller's own kernels
        dict(name="olmoe-decode", path="layer", shape="cfg2", layers=8, tokens=1, sigma=0.5),
        # the headline: a chain of 8 draft tokens through the whole stack, captured once and replayed
        dict(name="olmoe-chain8", path="graph", shape="cfg2", layers=16, tokens=8, sigma=0.5),
        # the same from host buffers: inputs and results cross PCIe inside the call
        dict(name="olmoe-host8", path="host", shape="cfg2", layers=16, tokens=8, sigma=0.5),
        # a draft tree of 16 tokens; few routed experts and one large gated shared expert
        dict(name="qwen15-tree16", path="stack", shape="cfg3", layers=8, tokens=16, sigma=0.3),
        # block-int4 weights, a chain of 8 and a batch of 32
        dict(name="mixtral-q4-8", path="stack", shape="cfg4", layers=4, tokens=8, sigma=0.5),
        dict(name="mixtral-q4-32", path="stack", shape="cfg4", layers=4, tokens=32, sigma=0.5),
        # a draft tree of 16 tokens with two shared experts; the largest tree with scattered routing
        dict(name="dsv2lite-tree16", path="stack", shape="cfg5", layers=8, tokens=16, sigma=0.3),
        dict(name="dsv2lite-tree64", path="stack", shape="cfg5", layers=8, tokens=64, sigma=1.0),
        # 128 experts: many narrow ones with an odd batch, few wide ones at a ragged width (45 tiles of 64)
        dict(name="qwen3-chain13", path="stack", shape="e128a", layers=6, tokens=13, sigma=0.5),
        dict(name="gptoss-chain8", path="stack", shape="e128b", layers=2, tokens=8, sigma=0.5),
        # the step in front of a verification: expert sets of 64 candidates over 16 layers, admission
        dict(name="expand-64", path="expand", layers=16, tokens=64, experts=64, topk=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: any family, 1 to 64 tokens, any noise, the gating's options."""
    family = rng.choice(["cfg1", "cfg2", "cfg2", "cfg3", "cfg3", "cfg4", "cfg4", "cfg5", "cfg5", "e128a", "e128b",
                         "ragged", "ragged", "expand"])
    if family == "expand":
        return dict(path="expand", layers=_log_int(rng, 2, 48), tokens=_log_int(rng, 4, 160),
                    experts=rng.choice([8, 60, 64, 128]), topk=rng.choice([2, 4, 6, 8]))
    case = dict(path=rng.choice(["stack", "stack", "graph", "layer", "host"]),
                shape="cfg2" if family == "ragged" else family, layers=rng.randint(1, 8),
                tokens=_log_int(rng, 1, 64), sigma=round(rng.uniform(0.1, 1.0), 2),
                alpha=rng.choice([0.0, 0.25, 0.5, 0.5, 1.0]), weight_mode=rng.choice([0, 0, 1]),
                seed_conf=rng.random() < 0.75)
    wl = workloads.CONFIGS[case["shape"]]
    if family == "cfg1":
        case.update(path="layer", layers=1, tokens=rng.randint(1, 16), d_model=64 * rng.randint(2, 12),
                    d_ff=32 * rng.randint(8, 32))
    elif family == "ragged":
        # widths that are no multiple of the tiles, shared experts of another width than the routed ones
        experts = rng.choice([16, 24, 40, 64, 72])
        topk = rng.randint(2, 8)
        n_shared = rng.choice([0, 1, 2])
        case.update(d_model=64 * rng.randint(12, 56), d_ff=32 * rng.randint(16, 64), n_experts=experts, top_k=topk,
                    cap=min(experts, rng.randint(topk + 1, 3 * topk)), n_shared=n_shared,
                    d_ff_shared=32 * rng.randint(16, 96) if n_shared else 0, renorm=rng.randint(0, 1))
    else:
        case["cap"] = min(wl.n_experts, round(wl.top_k * rng.uniform(1.5, 2.5)))
    w = _workload(case, 0)
    per_layer = w.expert_bytes() * min(w.n_experts, w.top_k * (1 + case["tokens"])) + w.shared_bytes()
    held = w.expert_bytes() * w.n_experts + w.shared_bytes()
    case["layers"] = max(1, min(case["layers"], int(LARGEST / per_layer), int(STATE / held)))
    return case


def _workload(case, seed):
    wl = workloads.CONFIGS[case["shape"]]
    fields = {n: case[n] for n in ("d_model", "d_ff", "n_experts", "top_k", "cap", "n_shared", "d_ff_shared", "renorm",
                                   "alpha", "weight_mode", "sigma") if n in case}
    return wl.with_(n_tokens=case["tokens"], n_layers=case["layers"], seed=int(seed), **fields)


def _inputs(wl, case, device):
    """Hidden states [L][B][d] and prefix confidences [L][B] (or None: all ones)."""
    hidden = torch.stack([workloads.hidden_states(wl, i, device=device) for i in range(wl.n_layers)]).contiguous()
    conf = None
    if case.get("seed_conf", True):
        conf = torch.stack([workloads.confidences(wl, i) for i in range(wl.n_layers)]).to(device).contiguous()
    return hidden, conf


def _prepare_expand(case, seed):
    n, layers, experts, k = case["tokens"], case["layers"], case["experts"], case["topk"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    # every candidate's predicted experts: the best of a preference shared by the layer plus its own noise
    base = torch.randn((layers, 1, experts), generator=gen, device="cuda")
    own = torch.randn((layers, n, experts), generator=gen, device="cuda")
    sel = (base + 0.7 * own).topk(k, dim=-1).indices.to(torch.int32).contiguous()
    # a draft tree in heap order below four roots, the confidences of a drafter that is mostly right
    parent = torch.tensor([-1 if i < 4 else (i - 4) // 2 for i in range(n)], dtype=torch.int32, device="cuda")
    p_tok = (0.55 + 0.44 * torch.rand((n,), generator=gen, device="cuda")).contiguous()
    c_draft = torch.full((n,), 4.0, device="cuda")
    masks = torch.zeros((n, layers, (experts + 63) // 64), dtype=torch.int64, device="cuda")
    # microseconds: an autoregressive step of the target, one more expert in one layer
    return dict(case=case, sel=sel, parent=parent, p_tok=p_tok, c_draft=c_draft, masks=masks, t_ar=45.0 * layers, t_exp=2.1)


def prepare(case, seed):
    """Weights, the context that holds them, inputs and output buffers: what the program has before the call."""
    if case["path"] == "expand":
        return _prepare_expand(case, seed)
    wl = _workload(case, seed)
    device = torch.device("cuda", torch.cuda.current_device())
    weights = [workloads.layer_weights(wl, i, device) for i in range(wl.n_layers)]
    ctx = binding.S2MoE(binding.Config.from_workload(wl, max_tokens=case["tokens"]), weights)
    hidden, conf = _inputs(wl, case, device)
    s = dict(case=case, ctx=ctx, hidden=hidden, conf=conf)
    if case["path"] == "host":
        B, L = case["tokens"], wl.n_layers
        s["hidden"] = hidden.cpu().pin_memory()
        s["conf"] = None if conf is None else conf.cpu().pin_memory()
        s["out"] = [torch.empty((L, B, wl.d_model), dtype=torch.float32, pin_memory=True),
                    torch.empty((L, B, wl.top_k), dtype=torch.int32, pin_memory=True),
                    torch.empty((L, B, wl.top_k), dtype=torch.float32, pin_memory=True),
                    torch.empty((L,), dtype=torch.int32, pin_memory=True)]
        return s
    s["out"] = out = ctx.alloc_outputs(case["tokens"], stack=True)
    if case["path"] == "layer":
        s["views"] = [binding.LayerOutput(out.out[i], out.sel_idx[i], out.sel_w[i], out.n_unique[i:i + 1])
                      for i in range(wl.n_layers)]
        s["rows"] = [(hidden[i], None if conf is None else conf[i]) for i in range(wl.n_layers)]
    elif case["path"] == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            ctx.verify_stack(hidden, conf, out)
        side.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=side):
            ctx.verify_stack(hidden, conf, out, stream=side)
    return s


def run(state):
    """One pass: every layer's outputs, selected experts, mixing weights and unique-expert count."""
    path = state["case"]["path"]
    if path == "expand":
        for layer in range(state["case"]["layers"]):
            binding.expert_masks(state["sel"][layer], state["case"]["experts"], out=state["masks"], layer=layer)
        admitted, order, n_admitted, union = binding.adaptive_expand(
            state["parent"], state["p_tok"], state["masks"], state["case"]["experts"], state["c_draft"], state["t_ar"],
            state["t_exp"])
        return [state["masks"], admitted, order, n_admitted, union]
    ctx, out = state["ctx"], state["out"]
    if path == "host":
        ctx.verify_stack_host(state["hidden"], state["conf"], *out)
        return out
    if path == "graph":
        state["graph"].replay()
    elif path == "stack":
        ctx.verify_stack(state["hidden"], state["conf"], out)
    else:
        for layer, (hidden, conf) in enumerate(state["rows"]):
            ctx.verify_layer(layer, hidden, conf, state["views"][layer])
    return [out.out, out.sel_idx, out.sel_w, out.n_unique]


def work(case):
    """The distinct selected experts' weights once (their number counted on inputs of seed 0), the
    shared experts, router, hidden states and outputs; two operations per weight and token."""
    if case["path"] == "expand":
        words = case["layers"] * ((case["experts"] + 63) // 64)
        n = case["tokens"]
        return {"bytes": 4.0 * case["layers"] * n * case["topk"] + 8.0 * words * (n + 1) + 20.0 * n, "flops": 0.0}
    wl = _workload(case, 0)
    device = torch.device("cuda", torch.cuda.current_device())
    hidden, conf = _inputs(wl, case, device)
    cfg = binding.Config.from_workload(wl, max_tokens=case["tokens"])
    unique = 0
    for i in range(wl.n_layers):
        router = torch.randn((wl.n_experts, wl.d_model), generator=workloads._gen(wl, i, "router", device), device=device)
        router = (router * wl.weight_std).to(workloads._TORCH_DTYPE[wl.router_dtype])
        unique += int(binding.route_noalloc(cfg, hidden[i], router, None if conf is None else conf[i])[2])
    L, B, d = wl.n_layers, case["tokens"], wl.d_model
    plain = 4.0 if wl.act_dtype == workloads.F32 else 2.0
    nbytes = unique * wl.expert_bytes() + L * (wl.shared_bytes() + plain * d * (wl.n_experts + B) + 4.0 * B * d)
    per_token = wl.top_k * 3.0 * d * wl.d_ff + wl.n_shared * 3.0 * d * wl.d_ff_shared + wl.n_experts * d
    return {"bytes": nbytes, "flops": 2.0 * L * B * per_token}


def tolerance(case):
    """Indices, counts and masks exactly.  Floating outputs: float32 sums of exact products (fp32
    and bf16 weights; the SwiGLU activations keep 16 bits of mantissa or more), or products of
    weights that were rounded to binary16 once (block-int4).  About four times the difference from
    the float64 oracle: 2.7e-6 to 3.8e-6 and at most 2.1e-5 in one value, int4 3.2e-4 and 1.4e-3."""
    if case["path"] == "expand":
        return "exact"
    if workloads.CONFIGS[case["shape"]].weight_dtype == workloads.Q4B32:
        return {"rel": 1.3e-3, "max": 6e-3}
    return {"rel": 1.4e-5, "max": 9e-5}
