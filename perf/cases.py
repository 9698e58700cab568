"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one of seven kinds of call sequence on one MoE layer shape (or a stack of equal layers):

  step       one decode token of a layer: slicemoe_route_topk, then slicemoe_layer with the list it wrote
             (T tokens at once when the case says so: a small batch of sequences)
  routed     the same in one call: slicemoe_layer_routed
  host       the same with pinned host buffers in and out: slicemoe_decode_step_host
  stack      one decode token through all layers of a stack, captured once as a CUDA graph and replayed
  cached     one decode token through a few layers with the host slice cache in the loop: the list goes to the host,
             the cache decides the precision of every expert, the precision list goes back, the layer runs
  prefill    a prompt of T tokens: slicemoe_route_topk, then slicemoe_prefill_layer
  pack       preparation of one expert: slicemoe_pack of its gate, up and down matrices

Shapes are those of the two models whose layers the library's benchmark is quoted on (hidden 2048, experts of width
1408, top-6 of 64 with two shared experts of 1408, or top-4 of 60 with one gated shared expert of 5632), the tiny
layer of its tests, and generic ones.  Weights are N(0, 0.02), activations N(0, 1) in bf16; router logits are N(0, 1)
for single decode steps and log(Zipf popularity) + Gumbel noise where many tokens are routed.
"""
import torch

from paper_2512_12990_b200 import binding as B

LAYER_A = dict(hidden=2048, inter=1408, experts=64, top_k=6, group=128, shared=2, shared_inter=1408, gated=False)
LAYER_B = dict(hidden=2048, inter=1408, experts=60, top_k=4, group=128, shared=1, shared_inter=5632, gated=True)
TINY = dict(hidden=256, inter=128, experts=8, top_k=2, group=64, shared=0, shared_inter=0, gated=False)


def _case(name, kind, layer, **more):
    c = dict(kind=kind, b_high=8, b_low=4, tokens=1, layers=1, renorm=False, rank_high=layer["top_k"] // 2, zipf=0.0)
    c.update(layer)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a layer whose kernels are all latency
        _case("tiny layer, one token", "step", TINY, rank_high=1),
        # the headline use: one token of a layer, the three best experts from both slices, three from the MSB slice
        _case("decode step, top-6 + 2 shared", "step", LAYER_A),
        # the other model's layer, routed inside the kernel, four experts and a wide gated shared one
        _case("decode step, routed, gated shared", "routed", LAYER_B),
        # a serving loop that keeps activations on the host: pinned buffers in, pinned buffer out
        _case("decode step, host buffers", "host", LAYER_A),
        # a whole token: 26 layers in one CUDA graph, which is how a latency-bound decode is run
        _case("decode token, 26-layer graph", "stack", LAYER_A, layers=26),
        # the method's own decode loop: the slice cache on the host decides every expert's precision
        _case("decode token, cache in the loop", "cached", LAYER_A, layers=4, zipf=1.1),
        # eight sequences decoded together
        _case("decode batch of 8", "step", LAYER_A, tokens=8, zipf=1.1),
        # narrow slices, small groups, a hidden width that is no multiple of the 2048-column chunk, no shared expert
        _case("decode step, 6-bit codes, group 32", "step",
              dict(hidden=2688, inter=896, experts=24, top_k=5, group=32, shared=0, shared_inter=0, gated=False),
              b_high=6, b_low=3),
        # a short question: every expert is visited by a handful of tokens
        _case("prefill of 77 tokens", "prefill", LAYER_A, tokens=77, zipf=1.0),
        # the benchmark's prompt
        _case("prefill of 2048 tokens", "prefill", LAYER_B, tokens=2048, zipf=1.0, renorm=True),
        # a long document
        _case("prefill of 8192 tokens", "prefill", LAYER_A, tokens=8192, zipf=1.0),
        # offline preparation, one expert at a time
        _case("pack one expert", "pack", LAYER_A),
    ]


def _log_uniform(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def _multiple(v, m, lo):
    return max(lo, int(round(v / m)) * m)


def draw(rng):
    kind = rng.choice(["step", "step", "routed", "host", "batch", "prefill", "prefill", "pack"])
    while True:
        layer = dict(
            hidden=_multiple(_log_uniform(rng, 256, 4096), 128, 256), inter=_multiple(_log_uniform(rng, 128, 2048), 128, 128),
            experts=int(_log_uniform(rng, 8, 129)), top_k=rng.randint(1, 8), group=rng.choice([128, 128, 64, 32]),
            shared=rng.choice([0, 1, 2]), shared_inter=0, gated=False)
        if layer["shared"]:
            layer["shared_inter"] = _multiple(_log_uniform(rng, 128, 4096), 128, 128)
            layer["gated"] = rng.random() < 0.5
        wide = layer["top_k"] * layer["inter"] + layer["shared"] * layer["shared_inter"]
        weights = layer["experts"] * layer["hidden"] * layer["inter"]
        # the single-token kernel's limit on the widths of a token's experts; no more weights than the largest listed layer
        if wide <= 12288 and weights <= 64 * 2048 * 1408:
            break
    b_high, b_low = rng.choice([(8, 4), (8, 4), (8, 4), (6, 3), (4, 2)])
    more = dict(b_high=b_high, b_low=b_low, rank_high=rng.randint(0, layer["top_k"]), renorm=rng.random() < 0.3)
    if kind == "batch":
        kind = "step"
        more.update(tokens=rng.randint(2, 16), zipf=1.1)
    elif kind == "prefill":
        largest = 8192 * 2048 * 8 * 1408  # token-weights of the largest listed case
        most = min(8192, largest // (layer["hidden"] * wide))
        more.update(tokens=int(_log_uniform(rng, 16, most + 1)), zipf=1.0)
    return _case(None, kind, layer, **more)


# ---- inputs --------------------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _weights(g, n, k):
    return torch.randn((n, k), generator=g, device="cuda").mul_(0.02)


def _expert(c, g, inter):
    out = {}
    for name, n, k in (("gate", inter, c["hidden"]), ("up", inter, c["hidden"]), ("down", c["hidden"], inter)):
        out[name] = B.slicemoe_pack(_weights(g, n, k), c["group"], c["b_high"], c["b_low"])
    return out


def _logits(c, g, tokens):
    if not c["zipf"]:
        return torch.randn((tokens, c["experts"]), generator=g, device="cuda")
    p = torch.arange(1, c["experts"] + 1, device="cuda", dtype=torch.float32) ** -c["zipf"]
    p = (p / p.sum())[torch.randperm(c["experts"], generator=g, device="cuda")]
    u = torch.rand((tokens, c["experts"]), generator=g, device="cuda").clamp_(1e-7, 1 - 1e-7)
    return p.log() - (-u.log()).log()


def _one_layer(c, g):
    experts = [_expert(c, g, c["inter"]) for _ in range(c["experts"])]
    shared = [_expert(c, g, c["shared_inter"]) for _ in range(c["shared"])]
    return dict(
        keep=(experts, shared), experts=B.expert_table(experts), shared=B.expert_table(shared) if shared else None,
        gate=torch.randn(c["hidden"], generator=g, device="cuda").mul_(0.02) if c["gated"] else None,
        x=torch.randn((c["tokens"], c["hidden"]), generator=g, device="cuda").to(torch.bfloat16),
        logits=_logits(c, g, c["tokens"]))


def prepare(case, seed):
    c, g = case, _generator(seed)
    if c["kind"] == "pack":
        i, h = c["inter"], c["hidden"]
        return dict(c=c, w=[_weights(g, i, h), _weights(g, i, h), _weights(g, h, i)])
    s = dict(c=c, layers=[_one_layer(c, g) for _ in range(c["layers"])])
    s["shape"] = B.make_shape(c["hidden"], c["inter"], c["experts"], c["top_k"], c["group"], c["shared"], c["shared_inter"],
                              c["gated"], c["b_high"], c["b_low"])
    if c["kind"] == "prefill":
        s["ws"] = B.new_prefill_workspace(s["shape"], c["tokens"])
        # half of the experts run from both slices, half from the MSB slice alone
        s["prec"] = (torch.randperm(c["experts"], generator=g, device="cuda") % 2).to(torch.uint8)
        return s
    s["ws"] = B.new_workspace(s["shape"])
    if c["kind"] == "host":
        L = s["layers"][0]
        s["x"], s["logits"] = L["x"][0].cpu().pin_memory(), L["logits"][0].cpu().pin_memory()
        s["y"] = torch.empty(c["hidden"], dtype=torch.float32).pin_memory()
    elif c["kind"] == "cached":
        msb, lsb = (_expert_bytes(c, c["inter"], False), c["hidden"] * c["inter"] * 3 // 2)
        s["cache"] = B.Dbsc(int(0.3 * c["layers"] * c["experts"] * (msb + lsb)), msb, lsb)
        s["prec"] = torch.empty((c["layers"], c["top_k"]), dtype=torch.uint8).pin_memory()
        s["step"] = 0
    elif c["kind"] == "stack":
        s["y"] = torch.empty((c["layers"], c["hidden"]), device="cuda")
        _stack_token(s)  # before the capture, as for any CUDA graph
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["lists"] = _stack_token(s)
    return s


# ---- one pass ------------------------------------------------------------------------------------------------
def _route(c, L):
    return B.slicemoe_route_topk(L["logits"], c["top_k"], renorm=c["renorm"], rank_high=c["rank_high"])


def _stack_token(s):
    lists = []
    for i, L in enumerate(s["layers"]):
        ids, w, prec = _route(s["c"], L)
        B.slicemoe_layer(s["shape"], L["experts"], L["shared"], L["gate"], L["x"], ids, prec, w, s["ws"], y=s["y"][i:i + 1])
        lists.append((ids, w))
    return lists


def run(state):
    s, c = state, state["c"]
    kind = c["kind"]
    if kind == "pack":
        out = [B.slicemoe_pack(w, c["group"], c["b_high"], c["b_low"]) for w in s["w"]]
        return [(m.msb, m.lsb, m.scale, m.zp) for m in out]
    L = s["layers"][0]
    if kind == "step":
        ids, w, prec = _route(c, L)
        y = B.slicemoe_layer(s["shape"], L["experts"], L["shared"], L["gate"], L["x"], ids, prec, w, s["ws"])
        return y, ids, w, prec
    if kind == "routed":
        return B.slicemoe_layer_routed(s["shape"], L["experts"], L["shared"], L["gate"], L["x"], L["logits"], s["ws"],
                                       renorm=c["renorm"], rank_high=c["rank_high"])
    if kind == "host":
        return B.slicemoe_decode_step_host(s["shape"], L["experts"], L["shared"], L["gate"], s["x"], s["logits"], s["y"],
                                           s["ws"], renorm=c["renorm"], rank_high=c["rank_high"])
    if kind == "stack":
        s["graph"].replay()
        return s["y"], s["lists"]
    if kind == "cached":
        ys = []
        for i, L in enumerate(s["layers"]):
            ids, w, request = _route(c, L)
            s["prec"][i] = torch.from_numpy(s["cache"].assign(s["step"], i, ids[0].cpu().numpy(), request[0].cpu().numpy()))
            prec = s["prec"][i:i + 1].to("cuda", non_blocking=True)
            ys.append(B.slicemoe_layer(s["shape"], L["experts"], L["shared"], L["gate"], L["x"], ids, prec, w, s["ws"]))
        s["step"] += 1
        return ys, s["prec"]
    ids, w, _ = B.slicemoe_route_topk(L["logits"], c["top_k"], renorm=c["renorm"], want_prec=False)
    y, status = B.slicemoe_prefill_layer(s["shape"], L["experts"], L["shared"], L["gate"], L["x"], ids, w, s["prec"], s["ws"])
    return y, ids, w, status


# ---- what a pass cannot do without --------------------------------------------------------------------------
def _expert_bytes(c, inter, both):
    """Planes, scales and zero-points of one expert's three matrices, from both slices or from the MSB slice alone."""
    n = 3 * c["hidden"] * inter
    return (n if both else n // 2) + 3 * n // c["group"]


def work(case):
    c = case
    h, k, T = c["hidden"], c["top_k"], c["tokens"]
    if c["kind"] == "pack":
        n = 3 * h * c["inter"]
        return {"bytes": 4 * n + n + 3 * n // c["group"], "flops": 0}
    if c["kind"] == "prefill":
        high = 0.5
    else:
        high = c["rank_high"] / k
    # experts that T tokens are expected to name, were all equally likely (k for one token; fewer where some are popular)
    used = k if T == 1 else c["experts"] * (1 - (1 - k / c["experts"]) ** T)
    bytes_ = used * (high * _expert_bytes(c, c["inter"], True) + (1 - high) * _expert_bytes(c, c["inter"], False))
    bytes_ += c["shared"] * _expert_bytes(c, c["shared_inter"], True)
    bytes_ += T * (2 * h + 4 * h + 4 * c["experts"])
    flops = 2 * T * 3 * h * (k * c["inter"] + c["shared"] * c["shared_inter"])
    return {"bytes": int(c["layers"] * bytes_), "flops": c["layers"] * flops}


def tolerance(case):
    if case["kind"] == "pack":
        return "exact"
    if case["kind"] == "prefill":
        # h crosses the two projections as fp16 (11 significant bits), everything else is wider
        return {"rel": 5e-4, "max": 5e-3}
    return {"rel": 1e-5, "max": 1e-4}
