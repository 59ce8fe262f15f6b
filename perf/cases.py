"""The workloads that this library's performance is measured on.

A case is one step of a serving engine that applies per-token routed LoRA: route the step's tokens to adapters, group
them, and add every token's delta into the base projections of one or more layers.  `prepare` makes what the engine has
in hand before the step (activations, base projections, adapter stacks, router weights, kept workspaces, and for decode
a captured CUDA graph), `run` is the step through the package's public entry points.

Keys of a case
  call         "eager": one Python call per step of the path; "graph": the step's calls captured once and replayed, the
               way a decode loop runs; "host": activations in pinned host memory, molora_forward_host
  tokens       rows of the step (sequences x new tokens)
  adapters, rank, dtype
  router       "given" (per-request adapter known to the scheduler), "vocab" (modality by token id), "composite"
               (request adapter x modality), "gate" (linear gate), "mlp" (two-layer router)
  top          adapters kept per token (1, or 2 with softmax weights)
  projections  "layer": the seven projections of a transformer layer; "one": hidden -> hidden; "two": hidden -> hidden
               and hidden -> 3 x hidden on the same activations; "attention": q, k, v, o
  hidden, kv, inter   widths (inter = the MLP's)
  layers       layers per step; they share the activation buffers, as an engine does, and have adapters of their own
  load         "even", "zipf" (exponent 1.1) or "runs" (modality runs, geometric with mean 64): tokens per adapter
"""
import math

import torch

import paper_2603_15965_b200 as molora
from paper_2603_15965_b200.binding import molora_apply_batched_workspace_bytes, pack_proj_descs

VOCABULARY = 163840
MODALITIES = 4          # of the composite router: targets = request adapters x modalities
MLP_HIDDEN = 64


def _case(name, call, tokens, adapters, rank, router, projections, hidden, kv=0, inter=0, dtype="bf16", top=1, layers=1,
          load="even"):
    case = dict(call=call, tokens=tokens, adapters=adapters, rank=rank, router=router, projections=projections,
                hidden=hidden, kv=kv, inter=inter, dtype=dtype, top=top, layers=layers, load=load)
    return dict(case, name=name) if name else case


def listed():
    return [
        # The smallest call: two short sequences of a small fp32 model, two modalities by vocabulary range.
        _case("tiny-fp32", "eager", 256, 2, 8, "vocab", "one", 512, dtype="f32"),
        # A nearly idle server: eight sequences, one token each, one layer called from Python; latency is all there is.
        _case("decode-8", "eager", 8, 8, 16, "given", "layer", 2048, 1024, 6144, load="zipf"),
        # A full decode batch, sixteen layers replayed from a graph, requests spread over adapters by popularity.
        _case("decode-256", "graph", 256, 8, 16, "given", "layer", 2048, 1024, 6144, layers=16, load="zipf"),
        # A ragged decode batch of a wide model with large adapters, gated in every layer.
        _case("decode-wide-93", "graph", 93, 16, 64, "gate", "layer", 4096, 1024, 12288, layers=4, load="zipf"),
        # Chunked prefill beside decode: an odd number of tokens through one layer of a small model.
        _case("mixed-777", "eager", 777, 8, 16, "gate", "layer", 2048, 1024, 6144, load="zipf"),
        # Medium batch, one wide projection with rank 64, routed by the two-layer router.
        _case("mlp-1000", "eager", 1000, 8, 64, "mlp", "one", 4096),
        # Prefill of four sequences, only the query projection adapted (the most common LoRA target).
        _case("prefill-query-4096", "eager", 4096, 4, 16, "gate", "one", 2048),
        # Many small targets: 64 request adapters x 4 modalities on the attention projections.
        _case("composite-3001", "eager", 3001, 256, 16, "composite", "attention", 2048, 1024, load="runs"),
        # Weighted routing with two adapters a token.
        _case("top2-2048", "eager", 2048, 8, 16, "gate", "layer", 2048, 1024, 6144, top=2),
        # Interleaved multimodal prefill, routed by vocabulary.
        _case("multimodal-16384", "eager", 16384, 4, 32, "vocab", "two", 2048, load="runs"),
        # Prefill of a whole wide layer: the largest step.
        _case("prefill-wide-8192", "eager", 8192, 16, 64, "gate", "layer", 4096, 1024, 12288),
        # Activations that live in host memory: one layer's attention projections, copied in and out.
        _case("host-2048", "host", 2048, 8, 16, "gate", "attention", 2048, 1024),
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _widths(rng, least, most):
    hidden = rng.choice([w for w in (512, 960, 1024, 1536, 2048, 2560, 3072, 4096) if least <= w <= most])
    return hidden, hidden // rng.choice((2, 4)) // 64 * 64, hidden * 3


def draw(rng):
    """Another step of the same kinds; sizes over the whole range, token counts odd as often as not."""
    kind = rng.choice(("tiny", "decode", "decode-graph", "decode-graph", "mixed", "medium", "prefill", "prefill", "composite", "top2",
                       "multimodal", "host"))
    hidden, kv, inter = _widths(rng, 512, 4096)
    load = rng.choice(("even", "zipf", "runs"))
    if kind == "tiny":
        return _case(None, "eager", _log_int(rng, 16, 600), rng.randint(2, 4), 8, "vocab", "one", rng.choice((256, 512, 1024)),
                     dtype="f32", load=load)
    if kind == "decode":
        return _case(None, "eager", _log_int(rng, 1, 64), rng.choice((4, 8, 16)), rng.choice((16, 32, 64)), "given", "layer",
                     hidden, kv, inter, load=load)
    if kind == "decode-graph":
        return _case(None, "graph", _log_int(rng, 16, 512), rng.choice((4, 8, 16)), rng.choice((16, 32, 64)),
                     rng.choice(("given", "given", "gate")), "layer", hidden, kv, inter, layers=rng.randint(2, 8), load=load)
    if kind == "mixed":
        return _case(None, "eager", _log_int(rng, 257, 2000), rng.choice((4, 8, 16)), rng.choice((16, 32, 64)),
                     rng.choice(("gate", "vocab")), rng.choice(("layer", "attention")), hidden, kv, inter, load=load)
    if kind == "medium":
        return _case(None, "eager", _log_int(rng, 64, 2048), rng.choice((4, 8)), rng.choice((16, 32, 64)),
                     rng.choice(("mlp", "given")), "one", hidden, load=load)
    if kind == "prefill":
        return _case(None, "eager", _log_int(rng, 1024, 8192), rng.choice((4, 8, 16)), rng.choice((16, 32, 64)), "gate",
                     rng.choice(("one", "attention", "layer")), hidden, kv, inter, load=load)
    if kind == "composite":
        return _case(None, "eager", _log_int(rng, 256, 4096), MODALITIES * rng.choice((4, 16, 32, 64)), rng.choice((16, 32)),
                     "composite", rng.choice(("one", "attention")), hidden, kv, load="runs")
    if kind == "top2":
        return _case(None, "eager", _log_int(rng, 128, 4096), rng.choice((4, 8)), rng.choice((16, 32)), "gate",
                     rng.choice(("one", "layer")), hidden, kv, inter, top=2, load=load)
    if kind == "multimodal":
        return _case(None, "eager", _log_int(rng, 2048, 24576), rng.randint(2, 6), rng.choice((16, 32, 64)), "vocab", "two", hidden,
                     load="runs")
    return _case(None, "host", _log_int(rng, 128, 4096), rng.choice((4, 8)), rng.choice((16, 32)), "gate", "attention",
                 hidden, kv, load=load)


# ------------------------------------------------------------------------------------------------ shapes of a case
def _projections(case):
    """[(activation buffer, d_in, d_out)] of one layer."""
    h, kv, inter = case["hidden"], case["kv"], case["inter"]
    attention = [("attn", h, h), ("attn", h, kv), ("attn", h, kv), ("out", h, h)]
    return {"one": [("attn", h, h)],
            "two": [("attn", h, h), ("attn", h, 3 * h)],
            "attention": attention,
            "layer": attention + [("mlp", h, inter), ("mlp", h, inter), ("down", inter, h)]}[case["projections"]]


def _shares(case):
    C = case["adapters"]
    p = [1.0 / C] * C if case["load"] != "zipf" else [(c + 1) ** -1.1 for c in range(C)]
    return [v / sum(p) for v in p]


def work(case):
    """Bytes: every projection's x once (once per buffer), y read and written, the adapters that own tokens once, per layer;
    the router's input is the first projection's x.  Operations: shrink and expand of every kept adapter, and the router."""
    n, r, size = case["tokens"], case["rank"], 4 if case["dtype"] == "f32" else 2
    used = sum(1.0 - (1.0 - p) ** (n * case["top"]) for p in _shares(case))
    projs = _projections(case)
    x = sum(d for d in dict((buf, d_in) for buf, d_in, _ in projs).values())
    y = sum(d_out for _, _, d_out in projs)
    both = sum(d_in + d_out for _, d_in, d_out in projs)
    layer_bytes = size * (n * (x + 2 * y) + used * r * both)
    layer_flops = 2.0 * n * r * both * case["top"]
    h, C = case["hidden"], case["adapters"]
    route_bytes, route_flops = 4.0 * n, 0.0
    if case["router"] == "gate":
        route_bytes, route_flops = 4.0 * (n + h * C), 2.0 * n * h * C
    elif case["router"] == "mlp":
        route_bytes, route_flops = 4.0 * (n + MLP_HIDDEN * (h + C)), 2.0 * n * MLP_HIDDEN * (h + C)
    elif case["router"] in ("vocab", "composite"):
        route_bytes = 4.0 * n * (2 if case["router"] == "vocab" else 3)
    routings = case["layers"] if case["router"] in ("gate", "mlp") else 1
    return {"bytes": case["layers"] * layer_bytes + routings * route_bytes,
            "flops": case["layers"] * layer_flops + routings * route_flops}


def tolerance(case):
    """Routing, counts, offsets and permutation exactly.  Measured against 64-bit arithmetic on the same inputs: bf16 results
    are off by 1.7e-3 (2-norm) and 3.9e-3 (largest) where y is rounded once; sixteen layers into the same y, which round it
    sixteen times, by 5.4e-3 and 4.2e-2; fp32 by 4e-8 and 2e-7.  Four times that, by the number of roundings."""
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 1e-5}
    roundings = case["layers"] * case["top"]
    return {"rel": 6e-3 * roundings ** 0.5, "max": 0.016 * roundings}


# ------------------------------------------------------------------------------------------------ inputs
class _Inputs:
    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(self, shape, sigma, dtype):
        t = torch.empty(shape, dtype=dtype, device="cuda")
        return t.normal_(0.0, sigma, generator=self.gen)

    def uniform(self, n):
        return torch.rand(n, generator=self.gen, device="cuda")

    def spread(self, n, shares, load, mean_run=64):
        """Adapter of every token: drawn token by token from `shares`, or in runs that always change the adapter."""
        if load != "runs" or len(shares) == 1:
            p = torch.tensor(shares, device="cuda")
            return torch.multinomial(p, n, replacement=True, generator=self.gen)
        starts = self.uniform(n) < 1.0 / mean_run
        step = torch.where(starts, 1 + (self.uniform(n) * (len(shares) - 1)).long(), 0)
        return torch.cumsum(step, 0) % len(shares)


def _route_inputs(case, inp, x):
    """What the router reads.  Gate inputs lean towards the adapters of the drawn load: a trained gate separates its tokens."""
    n, C, h = case["tokens"], case["adapters"], case["hidden"]
    want = inp.spread(n, _shares(case), case["load"])
    state = {}
    if case["router"] == "given":
        state["r"] = want.int()
    elif case["router"] == "vocab":
        breaks = torch.tensor([VOCABULARY * m // C for m in range(C + 1)], device="cuda")
        low, high = breaks[want], breaks[want + 1]
        state["ids"] = (low + (inp.uniform(n) * (high - low)).long()).clamp_(max=VOCABULARY - 1).int()
        state["breaks"] = breaks.int()
    elif case["router"] == "composite":
        breaks = torch.tensor([VOCABULARY * m // MODALITIES for m in range(MODALITIES + 1)], device="cuda")
        modality = inp.spread(n, [1.0 / MODALITIES] * MODALITIES, "runs", 16)
        state["ids"] = (breaks[modality] + (inp.uniform(n) * (VOCABULARY // MODALITIES - 1)).long()).int()
        state["breaks"] = breaks.int()
        state["request"] = inp.spread(n, [1.0] * (C // MODALITIES), "runs", 47).int()
    elif case["router"] == "gate":
        state["G"] = inp.normal((h, C), h ** -0.5, torch.float32)
        lean = state["G"] / state["G"].norm(dim=0)
        x.copy_(x.float() + 6.0 * lean.T[want])
        if case["top"] > 1:
            x.copy_(x.float() + 4.0 * lean.T[(want + 1 + (inp.uniform(n) * (C - 1)).long()) % C])
    else:
        state["W1"] = inp.normal((h, MLP_HIDDEN), h ** -0.5, torch.float32)
        state["b1"] = inp.normal((MLP_HIDDEN,), 0.1, torch.float32)
        state["W2"] = inp.normal((MLP_HIDDEN, C), MLP_HIDDEN ** -0.5, torch.float32)
        state["b2"] = inp.normal((C,), 0.1, torch.float32)
    return state


def _draw_inputs(case, seed):
    """Activations, what the router reads, base projections and the adapter stacks of every layer."""
    inp = _Inputs(seed)
    n, C, r = case["tokens"], case["adapters"], case["rank"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    projs = _projections(case)
    x = {}
    for buf, d_in, _ in projs:
        if buf not in x:
            x[buf] = inp.normal((n, d_in), 1.0, dtype)
    state = {"case": case, "x": x}
    state.update(_route_inputs(case, inp, x["attn"]))
    y = [inp.normal((n, d_out), 1.0, dtype) for _, _, d_out in projs]
    state["y"] = y
    weights = [[(inp.normal((C, d_in, r), d_in ** -0.5, dtype), inp.normal((C, r, d_out), 0.1, dtype))
                for _, d_in, d_out in projs] for _ in range(case["layers"])]
    return state, weights


def prepare(case, seed):
    n, C = case["tokens"], case["adapters"]
    projs = _projections(case)
    state, weights = _draw_inputs(case, seed)
    x, y = state["x"], state["y"]
    if case["router"] == "mlp":
        state["image"] = molora.molora_route_mlp_prepare(x["attn"].dtype, state["W1"], C)
    if case["router"] == "gate" and case["layers"] > 1:
        # a decode loop lays the gate's weights out once
        state["image"] = molora.molora_route_gate_prepare(x["attn"].dtype, state["G"])
    if case["call"] == "host":
        host = {buf: t.cpu().pin_memory() for buf, t in x.items()}
        state["y"] = [t.cpu().pin_memory() for t in y]
        state["projs"] = [molora.HostProj(host[buf], t, A, B) for (buf, _, _), t, (A, B) in zip(projs, state["y"], weights[0])]
        room = molora.molora_forward_host_arena_bytes(state["projs"], molora.ROUTE_GATE)
        state["arena"] = torch.zeros(room, dtype=torch.uint8, device="cuda")
        return state
    state["projs"] = [[molora.ProjDesc(x[buf], t, A, B) for (buf, _, _), t, (A, B) in zip(projs, y, layer)] for layer in weights]
    if case["top"] == 1:
        packed = pack_proj_descs(state["projs"][0])
        room = molora_apply_batched_workspace_bytes(packed[0], n, C)
        state["ws"] = torch.zeros(room, dtype=torch.uint8, device="cuda") if room else None
    if case["call"] == "graph":
        kept = [t.clone() for t in y]
        _step(state)                                    # first use of every kernel before the capture
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            state["out"] = _step(state)
        for t, k in zip(y, kept):
            t.copy_(k)
    return state


# ------------------------------------------------------------------------------------------------ the step
def _route(state):
    case, x = state["case"], state["x"]["attn"]
    if case["router"] == "given":
        return state["r"]
    if case["router"] == "vocab":
        return molora.molora_route_vocab(state["ids"], state["breaks"])
    if case["router"] == "composite":
        return molora.molora_route_composite(state["ids"], state["request"], state["breaks"], case["adapters"] // MODALITIES)
    if case["router"] == "gate":
        return molora.molora_route_gate(x, state["G"], prepared=state.get("image"))
    return molora.molora_route_mlp(x, state["W1"], state["b1"], state["W2"], state["b2"], prepared=state["image"])


def _step(state):
    case = state["case"]
    if case["top"] > 1:
        logits = torch.empty(case["tokens"], case["adapters"], dtype=torch.float32, device="cuda")
        r = molora.molora_route_gate(state["x"]["attn"], state["G"], logits_out=logits)
        idx, weight = molora.molora_topk_softmax(logits, case["top"])
        molora.molora_apply_topk(state["projs"][0], idx, weight, case["adapters"])
        return {"r": r, "idx": idx, "weight": weight, "y": state["y"]}
    if case["layers"] > 1 and case["router"] == "given":
        # one routing for all layers: grouped once
        counts, offsets, perm = molora.molora_group(state["r"], case["adapters"])
        for projs in state["projs"]:
            molora.molora_apply_batched(projs, offsets, perm, ws=state["ws"])
        return {"counts": counts, "offsets": offsets, "perm": perm, "y": state["y"]}
    for projs in state["projs"]:
        r = _route(state)
        counts, offsets, perm = molora.molora_group_apply_batched(r, projs, ws=state["ws"])
    return {"r": r, "counts": counts, "offsets": offsets, "perm": perm, "y": state["y"]}


def run(state):
    """One step; y is updated in place."""
    if state["case"]["call"] == "graph":
        state["graph"].replay()
        return state["out"]
    if state["case"]["call"] == "host":
        molora.molora_forward_host(molora.ROUTE_GATE, state["projs"], state["arena"], G=state["G"])
        return {"y": state["y"]}
    return _step(state)


# ------------------------------------------------------------------------------------------------ 64 bits
def _exact_targets(state):
    """(idx [top, n], weight [top, n]) of every token in 64-bit arithmetic."""
    case, x = state["case"], state["x"]["attn"].double()
    if case["router"] == "given":
        return state["r"].long()[None], None
    if case["router"] in ("vocab", "composite"):
        r = torch.bucketize(state["ids"], state["breaks"], right=True) - 1
        if case["router"] == "composite":
            r = state["request"].long() * MODALITIES + r
        return r[None], None
    if case["router"] == "gate":
        logits = x @ state["G"].double()
    else:
        hidden = torch.nn.functional.gelu(x @ state["W1"].double() + state["b1"].double())
        logits = hidden @ state["W2"].double() + state["b2"].double()
    best, idx = logits.topk(case["top"], dim=1)
    return idx.T, torch.softmax(best, dim=1).T if case["top"] > 1 else None


def exact(case, seed):
    """What the first `run` returns, in 64 bits: y (and the routing weights); whole numbers have no rounding to measure."""
    state, weights = _draw_inputs(case, seed)
    idx, weight = _exact_targets(state)
    ys = []
    for p, (buf, _, _) in enumerate(_projections(case)):
        x, y = state["x"][buf].double(), state["y"][p].double()
        for layer in weights:
            A, B = layer[p]
            for slot in range(len(idx)):
                for c in range(case["adapters"]):
                    rows = (idx[slot] == c).nonzero()[:, 0]
                    if len(rows):
                        delta = x[rows] @ A[c].double() @ B[c].double()
                        y[rows] += delta if weight is None else weight[slot, rows, None] * delta
        ys.append(y)
    if case["call"] == "host":
        return {"y": [y.cpu() for y in ys]}
    if case["top"] > 1:
        return {"r": None, "idx": None, "weight": weight, "y": ys}
    out = {"counts": None, "offsets": None, "perm": None, "y": ys}
    return out if case["layers"] > 1 and case["router"] == "given" else dict(out, r=None)
