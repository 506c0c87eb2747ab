"""The work that users of this library have it do, as cases that can be timed and compared.

A case names a public entry point, the sizes of one MoE layer, and the options in use:

  entry   "layer"  moe_layer: routing build -> analytical plan -> fused GEMM2 + combine on activations that are
                   already in routed order (the paper's operator; the loop object binding.LayerCall);
          "moe"    moe_post_router_layer: routing build -> gather + GEMM1 + gated activation -> GEMM2 + combine,
                   what a model's forward pass calls after its router;
          "host"   moe_layer_host: the layer from pinned host buffers, result back in host memory;
          "steps"  moe_build_routing, plan_partition, moe_gemm2_combine as three calls, with the stream
                   synchronised in between, as the paper's integration describes it.
  counts  "host" (the plan is made from this batch's routed-tile counts) or "device" (the counts stay on the
          device, the call never waits; "layer" and "moe" only).
  partition  "dynamic" (compute CTAs help with the communication work that is left) or "static" (the paper's
          fixed partition of the SMs).
  skew    0: all experts equally popular; s > 0: expert popularity follows Zipf(s), softened by per-token noise
          so that the busiest expert gets about 2.5 to 3 times the mean load.

Sizes are the repository's four configurations (tiny, Granite-3-MoE-, Qwen1.5-MoE- and DeepSeek-V2-Lite-shaped),
with the number of tokens from one (a single stream decoding) over serving batches and ragged prefill chunks to
a 16384-token prefill, one to four destination buffers and one or two tensor-parallel shards.  The tile family
is the one the library's own dispatch (moe_select_tile) picks.  Inputs are bf16 with fp32 routing weights, the
only types the path takes.
"""

import torch

from paper_2609_07536_b200 import binding as B

#: name -> (H, I, routed experts, experts per token, shared experts, Zipf exponent, noise that softens it)
FAMILIES = {
    "tiny": (256, 128, 8, 2, 0, 1.0, 3.2),
    "granite": (1536, 512, 40, 8, 0, 1.0, 3.2),
    "qwen": (2048, 1408, 60, 4, 0, 1.0, 5.8),
    "dsv2lite": (2048, 1408, 64, 6, 2, 1.2, 4.9),
}


def _case(entry, family, T, TP=1, EP=1, L=1, skewed=True, counts="host", partition="dynamic", name=None):
    H, I, E, k, shared, s, noise = FAMILIES[family]
    c = dict(entry=entry, T=T, H=H, I=I, E=E, k=k, shared=shared, TP=TP, EP=EP, L=L,
             skew=s if skewed else 0.0, noise=noise if skewed else 1.0, counts=counts, partition=partition)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest layer of the repository's configurations: launches and host work are all there is
        _case("layer", "tiny", 256, TP=1, EP=2, skewed=False, name="tiny_256"),
        # one stream decoding, whole layer: one token's experts are read, everything else is latency
        _case("moe", "dsv2lite", 1, skewed=False, counts="device", name="moe_decode_1"),
        # a small serving batch, the operator as the decode benchmark runs it (host counts, TP = EP = 2)
        _case("layer", "dsv2lite", 16, TP=2, EP=2, L=2, name="decode_16"),
        # a serving batch, whole layer, asynchronous (counts stay on the device)
        _case("moe", "qwen", 48, counts="device", name="moe_decode_48"),
        # a large serving batch: all experts' weights are read for a few dozen rows each
        _case("layer", "dsv2lite", 256, TP=2, EP=2, L=2, name="decode_256"),
        # a ragged prefill chunk, whole layer, host counts
        _case("moe", "granite", 1003, name="moe_chunk_1003"),
        # the paper's three-call integration with its static partition of the SMs, several destination ranks
        _case("steps", "dsv2lite", 2048, TP=2, EP=4, L=2, skewed=False, partition="static", name="steps_static_2048"),
        # a layer called with activations in host memory
        _case("host", "qwen", 512, name="host_512"),
        # the repository's three model-shaped configurations
        _case("layer", "granite", 4096, TP=2, EP=2, name="granite_4096"),
        _case("layer", "qwen", 8192, TP=2, EP=2, name="qwen_8192"),
        _case("layer", "dsv2lite", 16384, TP=2, EP=2, L=2, name="dsv2lite_16384"),
        # the largest: whole layer of a 16384-token prefill
        _case("moe", "dsv2lite", 16384, name="moe_prefill_16384"),
    ]


def _log_int(rng, lo, hi):
    """Integer in [lo, hi], even over its logarithm; odd and ragged values come as they fall."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    entry = rng.choice(["layer", "layer", "layer", "moe", "moe", "moe", "host", "steps"])
    family = rng.choice(["tiny", "granite", "qwen", "dsv2lite", "granite", "qwen", "dsv2lite"])
    most = {"layer": 16384, "moe": 16384, "host": 1024, "steps": 4096}[entry]
    T = _log_int(rng, 1, min(most, 4096) if family == "tiny" else most)
    counts = rng.choice(["host", "host", "device"]) if entry in ("layer", "moe") else "host"
    partition = rng.choice(["dynamic", "static"]) if entry == "steps" else "dynamic"
    return _case(entry, family, T, TP=rng.choice([1, 2]), EP=rng.choice([1, 2, 4]), L=rng.choice([1, 2]),
                 skewed=rng.random() < 0.7, counts=counts, partition=partition)


# ----------------------------------------------------------------------------- inputs

_handles = {}


def _handle():
    """One handle per process, as a serving program keeps it."""
    dev = torch.cuda.current_device()
    if dev not in _handles:
        _handles[dev] = B.moe_create(dev)
    return _handles[dev]


def _normal(gen, shape, std):
    x = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    return x.normal_(0.0, std, generator=gen)


def _route(c, gen):
    """Top-k of noisy logits and the softmax of the selected ones; shared experts with weight one behind them."""
    T, E, k = c["T"], c["E"], c["k"]
    if c["skew"] > 0:
        rank = torch.randperm(E, generator=gen, device="cuda") + 1
        logits = c["noise"] * torch.randn((T, E), generator=gen, device="cuda") - c["skew"] * torch.log(rank.float())
    else:
        logits = torch.rand((T, E), generator=gen, device="cuda")
    top, idx = torch.topk(logits, k, dim=1)
    w = torch.softmax(top, dim=1)
    if c["shared"]:
        more = torch.arange(E, E + c["shared"], device="cuda").expand(T, -1)
        idx = torch.cat([idx, more], dim=1)
        w = torch.cat([w, torch.ones((T, c["shared"]), device="cuda")], dim=1)
    return idx.to(torch.int32).contiguous(), w.to(torch.float32).contiguous()


def _written(ws):
    """The rows of every destination buffer that belong to one of its tokens (the rest is never written)."""
    s = ws.shape
    blk = -(-s.T // s.EP)
    own = [max(0, min(blk, s.T - d * blk)) for d in range(s.EP)]
    return [o[:n] for o, n in zip(ws.out, own) if n > 0]


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    h = _handle()
    k_tot, E_tot = c["k"] + c["shared"], c["E"] + c["shared"]
    R = c["T"] * k_tot
    shape = B.make_shape(c["T"], c["H"], c["I"], E_tot, k_tot, c["TP"], c["EP"], c["L"])
    tile_m, tile_n = B.moe_select_tile(h, shape)
    idx, wt = _route(c, gen)
    st = dict(entry=c["entry"], h=h, shape=shape, idx=idx, wt=wt, tile=(tile_m, tile_n))
    st["W2"] = _normal(gen, (E_tot, c["H"], c["I"]), 0.02)
    if c["entry"] == "host":
        x = _normal(gen, (R, c["I"]), 0.02)
        st["x_host"] = x.cpu().pin_memory()
        st["idx_host"], st["wt_host"] = idx.cpu().pin_memory(), wt.cpu().pin_memory()
        st["arena_bytes"] = B.moe_host_arena_bytes(shape, tile_m, tile_n)
        st["arena"] = torch.empty(st["arena_bytes"], dtype=torch.uint8, device="cuda")
        st["tile_counts"] = torch.zeros(E_tot + 1, dtype=torch.int32).pin_memory()
        st["out_host"] = torch.zeros((c["T"], c["H"]), dtype=torch.bfloat16).pin_memory()
        return st
    ws = B.alloc_workspace(shape, tile_m, tile_n, device=idx.device)
    st["ws"] = ws
    st["result"] = _written(ws)
    if c["counts"] == "host":
        st["result"] = st["result"] + [ws.tile_counts]
    st["on_device"] = c["counts"] == "device"
    if c["entry"] == "moe":
        st["hidden"] = _normal(gen, (c["T"], c["H"]), 1.0)
        st["W1"] = _normal(gen, (E_tot, 2, c["I"], c["H"]), 0.02)
        st["h_routed"] = torch.empty(B.moe_gemm1_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
        st["x_routed"] = torch.empty((R, c["I"]), dtype=torch.bfloat16, device="cuda")
    else:
        st["x"] = _normal(gen, (R, c["I"]), 0.02)
    if c["entry"] == "layer":
        st["call"] = B.LayerCall(h, st["x"], st["W2"], idx, wt, ws, counts_on_device=st["on_device"])
    if c["entry"] == "steps":
        st["occ"], st["limits"], st["rho"] = B.moe_query_occupancy(h, tile_m, tile_n)
        st["limits"].drain_help = 1 if c["partition"] == "dynamic" else 0
    return st


def run(state):
    s, h = state, state["h"]
    if s["entry"] == "layer":
        s["call"]()
    elif s["entry"] == "moe":
        B.moe_post_router_layer(h, s["hidden"], s["W1"], s["W2"], s["idx"], s["wt"], s["ws"], s["h_routed"],
                                s["x_routed"], counts_on_device=s["on_device"])
    elif s["entry"] == "host":
        B.moe_layer_host(h, s["x_host"], s["idx_host"], s["wt_host"], s["W2"], s["shape"], *s["tile"], None,
                         s["arena"], s["arena_bytes"], s["tile_counts"], s["out_host"])
        return [s["out_host"], s["tile_counts"]]
    else:
        ws, shape = s["ws"], s["shape"]
        B.moe_build_routing(h, s["idx"], shape, ws.tile_m, ws.routing, ws.tile_counts, ws.status)
        torch.cuda.current_stream().synchronize()          # the plan is made from the counts
        tiles = ws.tile_counts.tolist()
        plan = B.plan_partition(tiles[:shape.E_tot], s["occ"], s["limits"], shape, s["rho"])
        B.moe_gemm2_combine(h, s["x"], s["W2"], s["idx"], s["wt"], shape, s["occ"], ws.routing, tiles[shape.E_tot],
                            plan, ws.out, ws.y_ws, ws.flags_ws, ws.status)
    return s["result"]


# ----------------------------------------------------------------------------- what a pass needs

def work(case):
    """Bytes: activations, routing, the weights of the experts that some token chose (expected number, experts
    equally popular) and the result, each once.  Flops: the routed rows' products, without padding."""
    c = case
    k_tot = c["k"] + c["shared"]
    R = c["T"] * k_tot
    used = c["E"] * (1.0 - (1.0 - c["k"] / c["E"]) ** c["T"]) + c["shared"]
    w2 = used * c["H"] * c["I"] * 2
    n = w2 + R * 8 + c["T"] * c["H"] * 2
    flops = 2.0 * R * c["H"] * c["I"]
    if c["entry"] == "moe":
        n += 2 * w2 + c["T"] * c["H"] * 2                   # gate and up projections, hidden states
        flops *= 3.0
    else:
        n += R * c["I"] * 2                                 # activations in routed order
    return {"bytes": float(n), "flops": flops}


def tolerance(case):
    """bf16 inputs, intermediates and results with fp32 accumulation: a few times 2^-9 in the 2-norm."""
    return {"rel": 1e-2, "max": 0.1}
