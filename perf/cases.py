"""Performance cases of the Agent Attention module: the calls that a program using this package makes.

A case is one pass through a public entry point of `AgentAttention`:

    forward   Eq. 6 on dense [B, heads, N, d] tensors (inference, and the forward half of a training step)
    qkv       the same on views of an interleaved [B, N, 3, heads, d] projection output
    backward  the gradients of Eq. 6 (the other half of a training step)
    host      Eq. 6 on pinned host buffers, copies included

The sizes are those of the package's own workloads (`paper_2312_08874_b200.workloads`) and generic ones around them.
"""
import math

import torch

from paper_2312_08874_b200 import AgentAttention

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _case(name, entry, batch, heads, grid_h, grid_w, head_dim, pool, dtype, bias, dwc, given_agents=False):
    c = {"entry": entry, "batch": batch, "heads": heads, "grid_h": grid_h, "grid_w": grid_w, "head_dim": head_dim,
         "pool": pool, "dtype": dtype, "bias": bias, "dwc": dwc, "given_agents": given_agents}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One image through one block of a small classifier, in fp32 and without biases: latency is everything.
        _case("fwd_deit_f32_b1", "forward", 1, 3, 14, 14, 64, 7, "f32", "none", True),
        # A batch of images through the same block in bf16: many short slabs.
        _case("fwd_deit_bf16_b128", "forward", 128, 3, 14, 14, 64, 7, "bf16", "dense", True),
        # First stage of a pyramid network: long slabs, few agents.  The benchmark's workload.
        _case("fwd_pvt_bf16_b64", "forward", 64, 1, 56, 56, 64, 7, "bf16", "dense", True),
        # Image generation: a latent grid with 256 agents and 40 channels, neither biases nor depthwise term.
        _case("fwd_sd_f16_b2", "forward", 2, 8, 64, 64, 40, 16, "f16", "none", False),
        # High-resolution grids with 256 agents.
        _case("fwd_hires128_bf16_b2", "forward", 2, 8, 128, 128, 64, 16, "bf16", "dense", True),
        _case("fwd_hires256_bf16_b2", "forward", 2, 8, 256, 256, 64, 16, "bf16", "dense", True),
        # Dense prediction at a resolution that is not the training one: an odd grid wider than 64, windows that do
        # not tile it, and biases composed from their components on every pass.
        _case("fwd_odd_grid_f16_b4", "forward", 4, 2, 75, 117, 64, 7, "f16", "composed", True),
        # The pyramid stage fed straight from a fused projection, no transposes in between.
        _case("qkv_pvt_bf16_b64", "qkv", 64, 1, 56, 56, 64, 7, "bf16", "dense", True),
        # Training: the backward passes of the classifier block, the pyramid stage and the high-resolution grid.
        _case("bwd_deit_bf16_b128", "backward", 128, 3, 14, 14, 64, 7, "bf16", "dense", True),
        _case("bwd_pvt_bf16_b64", "backward", 64, 1, 56, 56, 64, 7, "bf16", "dense", True),
        _case("bwd_hires128_bf16_b2", "backward", 2, 8, 128, 128, 64, 16, "bf16", "dense", True),
        # A caller whose tensors live in (pinned) host memory.
        _case("host_pvt_bf16_b64", "host", 64, 1, 56, 56, 64, 7, "bf16", "dense", True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: grids from 7 x 7 to 256 x 256 (odd and oblong ones included), 9 to 256 agents, the head sizes of
    the networks above, from one image to a large batch."""
    entry = rng.choice(["forward"] * 10 + ["backward"] * 7 + ["qkv"] * 2 + ["host"])
    while True:
        dtype = rng.choice(["bf16"] * 5 + ["f16"] * 3 + ["f32"] * 2)
        d = rng.choice([64] * 6 + [32, 40, 80])
        gh = _log_int(rng, 7, 256)
        gw = _log_int(rng, max(7, gh // 3), min(256, gh * 3))
        p = rng.choice([3, 4, 5, 6, 7, 7, 7, 8, 9, 12, 14, 16, 16])
        heads = rng.choice([1, 2, 3, 4, 6, 8])
        batch = _log_int(rng, 1, 128)
        bias = rng.choice(["none", "dense", "dense", "composed"])
        dwc = rng.random() < 0.75
        given = entry == "forward" and rng.random() < 0.1
        if entry == "backward" and bias == "composed":
            bias = "dense"                    # kept from the forward half
        if entry == "qkv":
            # what the entry point takes: 16-bit types; up to 64 agents with windows that tile a grid of at most
            # 64 columns, or larger multiples of 8 on grids of a multiple of 8 tokens
            dtype = "bf16" if dtype == "f32" else dtype
            d = 64 if p <= 8 else min(d, 64)
            gh, gw = (max(p, gh // p * p), max(p, min(64, gw) // p * p)) if p <= 8 else (-(-gh // 8) * 8, gw)
            bias = "dense" if bias == "composed" else bias
            if (p > 8 and (p * p % 8 or gh * gw < 128)) or gw < 8:
                continue
        n, tokens, slabs = p * p, gh * gw, batch * heads
        if p > min(gh, gw):
            continue
        total = slabs * tokens
        # 16-bit: at most the tokens and products of the largest listed case of the direction; fp32 is for small jobs
        most_tokens, most_products = {"backward": (300_000, 262_144 * 256 * 64), "host": (250_000, 250_000 * 64 * 64)}.get(
            entry, (1_048_576, 1_048_576 * 256 * 64))
        if dtype == "f32":
            most_tokens, most_products = min(most_tokens, 40_000), 40_000 * 64 * 64
        if not 147 <= total <= most_tokens or total * n * d > most_products:
            continue
        if bias != "none" and heads * n * tokens > 8 * 256 * (65_536 if entry != "backward" else 16_384):
            continue
        return _case("", entry, batch, heads, gh, gw, d, p, dtype, bias, dwc, given)


def prepare(case, seed):
    c = case
    B, h, H, W, d, p = c["batch"], c["heads"], c["grid_h"], c["grid_w"], c["head_dim"], c["pool"]
    N, n, dt = H * W, p * p, DTYPES[c["dtype"]]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(shape, std=1.0):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(std).to(dt)

    s = {"case": c, "n": n, "bias": {}, "components": {},
         "mod": AgentAttention(B, h, d, N, n, dt)}
    # activations of unit variance (normalised inputs), with the 1/sqrt(d) range of the latent network's 40 channels
    std = d ** -0.5 if d == 40 else 1.0
    if c["entry"] == "qkv":
        qkv = normal((B, N, 3, h, d), std)
        s["q"], s["k"], s["v"] = (qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3))
    else:
        s["q"], s["k"], s["v"] = (normal((B, h, N, d), std) for _ in range(3))
    if c["bias"] == "dense":
        s["bias"] = {"b1": normal((h, n, N), 0.2), "b2": normal((h, N, n), 0.2)}
    elif c["bias"] == "composed":
        s["components"] = {k: (normal((h, n, W), 0.1), normal((h, n, H), 0.1), normal((h, n, 7, 7), 0.1))
                           for k in ("b1", "b2")}
    s["filter"] = normal((h, d, 3, 3), 0.1) if c["dwc"] else None
    s["agents"] = normal((B, h, n, d), std / 4) if c["given_agents"] else None
    if c["entry"] == "backward":
        s["d_out"] = normal((B, h, N, d))
    if c["entry"] == "host":
        def pinned(t):
            return None if t is None else torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)
        if c["bias"] == "composed":       # a host caller composes once, when it loads the network
            s["bias"] = _composed(s)
            s["components"] = {}
        for k in ("q", "k", "v", "filter"):
            s[k] = pinned(s[k])
        s["bias"] = {k: pinned(t) for k, t in s["bias"].items()}
        s["out"] = torch.empty((B, h, N, d), dtype=dt, pin_memory=True)
    return s


def _composed(s):
    c = s["case"]
    return {k: s["mod"].compose_bias(col, row, blk, c["grid_h"], c["grid_w"], s["n"], transpose=k == "b2")
            for k, (col, row, blk) in s["components"].items()}


def run(state):
    s, c = state, state["case"]
    bias = _composed(s) if s["components"] else s["bias"]
    args = (c["grid_h"], c["grid_w"], s["n"])
    if c["entry"] == "forward":
        out = s["mod"].forward(s["q"], s["k"], s["v"], *args, agents=s["agents"], dwc_weight=s["filter"], **bias)
    elif c["entry"] == "qkv":
        out = s["mod"].forward_strided(s["q"], s["k"], s["v"], *args, dwc_weight=s["filter"], **bias)
    elif c["entry"] == "backward":
        return s["mod"].backward(s["q"], s["k"], s["v"], s["d_out"], *args, dwc_weight=s["filter"], **bias)
    else:
        out = s["mod"].forward_host(s["q"], s["k"], s["v"], *args, dwc_weight=s["filter"], out=s["out"], **bias)
    return {"out": out, **bias} if s["components"] else out


def work(case):
    c = case
    h, d, n = c["heads"], c["head_dim"], c["pool"] ** 2
    tokens = c["grid_h"] * c["grid_w"]
    slabs, es = c["batch"] * h, 4 if c["dtype"] == "f32" else 2
    token_bytes, bias_bytes = slabs * tokens * d, 2 * h * n * tokens
    filt = 9 * h * d if c["dwc"] else 0
    product = 2 * slabs * n * tokens * d
    if c["entry"] == "backward":
        # reads Q, K, V, dO; writes three fp32 gradients (and those of the biases and the filter)
        b = token_bytes * (4 * es + 3 * 4) + (bias_bytes * (es + 4) if c["bias"] != "none" else 0) + filt * (es + 4)
        return {"bytes": b, "flops": 11 * product + 2 * 2 * 9 * slabs * tokens * d * bool(filt)}
    b = 4 * token_bytes * es + (bias_bytes * es if c["bias"] != "none" else 0) + filt * es
    if c["given_agents"]:
        b += slabs * n * d * es
    return {"bytes": b, "flops": 4 * product + 2 * 9 * slabs * tokens * d * bool(filt)}


def tolerance(case):
    c = case
    if c["dtype"] == "f32":
        return {"rel": 5e-5 if c["entry"] == "backward" else 1e-5}
    if c["entry"] == "backward":
        # The entry point's contract: 16-bit operands on the tensor cores up to 64 agents of 64 channels, fp32
        # arithmetic on the 16-bit inputs for every other shape.
        return {"rel": 1e-2} if c["pool"] <= 8 and c["head_dim"] == 64 else {"rel": 5e-5}
    return {"rel": 1e-2 if c["dtype"] == "bf16" else 5e-3}
