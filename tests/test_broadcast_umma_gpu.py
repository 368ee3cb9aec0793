"""Broadcast on tensor memory for large agent counts: ragged patches of the grid, runs of its tokens, agents that do not fill a step, references that move from step
to step, against the fp64 oracle."""
import pytest
import torch

from oracle import agent_attention_oracle as orc
from paper_2312_08874_b200 import AA_PATH_UNFUSED, Workload, make_inputs
from tests.parity_util import assert_close, gpu_forward, make_module, to_dev, to_np
from tests.test_stream_cut_gpu import KINDS, extreme

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H    W   d   agents dtype  bias  dwc  launches (3: aggregation, merge and broadcast; 2: register tiles)
    (1, 2, 65, 97, 64, 72, "bf16", True, True, 2),       # tokens no multiple of eight
    (1, 1, 8, 784, 64, 128, "f16", True, True, 3),       # one row of patches
    (1, 1, 787, 9, 64, 144, "bf16", True, True, 2),
    (2, 1, 88, 71, 40, 200, "f16", False, True, 3),      # four steps, channels padded, a last patch of seven columns
    (1, 1, 96, 64, 56, 248, "bf16", True, False, 3),
    (3, 2, 75, 117, 64, 256, "bf16", True, True, 2),
    # patches
    (1, 2, 72, 100, 64, 72, "bf16", True, True, 3),      # two steps, the second of eight agents; last patches of four columns
    (2, 1, 70, 112, 64, 144, "f16", True, True, 3),      # three steps; last patches of six rows
    (1, 1, 123, 104, 64, 256, "bf16", True, True, 3),    # both, a long axis
    # runs of 128 tokens
    (2, 2, 1, 3080, 64, 256, "bf16", True, True, 3),     # one row, a last run of eight tokens
    (1, 2, 3080, 1, 64, 200, "f16", True, True, 3),      # one column
    (1, 1, 2, 4100, 64, 144, "bf16", True, True, 3),     # two rows, a long axis
    (1, 1, 788, 10, 64, 144, "bf16", True, True, 3),     # more rows than one in a run
    (2, 1, 1048, 3, 56, 248, "bf16", True, True, 3),
    (2, 1, 3, 2736, 40, 256, "f16", False, True, 3),     # a run in the middle of a row, channels padded
    (1, 2, 66, 100, 64, 72, "bf16", True, False, 3),     # no window
]


@pytest.mark.parametrize("rising", [False, True], ids=["", "rising"])
@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_n{c[5]}" for c in SHAPES])
def test_patches_and_steps(case, rising):
    B, heads, H, W, d, n, dtype, bias, dwc, launches = case
    w = Workload("patch", B, heads, H, W, d, 9, dtype, False, dwc, 1.0, seed=300 + H * W + n)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    g = torch.Generator().manual_seed(n)
    t = inp["q"].dtype
    agents = torch.randn((B, heads, n, d), generator=g).to(t)
    b1 = b2 = None
    if bias:
        b1 = (torch.randn((heads, n, H * W), generator=g) * 0.5).to(t)
        b2 = torch.randn((heads, H * W, n), generator=g) * 0.5
        if rising:
            b2 += 8.0 * (torch.arange(n) // 64)                # every step of 64 agents outweighs those before
        b2 = b2.to(t)
    elif rising:
        agents[:, :, 64:] *= 4                                 # logits of the later steps grow
    mod = make_module(w, max_agents=n)
    out = torch.full_like(to_dev(inp["q"]), float("nan"))
    mod.forward(to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"]), H, W, n, agents=agents.cuda(), b1=to_dev(b1), b2=to_dev(b2),
                dwc_weight=to_dev(inp["dwc"]), out=out)
    torch.cuda.synchronize()
    assert mod.query_status() == 0 and mod.last_launch_count() == launches
    for b, h in {(0, 0), (B - 1, heads - 1)}:
        one = lambda x: None if x is None else to_np(x[b:b + 1, h:h + 1])
        hd = lambda x: None if x is None else to_np(x[h:h + 1])
        ref = orc.forward(one(inp["q"]), one(inp["k"]), one(inp["v"]), H, W, agents=one(agents), b1=hd(b1), b2=hd(b2), dwc_weight=hd(inp["dwc"]), threads=orc.max_threads())
        assert_close(out[b:b + 1, h:h + 1], ref, dtype, f"{case} slab {(b, h)}")


@pytest.mark.parametrize("n,dtype", [(256, "bf16"), (128, "bf16"), (256, "f16")])
def test_partial_states_of_the_aggregation_hold_the_weights_as_rounded(n, dtype):
    """With values of one, a row of a partial state's sums of products and its sum of weights are the same numbers added up: 8 tiles of 64 tokens a
    block, so at most 19 fp32 roundings of one and 16 of the other, 35 x 2^-23 = 4.2e-6 apart.  (Weights before rounding: 2^-9 / sqrt(512) in bf16.)"""
    w = Workload("states", 4, 8, 32, 64, 64, 16, dtype, True, False, 1.0, seed=77)
    inp = make_inputs(w, bias_std=0.5)
    mod = make_module(w, max_agents=n)
    a, k = (torch.randn((4, 8, m, 64), generator=torch.Generator().manual_seed(m)).to(inp["q"].dtype).cuda() for m in (n, 2048))
    ws = torch.zeros(mod.workspace_bytes(1, 2048, n), dtype=torch.uint8, device="cuda")
    mod.aggregate(a, k, torch.ones_like(k), b1=to_dev(inp["b1"][:, :n].contiguous()), workspace=ws)
    assert mod.last_launch_count() == 2 and mod.query_status() == 0
    rows = (n + 127) // 128 * 128
    state = ws[2 * a.numel() * 2:].view(torch.float32)[:rows * 66]                # the first block's: maxima, sums, products [rows][64]
    sums, products = state[rows:2 * rows][:n], state[2 * rows:].view(rows, 64)[:n]
    assert float(sums.min()) > 0
    assert float((products / sums[:, None] - 1).abs().max()) <= 4.2e-6


@pytest.mark.parametrize("H,W", [(1, 16384), (16384, 1), (2, 8192), (1640, 10)])
def test_thin_grids_take_as_long_as_square_ones(H, W):
    """The same tokens in a row, in a column or in a square are the same work.  (Patches of 8 x 16 tokens alone took 2.4 to 8 times as long.)"""
    def best(H, W):
        w = Workload("thin", 1, 16, H, W, 64, 1, "bf16", False, True, 1.0, seed=5)
        g = torch.Generator(device="cuda")
        q, k, v = (torch.randn((1, 16, H * W, 64), generator=g, device="cuda").bfloat16() for _ in range(3))
        a, f = torch.randn((1, 16, 256, 64), device="cuda").bfloat16(), torch.randn((16, 64, 3, 3), device="cuda").bfloat16()
        mod, times = make_module(w, max_agents=256), []
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(8):
                mod.forward(q, k, v, H, W, 256, agents=a, dwc_weight=f)
            t1.record()
            t1.synchronize()
            times.append(t0.elapsed_time(t1))
        return min(times)
    assert best(H, W) <= 1.6 * best(128, 128)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("case", [(2, 1, 72, 100, 64, 12), (1, 2, 656, 12, 64, 12), (1, 1, 96, 96, 40, 16)], ids=["patches", "runs", "d40"])
def test_extreme_numbers_reach_as_far_as_on_register_tiles(case, kind):
    """Rows of biases that remove everything, finite biases beyond +-30000, an infinite value under a positive filter, NaN: what is not finite is the
    same, and what is finite as close as the two kernels are otherwise."""
    B, heads, H, W, d, pool = case
    w = Workload("extreme", B, heads, H, W, d, pool, "bf16", True, True, 1.0, seed=130 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    extreme(inp, kind, "bf16", W)
    mod = make_module(w)
    out, tiles = gpu_forward(mod, w, inp), gpu_forward(make_module(w, path=AA_PATH_UNFUSED), w, inp)
    assert mod.last_launch_count() == 4
    assert torch.equal(out.isnan(), tiles.isnan()) and torch.equal(out.isinf(), tiles.isinf())
    both = out.isfinite()
    assert not both.any() or float((out[both].float() - tiles[both].float()).abs().max()) <= 2e-2


@pytest.mark.parametrize("case", [(2, 2, 656, 12), (3, 1, 656, 12), (1, 2, 14, 568), (2, 1, 64, 128), (2, 2, 64, 128)],
                         ids=["runs", "runs_one_head", "runs_one_entry", "patches_one_head", "patches"])
def test_token_major_views_run_on_tensor_memory_as_dense_tensors_do(case):
    B, heads, H, W = case
    w = Workload("views", B, heads, H, W, 64, 12, "bf16", True, True, 1.0, seed=170 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    dense = gpu_forward(mod, w, inp)
    qkv = torch.stack([to_dev(inp[x]).permute(0, 2, 1, 3) for x in "qkv"], dim=2).contiguous()          # [B, N, 3, heads, d]
    out = mod.forward_strided(*(qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3)), H, W, w.agents, b1=to_dev(inp["b1"]), b2=to_dev(inp["b2"]),
                              dwc_weight=to_dev(inp["dwc"]))
    assert mod.last_launch_count() == 4 and mod.query_status() == 0
    assert torch.equal(out, dense)
