"""Broadcast on tensor memory for large agent counts: ragged patches of the grid, agents that do not fill a step, references that move from step
to step, against the fp64 oracle."""
import pytest
import torch

from oracle import agent_attention_oracle as orc
from paper_2312_08874_b200 import Workload, make_inputs
from tests.parity_util import assert_close, make_module, to_dev, to_np

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H    W   d   agents dtype  bias  dwc
    (1, 2, 65, 97, 64, 72, "bf16", True, True),       # two steps, the second of eight agents; a last patch of one row, of one column
    (1, 1, 8, 784, 64, 128, "f16", True, True),       # one row of patches
    (1, 1, 787, 9, 64, 144, "bf16", True, True),      # patches nine columns wide, three steps
    (2, 1, 88, 71, 40, 200, "f16", False, True),      # four steps, channels padded
    (1, 1, 96, 64, 56, 248, "bf16", True, False),
    (3, 2, 75, 117, 64, 256, "bf16", True, True),
]


@pytest.mark.parametrize("rising", [False, True], ids=["", "rising"])
@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_n{c[5]}" for c in SHAPES])
def test_patches_and_steps(case, rising):
    B, heads, H, W, d, n, dtype, bias, dwc = case
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
    assert mod.query_status() == 0
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
