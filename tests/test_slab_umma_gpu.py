"""Whole forward pass of a short slab in one block on tensor memory, at the edges of its halves and layouts, against the fp64 oracle."""
import pytest
import torch

from paper_2312_08874_b200 import AA_PATH_UNFUSED, Workload, make_inputs
from tests.parity_util import assert_close, gpu_forward, make_module, oracle_forward, to_dev
from tests.test_masks_gpu import masked
from tests.test_stream_cut_gpu import KINDS, extreme

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W   d   pool dtype  bias  dwc
    (1, 2, 33, 1, 64, 1, "f16", True, True),          # one agent; tokens in a column; a second half of one token
    (3, 1, 7, 7, 56, 7, "bf16", True, True),          # as many agents as tokens, channels padded, odd bias rows
    (2, 3, 11, 11, 64, 5, "bf16", True, True),        # odd tokens and agents: biases that start in the middle of a vector
    (130, 3, 14, 14, 64, 7, "f16", True, True),       # more slabs than resident blocks
    (16, 1, 16, 16, 64, 7, "bf16", False, True),      # the largest halves
    (6, 3, 3, 85, 64, 3, "bf16", True, True),         # 255 tokens, wide windows
    (9, 2, 8, 24, 64, 8, "f16", True, False),         # 64 agents
    (40, 2, 10, 10, 40, 5, "bf16", True, True),
    (200, 3, 9, 11, 32, 4, "f16", True, True),
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}" for c in SHAPES])
def test_short_slabs_match_oracle(case):
    B, heads, H, W, d, pool, dtype, bias, dwc = case
    w = Workload("slab", B, heads, H, W, d, pool, dtype, bias, dwc, 1.0, seed=200 + H * W + d)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    out = gpu_forward(mod, w, inp)
    assert mod.last_launch_count() == 1
    slabs = [(0, 0), (B - 1, heads - 1)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert_close(out[b:b + 1, h:h + 1], ref, dtype, f"{case} slab {(b, h)}")
    assert torch.equal(out, gpu_forward(mod, w, inp)), "bit-reproducible"
    views = [to_dev(inp[x]).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for x in ("q", "k", "v")]
    if W >= 8 and d == 64 and H % pool == 0 and W % pool == 0 and W <= 64:         # what the strided entry point takes
        assert torch.equal(out, mod.forward_strided(*views, H, W, w.agents, b1=to_dev(inp["b1"]), b2=to_dev(inp["b2"]), dwc_weight=to_dev(inp["dwc"])))


# 72 slabs of 196 tokens; 160 of 100 tokens and 40 channels; 16 of 121 tokens, odd rows of biases
OTHERS = [(24, 3, 14, 14, 64, 7, "bf16", 0), (80, 2, 10, 10, 40, 5, "f16", 0), (16, 1, 11, 11, 64, 7, "bf16", 0)]
IDS = ["196x64", "100x40", "121x64"]


@pytest.mark.parametrize("value", ["inf", "lowest"])
@pytest.mark.parametrize("case", OTHERS, ids=IDS)
def test_masked_short_slabs_match_oracle(case, value):
    w, inp = masked(case, value)
    mod = make_module(w)
    out = gpu_forward(mod, w, inp)
    assert mod.last_launch_count() == 1
    assert_close(out, oracle_forward(w, inp), w.dtype, f"{case} {value}")


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("case", OTHERS, ids=IDS)
def test_extreme_numbers_reach_as_far_as_on_register_tiles(case, kind):
    B, heads, H, W, d, pool, dtype, _ = case
    w = Workload("extreme", B, heads, H, W, d, pool, dtype, True, True, 1.0, seed=150 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    extreme(inp, kind, dtype, W)
    mod = make_module(w)
    out, tiles = gpu_forward(mod, w, inp), gpu_forward(make_module(w, path=AA_PATH_UNFUSED), w, inp)
    assert mod.last_launch_count() == 1
    assert torch.equal(out.isnan(), tiles.isnan()) and torch.equal(out.isinf(), tiles.isinf())
    both = out.isfinite()
    assert not both.any() or float((out[both].float() - tiles[both].float()).abs().max()) <= 2e-2


@pytest.mark.parametrize("case", OTHERS, ids=IDS)
def test_given_agents_and_other_scales(case):
    """A caller's agents and scales that are no power of two: as close to 64 bits as on register tiles, which scale fp32 logits too (both round V_A, the
    weights and the output once: a tenth more is the luck of the draw)."""
    B, heads, H, W, d, pool, dtype, _ = case
    w = Workload("given", B, heads, H, W, d, pool, dtype, True, False, 1.0, seed=160 + H * W)
    inp = {k: None if t is None else (2 * t.float()).to(t.dtype) for k, t in make_inputs(w, bias_std=0.25).items()}
    n, scale = w.agents, d ** -0.15
    agents = (2 * torch.randn((B, heads, n, d), generator=torch.Generator().manual_seed(4))).to(inp["q"].dtype).cuda()
    q, k, v, b1, b2 = (to_dev(inp[x]).double() for x in ("q", "k", "v", "b1", "b2"))
    a = agents.double()
    va = torch.softmax(scale * a @ k.transpose(2, 3) + b1, -1) @ v
    ref = torch.softmax(0.5 * scale * q @ a.transpose(2, 3) + b2, -1) @ va
    err = []
    for path in (0, AA_PATH_UNFUSED):
        mod = make_module(w, path=path, scale1=scale, scale2=0.5 * scale)
        err.append(float((gpu_forward(mod, w, inp, agents=agents).double() - ref).norm() / ref.norm()))
        assert path or mod.last_launch_count() == 1
    assert err[0] <= 1.1 * err[1], err
