"""Streaming kernels on token-major views (no transposes): bit for bit the dense call, and the fp64 oracle."""
import pytest
import torch

from paper_2312_08874_b200 import Workload, make_inputs
from tests.parity_util import assert_close, gpu_forward, make_module, oracle_forward, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H  W   pool dtype  bias  dwc
    (2, 3, 56, 56, 7, "bf16", True, True),       # heads nested inside tokens
    (3, 1, 56, 56, 7, "bf16", True, True),       # a single head
    (1, 2, 32, 40, 8, "f16", True, True),        # a single batch entry, 64 agents
    (2, 2, 128, 8, 4, "f16", False, True),       # the narrowest grid, no biases
    (1, 1, 64, 64, 4, "bf16", True, False),      # the widest
]


@pytest.mark.parametrize("packed", [False, True], ids=["bnhd", "qkv_interleaved"])
@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_p{c[4]}" for c in SHAPES])
def test_strided_stream_matches_dense(case, packed):
    B, heads, H, W, pool, dtype, bias, dwc = case
    w = Workload("stream", B, heads, H, W, 64, pool, dtype, bias, dwc, 1.0, seed=500 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    dense = gpu_forward(mod, w, inp)
    assert mod.last_launch_count() == 3, "expected the streaming kernels"
    q, k, v = (to_dev(inp[x]) for x in ("q", "k", "v"))
    if packed:
        qkv = torch.stack([t.permute(0, 2, 1, 3) for t in (q, k, v)], dim=2).contiguous()    # [B, N, 3, heads, d]
        views = [qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3)]
    else:
        views = [t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (q, k, v)]
    out = mod.forward_strided(*views, H, W, w.agents, b1=to_dev(inp["b1"]), b2=to_dev(inp["b2"]), dwc_weight=to_dev(inp["dwc"]))
    assert mod.query_status() == 0 and mod.last_launch_count() == 3
    assert torch.equal(out, dense)
    slabs = [(0, 0), (B - 1, heads - 1)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert_close(out[b:b + 1, h:h + 1].contiguous(), ref, dtype, f"{case} slab {(b, h)}")
