"""Either side of the lines between the tensor-memory kernels and the register-tiled ones, and between one kernel and three, against the fp64
oracle."""
import pytest

from paper_2312_08874_b200 import Workload, make_inputs
from tests.parity_util import assert_close, gpu_forward, make_module, oracle_forward, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W   d   pool launches
    (1, 1, 64, 96, 64, 16, 4),        # 6144 tokens, filled blocks: tensor memory
    (1, 1, 64, 95, 64, 16, 3),        # fewer: register tiles
    (20, 2, 47, 80, 64, 16, 4),       # short axis, 150400 tokens in all: tensor memory
    (1, 2, 64, 128, 64, 12, 4),       # half-filled blocks on a long axis: tensor memory
    (1, 2, 64, 128, 32, 12, 3),       # and of few channels: register tiles
    (4, 4, 32, 64, 64, 16, 4),        # filled blocks, a tile for every SM: tensor memory
    (3, 5, 32, 64, 64, 16, 3),        # fewer: register tiles
    (1, 1, 64, 96, 64, 12, 4),        # half-filled blocks, 6144 tokens of few slabs: tensor memory
    (17, 1, 64, 96, 64, 12, 3),       # of many: register tiles
    (2, 1, 64, 128, 40, 16, 4),       # filled with agents, 40 channels: tensor memory
    (2, 1, 64, 128, 32, 16, 3),       # 32: register tiles
    (4, 8, 48, 64, 40, 10, 4),        # 100 agents, 32 slabs: tensor memory, the broadcast on register tiles
    (8, 8, 48, 64, 40, 10, 3),        # 64 slabs of few channels: register tiles
    (8, 8, 24, 32, 64, 11, 1),        # a short axis, 121 agents: one kernel
    (1, 1, 72, 96, 40, 15, 3),        # 225 agents of 40 channels, one slab: register tiles
    (2, 1, 72, 96, 40, 15, 4),        # two: tensor memory
    (1, 1, 72, 96, 40, 10, 4),        # one, 100 agents: tensor memory
    (2, 2, 96, 128, 32, 11, 4),       # 121 agents of 32 channels, four slabs: tensor memory
    (2, 1, 31, 33, 64, 8, 1),         # 1023 tokens: one kernel
    (2, 1, 15, 69, 64, 8, 3),         # 1035 on a grid too wide for the streaming kernels: three
    (48, 6, 9, 9, 128, 5, 1),         # slabs all resident: one kernel
    (50, 6, 9, 9, 128, 5, 3),         # more than fit: three
    (50, 6, 8, 8, 128, 5, 1),         # but not on the shortest grids
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}" for c in SHAPES])
def test_dispatch_lines(case):
    B, heads, H, W, d, pool, launches = case
    w = Workload("dispatch", B, heads, H, W, d, pool, "bf16", True, True, 1.0, seed=400 + H * W + d)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    out = gpu_forward(mod, w, inp)
    assert mod.last_launch_count() == launches
    slabs = [(0, 0), (B - 1, heads - 1)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert_close(out[b:b + 1, h:h + 1], ref, "bf16", f"{case} slab {(b, h)}")


@pytest.mark.parametrize("case", [(4, 4, 32, 64), (1, 2, 64, 96), (3, 1, 64, 128)], ids=["short", "one_entry", "one_head"])
def test_token_major_views_that_no_tensor_map_expresses(case):
    """[N, B, heads, d] storage, or heads outside the batch: strides do not nest as tensor maps want them, so the shapes of the tensor-memory
    kernels run on register tiles (with one batch entry or one head they nest)."""
    B, heads, H, W = case
    w = Workload("dispatch", B, heads, H, W, 64, 16, "bf16", True, True, 1.0, seed=500 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    kw = dict(b1=to_dev(inp["b1"]), b2=to_dev(inp["b2"]), dwc_weight=to_dev(inp["dwc"]))
    slabs = [(0, 0), (B - 1, heads - 1)]
    refs = oracle_forward(w, inp, slabs=slabs)
    for order in ((2, 0, 1, 3), (1, 2, 0, 3)):                 # storage [N, B, heads, d], and [heads, N, B, d]
        back = [order.index(i) for i in range(4)]
        views = [to_dev(inp[x]).permute(order).contiguous().permute(back) for x in ("q", "k", "v")]
        out = mod.forward_strided(*views, H, W, w.agents, **kw)
        assert mod.query_status() == 0
        if B > 1 and heads > 1:
            assert mod.last_launch_count() == 3
        for (b, h), ref in zip(slabs, refs):
            assert_close(out[b:b + 1, h:h + 1].contiguous(), ref, "bf16", f"{case} {order} slab {(b, h)}")
