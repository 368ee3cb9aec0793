"""Streaming kernels on grids whose rows are cut into shares and windows that do not tile them, against the fp64 oracle."""
import pytest
import torch

from paper_2312_08874_b200 import Workload, make_inputs
from tests.parity_util import assert_close, gpu_forward, make_module, oracle_forward

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W   pool dtype  bias  dwc
    (2, 2, 45, 46, 7, "bf16", True, True),        # whole rows, overlapping windows, a number of tokens that is no multiple of eight
    (2, 1, 33, 65, 8, "f16", True, True),         # one column past whole rows
    (4, 1, 75, 117, 7, "f16", True, True),        # even shares, the last one short
    (2, 1, 16, 126, 6, "bf16", True, False),      # the widest row in one piece
    (2, 1, 16, 127, 6, "bf16", False, True),      # one past it
    (2, 2, 5, 1024, 5, "bf16", True, True),       # many shares, windows wider than a block's turn
    (1, 2, 151, 200, 4, "bf16", True, True),      # few large windows: a block each
    (3, 1, 700, 8, 7, "f16", True, True),         # the narrowest grid
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_p{c[4]}" for c in SHAPES])
def test_cut_rows_and_ragged_windows(case):
    B, heads, H, W, pool, dtype, bias, dwc = case
    w = Workload("cut", B, heads, H, W, 64, pool, dtype, bias, dwc, 1.0, seed=100 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    out = gpu_forward(mod, w, inp)
    assert mod.last_launch_count() == 3
    slabs = [(0, 0), (B - 1, heads - 1)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert_close(out[b:b + 1, h:h + 1], ref, dtype, f"{case} slab {(b, h)}")
    assert torch.equal(out, gpu_forward(mod, w, inp)), "bit-reproducible"
