"""Register-tiled kernels at the edges of their tiles, against the fp64 oracle."""
import pytest
import torch

from paper_2312_08874_b200 import Workload, make_inputs
from tests.parity_util import assert_close, gpu_forward, make_module, oracle_forward

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W   d   pool dtype  bias  dwc
    (1, 1, 4, 4, 8, 4, "f16", True, True),           # as many agents as tokens, channels padded from 8 to 32
    (2, 1, 31, 33, 72, 4, "bf16", True, True),       # 1023 tokens: one kernel; 16 agents, odd bias rows, channels padded
    (2, 2, 32, 33, 64, 5, "bf16", True, True),       # 1056 tokens: three kernels; two row groups, ragged last tile
    (1, 3, 5, 300, 64, 5, "f16", True, True),        # W > tile: the halo in three runs
    (1, 1, 3, 131, 40, 3, "bf16", False, True),      # W one past the single-run halo
    (1, 2, 130, 9, 104, 9, "bf16", True, True),      # 81 agents (six row groups), 104 channels padded to 128
    (1, 1, 45, 45, 64, 11, "f16", True, True),       # 121 agents: the last block that fits one row block, unaligned bias rows
    (1, 1, 40, 41, 32, 13, "bf16", True, False),     # 169 agents: two row blocks, bias rows read from global memory
    (1, 1, 33, 32, 128, 16, "bf16", True, True),     # 256 agents of 128 channels
    (160, 2, 11, 13, 64, 7, "bf16", True, True),     # more slabs than resident blocks: a cluster of one
    (7, 2, 23, 70, 64, 5, "f16", True, True),        # fourteen slabs: clusters of sixteen, the last one without tokens
    (5, 3, 23, 70, 64, 5, "f16", True, True),        # fifteen: clusters of eight
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}" for c in SHAPES])
def test_tile_edges_match_oracle(case):
    B, heads, H, W, d, pool, dtype, bias, dwc = case
    w = Workload("tile", B, heads, H, W, d, pool, dtype, bias, dwc, 1.0, seed=700 + H * W + d)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    out = gpu_forward(mod, w, inp)
    slabs = [(0, 0), (B - 1, heads - 1)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert_close(out[b:b + 1, h:h + 1], ref, dtype, f"{case} slab {(b, h)}")
    assert torch.equal(out, gpu_forward(mod, w, inp)), "bit-reproducible"


WEIGHTS = {
    "one_kernel": (2, 2, 14, 14, 64, 7, "bf16"), "three_kernels": (1, 2, 45, 45, 64, 11, "f16"), "d40": (1, 1, 33, 32, 40, 16, "bf16"),
    "wide_grid": (2, 1, 75, 117, 64, 7, "bf16"), "odd_tokens": (2, 2, 45, 47, 64, 7, "f16"), "ragged_windows": (2, 1, 40, 46, 64, 7, "bf16"),
    # tensor memory, where register tiles are the other choice
    "short_slabs": (128, 3, 14, 14, 64, 7, "bf16"), "latent_grid": (2, 8, 64, 64, 40, 16, "bf16"), "latent_grid_f16": (2, 8, 64, 64, 40, 16, "f16"),
    "short_axis": (4, 8, 32, 64, 64, 16, "bf16"), "half_filled": (1, 2, 56, 144, 64, 12, "bf16"),
}


@pytest.mark.parametrize("case", list(WEIGHTS.values()), ids=list(WEIGHTS))
def test_weights_and_their_sums_agree(case):
    """Values that are all one, less themselves through the depthwise term: what is left is how far the rounded weights are from adding up to
    their normaliser.  Both are sums of the same 16-bit numbers, rounded once per 16 of at most 256: 2 x 16 x 2^-23 = 4e-6.  (A normaliser of
    the weights before rounding leaves 2^-9 / sqrt(agents) in bf16.)"""
    B, heads, H, W, d, pool, dtype = case
    w = Workload("weights", B, heads, H, W, d, pool, dtype, True, True, 1.0, seed=36)
    inp = make_inputs(w, bias_std=0.5)
    inp["v"].fill_(1)
    inp["dwc"].zero_()[:, :, 1, 1] = -1
    assert float(gpu_forward(make_module(w), w, inp).abs().max()) <= 4e-6
