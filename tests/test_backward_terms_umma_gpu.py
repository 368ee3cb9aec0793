"""Gradients with fp32 accuracy on tensor memory (bf16, up to 64 channels) at the edges of tiles, agent blocks and runs, against the fp64 oracle."""
import numpy as np
import pytest

from paper_2312_08874_b200 import AA_PATH_AUTO, Workload, make_inputs
from tests.test_backward_gpu import check, run_both

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W   d  pool dtype bias
    (140, 1, 2, 63, 56, 2, "bf16", True),     # two tokens short of a tile, few agents
    (1, 1, 96, 87, 32, 5, "bf16", True),      # 25 agents of 32 channels on a long axis
    (2, 1, 8, 16, 40, 6, "bf16", True),       # exactly one tile, agents in both halves, ragged channels
    (1, 3, 9, 43, 64, 9, "bf16", True),       # a batch of one: bias gradients are stored; odd rows of both biases
    (2, 2, 16, 16, 64, 16, "bf16", False),    # four full blocks of agents, two full tiles, no bias
    (75, 2, 15, 20, 64, 9, "bf16", True),     # more units than blocks: runs that start and end inside a block of agents
    (40, 3, 12, 12, 48, 12, "bf16", True),    # runs of several blocks of agents of two ragged tiles
    (2, 1, 61, 83, 64, 14, "bf16", True),     # many tiles per block of agents
    (1, 1, 33, 32, 40, 7, "bf16", True),      # agent values on tensor memory: two rows per agent, a token past a multiple of eight tiles
    (1, 2, 105, 79, 64, 11, "bf16", True),    # one block of 128 agents, N and n odd: both biases are padded
    (3, 2, 64, 43, 64, 13, "bf16", False),    # two blocks, runs that hold parts of two slabs
    (1, 1, 70, 41, 64, 9, "bf16", True),      # agent values: 24 states a row, three for a warp
    (1, 2, 64, 65, 40, 6, "bf16", True),      # two rows per agent, 66 states, slabs that begin inside a run
    (3, 4, 95, 100, 56, 16, "bf16", True),    # 300 tiles of the axis on 37 runs: blocks own their bias gradients, stretches that end with a run or a head
    (2, 2, 168, 169, 32, 9, "bf16", True),    # three tiles of the axis a block, with both blocks of agents and batch entries; the last one is ragged
    (1, 8, 111, 128, 56, 9, "bf16", True),    # six, one batch entry
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}" for c in SHAPES])
def test_tiles_and_agent_blocks_match_oracle(case):
    B, heads, H, W, d, pool, dtype, bias = case
    w = Workload("terms_umma", B, heads, H, W, d, pool, dtype, bias, True, 1.0, seed=900 + H * W + pool)
    mod, got, ref = run_both(w, make_inputs(w, bias_std=0.5, dwc_std=0.2), path=AA_PATH_AUTO)
    check(got, ref, str(case))
    values = H * W > 1024 or (pool > 8 and B * heads * H * W >= 16384)
    assert mod.last_launch_count() == 8 + (pool > 8) + values, "expected the tensor-memory gradient kernels"


# both sides of the lines between these kernels (8 launches, 9 past 1024 tokens) and those on mma.sync (10) for up to 32 agents
LINES = [
    # batch heads H   W   d  pool launches
    (1, 1, 13, 15, 56, 5, 10), (1, 1, 14, 14, 56, 5, 8), (30, 2, 10, 15, 56, 5, 8),
    (1, 1, 33, 31, 56, 3, 10), (1, 1, 32, 32, 56, 3, 8), (16, 4, 10, 25, 56, 4, 8),
    (1, 1, 33, 31, 40, 5, 10), (1, 1, 32, 32, 48, 5, 8), (50, 4, 14, 10, 40, 5, 8),
    (1, 1, 91, 90, 40, 4, 10), (1, 1, 64, 128, 40, 3, 9), (56, 1, 20, 25, 48, 2, 8), (50, 1, 27, 21, 40, 3, 10),
    (1, 1, 2, 63, 32, 2, 10), (1, 1, 91, 90, 32, 5, 10), (1, 1, 64, 128, 32, 5, 9), (1, 1, 64, 128, 32, 4, 10), (110, 1, 16, 16, 24, 5, 8), (105, 1, 16, 17, 32, 5, 10),
]


@pytest.mark.parametrize("case", LINES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}" for c in LINES])
def test_lines_between_both_paths(case):
    B, heads, H, W, d, pool, launches = case
    w = Workload("lines", B, heads, H, W, d, pool, "bf16", True, True, 1.0, seed=970 + H * W + pool)
    mod, got, ref = run_both(w, make_inputs(w, bias_std=0.5, dwc_std=0.2), path=AA_PATH_AUTO)
    check(got, ref, str(case))
    assert mod.last_launch_count() == launches


@pytest.mark.parametrize("case", [(2, 2, 64, 64, 64, 9), (3, 2, 20, 20, 64, 9), (4, 2, 28, 28, 40, 5)], ids=["values_umma", "sums_n81", "sums_d40"])
def test_probabilities_stay_normalised(case):
    """Queries and keys with a common part, logits of 32 (46 in log2 units, whose fp32 unit is 2^-18).  Tensor memory rounds towards zero: a
    step of an accumulation loses half a unit on average, which the statistics of the softmax have to share.  Else every probability, and dV
    with them, is off by one factor of 2^-19 ln 2 = 1.3e-6 a step.  Bound: less than one step."""
    B, heads, H, W, d, pool = case
    w = Workload("mean", B, heads, H, W, d, pool, "bf16", False, False, 1.0, seed=950)
    inp = make_inputs(w)
    for k in ("q", "k"):
        inp[k] = (inp[k].float() + 2.0).to(inp[k].dtype)
    _, got, ref = run_both(w, inp, path=AA_PATH_AUTO)
    g, r = got["dv"].double().cpu().numpy(), ref["dv"]
    bias = float(((g - r) * np.sign(r)).sum() / np.abs(r).sum())
    print(f"{case}: factor of dV 1 + {bias:.2e}")
    assert abs(bias) < 1e-6, bias
