"""Gradient stages on tensor memory (n <= 64 agents, 64 channels) at the edges of their tiles and runs, against the fp64 oracle."""
import pytest

from paper_2312_08874_b200 import AA_PATH_AUTO, Workload, make_inputs
from tests.parity_util import make_module
from tests.test_backward_gpu import check, run_both

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W  pool dtype bias
    (1, 1, 1, 127, 1, "bf16", True),      # one token short of a tile, one agent
    (2, 1, 8, 16, 6, "f16", True),        # exactly one tile, agents in both halves
    (1, 3, 3, 43, 3, "bf16", True),       # one token past a tile, odd rows of both biases in every head
    (1, 2, 16, 16, 8, "bf16", False),     # two full tiles, every agent column in use, no bias
    (75, 2, 15, 20, 5, "bf16", True),     # more slabs than blocks: runs that start and end inside a slab
    (50, 3, 7, 7, 7, "f16", True),        # runs of several slabs of one ragged tile
    (1, 1, 61, 83, 7, "f16", True),       # several blocks per slab
    (2, 2, 33, 32, 4, "bf16", True),      # 16 agents: B2 is read as it is, rows of 32 bytes; B1 with a row of agents in use past 1024 tokens
    (3, 2, 22, 14, 8, "f16", True),       # bias gradients by bulk reductions: 64 agents, a tile of 52 tokens
    (2, 3, 20, 15, 7, "bf16", True),      # the same, token rows of 49 agents
    (1, 1, 200, 201, 3, "bf16", True),    # agent values: more than 32 states for each warp of a row's block
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_p{c[4]}_{c[5]}" for c in SHAPES])
def test_tiles_and_runs_match_oracle(case):
    B, heads, H, W, pool, dtype, bias = case
    w = Workload("umma", B, heads, H, W, 64, pool, dtype, bias, True, 1.0, seed=800 + H * W + pool)
    mod, got, ref = run_both(w, make_inputs(w, bias_std=0.5, dwc_std=0.2), path=AA_PATH_AUTO)
    check(got, ref, str(case), tc=True)
    assert mod.last_launch_count() == (7 if H * W > 1024 else 6), "expected the tensor-memory gradient kernels"


@pytest.mark.parametrize("pool,copies", [(3, 2), (8, 1)], ids=["p3", "p8"])
def test_workspace_holds_biases_as_wide_as_their_agents(pool, copies):
    """Copies of the biases have rows of n agents rounded up to 8 (16 bytes), and B2 none where its rows are that already.  Beside them: four
    fp32 words per agent and channel and the partial states of V_A, one 35 KB state per tile run, at most as many as blocks and slabs."""
    w = Workload("ws", 1, 8, 256, 256, 64, pool, "bf16", True, True, 1.0)
    mod, n = make_module(w), pool * pool
    rows = 8 * 65536 * ((n + 7) // 8 * 8) * 2
    assert mod.lib.agent_attn_backward_workspace_bytes(mod._h, 256, 256, n) <= copies * rows + (8 << 20)
