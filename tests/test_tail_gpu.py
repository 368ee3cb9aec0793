"""Token-wise tail of the backward pass (pooling, depthwise and filter gradients) at the edges of its strips and blocks, against the fp64 oracle."""
import pytest
import torch

from paper_2312_08874_b200 import AA_PATH_AUTO, Workload, make_inputs, make_upstream_grad
from tests.parity_util import make_module, to_dev
from tests.test_backward_gpu import check, run_both

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W   d   pool dtype
    (1, 1, 3, 131, 40, 3, "bf16"),        # six columns at once (eight threads idle), the last group short
    (1, 2, 5, 300, 64, 5, "f16"),         # many columns of few rows, unequal windows
    (2, 1, 130, 9, 104, 4, "bf16"),       # several strips of rows, two columns at once (24 threads idle)
    (3, 1, 8, 16, 16, 2, "f16"),          # every column of the grid at once, exactly
    (1, 1, 43, 3, 8, 3, "bf16"),          # more columns at once than the grid has
    (160, 2, 9, 15, 80, 3, "bf16"),       # blocks that go through several batch entries of their head
    (2, 2, 30, 41, 128, 6, "f16"),
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}" for c in SHAPES])
def test_tail_edges_match_oracle(case):
    B, heads, H, W, d, pool, dtype = case
    w = Workload("tail", B, heads, H, W, d, pool, dtype, True, True, 1.0, seed=600 + H * W + d)
    _, got, ref = run_both(w, make_inputs(w, bias_std=0.5, dwc_std=0.2), path=AA_PATH_AUTO)
    check(got, ref, str(case), tc=d == 64)


# strips of rows and runs of columns: fewer rows than a strip starts ahead, more rows than the window table holds, strips and columns
# that do not divide, several passes of a block, the smallest and largest head sizes, fp32
STRIPS = [
    (1, 1, 1, 70, 64, 1, "bf16"),
    (2, 1, 2, 5, 8, 2, "f32"),
    (1, 1, 600, 4, 16, 4, "f16"),
    (1, 2, 37, 33, 48, 7, "f32"),
    (40, 2, 29, 31, 64, 4, "bf16"),
    (1, 1, 25, 27, 128, 5, "bf16"),
]


@pytest.mark.parametrize("case", STRIPS, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}_{c[6]}" for c in STRIPS])
def test_strips_match_oracle(case):
    B, heads, H, W, d, pool, dtype = case
    w = Workload("tail", B, heads, H, W, d, pool, dtype, True, True, 1.0, seed=700 + H * W + d)
    _, got, ref = run_both(w, make_inputs(w, bias_std=0.5, dwc_std=0.2), path=AA_PATH_AUTO)
    check(got, ref, str(case), tc=d == 64 and dtype != "f32")


@pytest.mark.parametrize("case", [(64, 8, 7), (64, 16, 7), (128, 4, 7), (32, 16, 14)], ids=lambda c: f"B{c[0]}h{c[1]}_{c[2]}x{c[2]}")
def test_filter_gradient_is_shared_by_every_copy(case):
    """Blocks add their share of a head's filter gradient to one of sixteen copies, so that a word takes a sixteenth of the roundings and of
    the atomics.  Every copy of every head is in use where a head has at least as many blocks (here 40 to 90)."""
    B, heads, grid = case
    w = Workload("copies", B, heads, grid, grid, 64, 7, "bf16", False, True, 1.0, seed=770)
    inp, mod = make_inputs(w, dwc_std=0.2), make_module(w)
    ws = torch.zeros(mod.lib.agent_attn_backward_workspace_bytes(mod._h, grid, grid, 49), dtype=torch.uint8, device="cuda")
    mod.backward(to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"]), to_dev(make_upstream_grad(w)), grid, grid, 49,
                 dwc_weight=to_dev(inp["dwc"]), workspace=ws)
    torch.cuda.synchronize()
    up = lambda x: (x + 255) // 256 * 256
    at = 4 * up(B * heads * 49 * 64 * 4) + 2 * up(B * heads * 49 * 4)             # A, V_A, dV_A, dA, then two words per agent
    copies = ws[at:at + 16 * heads * 64 * 9 * 4].view(torch.float32).view(16, heads, 64 * 9)
    used = (copies != 0).any(dim=2).sum(dim=0).tolist()
    assert used == [16] * heads, used


@pytest.mark.parametrize("filter_grad", [True, False])
def test_pooling_beside_the_depthwise_part_changes_nothing(filter_grad):
    """dQ does not depend on the depthwise term.  Slabs of one tile have sums of a fixed order, so it is the same bit for bit with the term, whose
    kernel the pooling then runs beside, and without."""
    w = Workload("beside", 300, 3, 11, 11, 64, 3, "bf16", False, True, 1.0, seed=78)
    inp, go, mod = make_inputs(w, dwc_std=0.2), to_dev(make_upstream_grad(w)), make_module(w)
    q, k, v, f = (to_dev(inp[x]) for x in ("q", "k", "v", "dwc"))
    want = mod.backward(q, k, v, go, 11, 11, 9)["dq"]
    for _ in range(30):
        got = mod.backward(q, k, v, go, 11, 11, 9, dwc_weight=f, need_filter_grad=filter_grad)
        assert torch.equal(got["dq"], want)
    assert mod.query_status() == 0
