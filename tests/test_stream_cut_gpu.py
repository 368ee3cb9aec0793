"""Grids that the streaming kernels do not take (wider than 64 columns, windows that do not tile them, odd numbers of tokens): register tiles, against
the fp64 oracle and, where the numbers are extreme, the call that is kept on them."""
import pytest
import torch

from paper_2312_08874_b200 import AA_PATH_UNFUSED, Workload, make_inputs
from tests.parity_util import assert_close, gpu_forward, make_module, oracle_forward, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H   W   pool dtype  bias  dwc
    (2, 2, 45, 46, 7, "bf16", True, True),        # overlapping windows, a number of tokens that is no multiple of eight
    (2, 1, 33, 65, 8, "f16", True, True),         # one column past the widest grid of the streaming kernels
    (4, 1, 75, 117, 7, "f16", True, True),        # odd and wide
    (2, 1, 16, 126, 6, "bf16", True, False),      # the halo of a block in one run
    (2, 1, 16, 127, 6, "bf16", False, True),      # the same
    (2, 2, 5, 1024, 5, "bf16", True, True),       # few long rows: the halo in three runs
    (1, 2, 151, 200, 4, "bf16", True, True),      # few large windows: a block of the pooling kernel each
    (3, 1, 700, 8, 7, "f16", True, True),         # a narrow grid, windows that do not tile it
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


def extreme(inp, kind, dtype, W):
    b1, b2 = inp["b1"], inp["b2"]
    if kind == "removed_rows":
        b1[0, 1, :] = b2[0, 5, :] = float("-inf")
    elif kind == "lowest_rows":
        b1[0, 1, :] = b2[0, 5, :] = torch.finfo(b1.dtype).min
    elif kind == "beyond_30000":
        b2[0, 5, :], b2[0, 5, 3], b2[0, 6, 4], b2[0, 6, 7] = -60000, -40000, 60000, 40000
        b1[0, 2, 9], b1[0, 2, 10] = 50000, 35000
    elif kind == "infinite_value":
        inp["v"][0, 0, 3 * W + 5, 21] = float("inf")
        inp["dwc"] = inp["dwc"].abs()
    elif kind == "nan_bias":
        b2[0, 7, 3] = float("nan")
    elif kind == "infinite_bias":
        b2[0, 8, 3] = float("inf")


KINDS = ["removed_rows", "lowest_rows", "beyond_30000", "infinite_value", "nan_bias", "infinite_bias"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("case", [(2, 1, 75, 117, 7, "bf16"), (1, 2, 46, 64, 7, "f16"), (2, 1, 151, 45, 5, "bf16")], ids=["wide", "ragged", "odd"])
def test_extreme_numbers_do_what_they_do_on_register_tiles(case, kind):
    """Rows of biases that remove everything, finite biases beyond +-30000, an infinite value under a positive filter, NaN."""
    B, heads, H, W, pool, dtype = case
    w = Workload("extreme", B, heads, H, W, 64, pool, dtype, True, True, 1.0, seed=130 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    extreme(inp, kind, dtype, W)
    out, tiles = (gpu_forward(make_module(w, path=p), w, inp) for p in (0, AA_PATH_UNFUSED))
    assert torch.equal(torch.nan_to_num(out, 7e4), torch.nan_to_num(tiles, 7e4)) and torch.equal(out.isnan(), tiles.isnan())


@pytest.mark.parametrize("case", [(4, 2, 75, 117, 7), (2, 2, 45, 47, 7)], ids=["wide", "odd"])
def test_logits_of_given_agents_are_scaled_in_fp32(case):
    """A caller's agents and a scale that is no power of two: one rounding of V_A, one of the weights (2^-9 at most each, 0.29 of it in the mean
    square) and one of the output: 2^-9 x 0.29 x sqrt(3) = 1e-3, times 2 for what the weights' errors share.  (scale A rounded to bf16 before the
    products moves the logits, of up to 10 here, by up to 2^-8 of them: 1e-2.)"""
    B, heads, H, W, pool = case
    w = Workload("scale", B, heads, H, W, 64, pool, "bf16", False, False, 1.0, seed=140 + H * W)
    inp = {k: None if v is None else (2 * v.float()).to(v.dtype) for k, v in make_inputs(w).items()}
    agents = (2 * torch.randn((B, heads, w.agents, 64), generator=torch.Generator().manual_seed(3))).to(inp["q"].dtype).cuda()
    scale = 64 ** -0.15
    out = gpu_forward(make_module(w, scale1=scale, scale2=scale), w, inp, agents=agents)[B - 1, 0].double()
    q, k, v = (to_dev(inp[x])[B - 1, 0].double() for x in "qkv")
    a = agents[B - 1, 0].double()
    ref = torch.softmax(scale * q @ a.T, -1) @ (torch.softmax(scale * a @ k.T, -1) @ v)
    assert float((out - ref).norm() / ref.norm()) <= 2.5e-3
