"""fp32 tensors on the tensor cores (operands as sums of 16-bit terms) at the edges of their tiles, against the fp64 oracle."""
import pytest
import torch

from oracle import agent_attention_oracle as orc
from paper_2312_08874_b200 import AA_PATH_AUTO, Workload, make_inputs, make_upstream_grad
from tests.parity_util import assert_close, errors, make_module, oracle_forward, to_dev, to_np
from tests.test_backward_gpu import check, run_both

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H  W   d   pool bias  dwc
    (1, 1, 4, 4, 8, 4, True, True),           # as many agents as tokens, channels padded from 8 to 32
    (2, 1, 31, 33, 72, 3, True, True),        # one row group, unaligned bias rows, channels padded to 80
    (1, 2, 37, 36, 64, 6, True, True),        # 36 agents: three row groups, ragged last tile
    (1, 2, 20, 20, 48, 9, True, False),       # 81 agents: six row groups
    (1, 1, 40, 41, 64, 16, True, True),       # 256 agents: two row blocks
    (1, 1, 33, 12, 128, 8, True, True),       # 128 channels: two row blocks of 32 agents
    (2, 1, 9, 300, 32, 5, False, True),
    (40, 4, 7, 7, 40, 7, True, True),         # every token its own agent, many slabs
]
IDS = [f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}" for c in SHAPES]


def workload(case):
    B, heads, H, W, d, pool, bias, dwc = case
    return Workload("terms", B, heads, H, W, d, pool, "f32", bias, dwc, 1.0, seed=800 + H * W + d)


@pytest.mark.parametrize("case", SHAPES, ids=IDS)
def test_fp32_forward_matches_oracle(case):
    w = workload(case)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    ws = mod.workspace(w.grid_h, w.grid_w, w.agents)
    out = mod.forward(to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"]), w.grid_h, w.grid_w, w.agents, b1=to_dev(inp["b1"]),
                      b2=to_dev(inp["b2"]), dwc_weight=to_dev(inp["dwc"]), workspace=ws)
    assert mod.last_launch_count() == 3
    slabs = [(0, 0), (w.batch - 1, w.heads - 1)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert_close(out[b:b + 1, h:h + 1], ref, "f32", f"{case} slab {(b, h)}")
    # the same with the agents handed in
    agents, va = (t.clone() for t in mod.intermediates(ws, w.agents))
    again = mod.forward(to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"]), w.grid_h, w.grid_w, w.agents, agents=agents, b1=to_dev(inp["b1"]),
                        b2=to_dev(inp["b2"]), dwc_weight=to_dev(inp["dwc"]))
    assert torch.equal(out, again) and bool(torch.isfinite(va).all())


@pytest.mark.parametrize("case", [c for c in SHAPES if c[4] <= 80], ids=[i for i, c in zip(IDS, SHAPES) if c[4] <= 80])
def test_fp32_backward_matches_oracle(case):
    w = workload(case)
    _, got, ref = run_both(w, make_inputs(w, bias_std=0.5, dwc_std=0.2), path=AA_PATH_AUTO)
    check(got, ref, str(case))


# Many slabs: a block takes thousands of tokens of one.  fp32 arithmetic that rounds to nearest: an output passes through about eight
# rounded stages (operands, logits, exponential, weights, two sums, the merge) of 2^-24 each, random sums of their errors well below
# 16 x 2^-24 = 1e-6; the logit gradients are differences dP - rowsum(P dP) that cancel up to three quarters of dP: 4e-6.
LONG_FORWARD, LONG_BACKWARD = 1e-6, 4e-6


def test_fp32_forward_of_many_long_slabs_stays_fp32_accurate():
    w = Workload("long", 2, 8, 128, 128, 64, 7, "f32", True, False, 1.0, seed=31)
    inp = make_inputs(w, bias_std=0.2)
    out = make_module(w).forward(to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"]), w.grid_h, w.grid_w, w.agents, b1=to_dev(inp["b1"]), b2=to_dev(inp["b2"]))
    slabs = [(0, 0), (1, 7)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert errors(out[b:b + 1, h:h + 1], ref)["rel_l2"] <= LONG_FORWARD


def test_term_gradients_of_many_long_slabs_stay_fp32_accurate():
    w = Workload("long", 2, 8, 128, 128, 64, 16, "bf16", True, False, 1.0, seed=32)
    inp, go = make_inputs(w, bias_std=0.2), make_upstream_grad(w)
    got = make_module(w).backward(to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"]), to_dev(go), w.grid_h, w.grid_w, w.agents,
                                  b1=to_dev(inp["b1"]), b2=to_dev(inp["b2"]))
    b, h = 1, 6
    one = lambda t: to_np(t[b:b + 1, h:h + 1])
    ref = orc.backward(one(inp["q"]), one(inp["k"]), one(inp["v"]), one(go), w.grid_h, w.grid_w, (w.pool, w.pool),
                       b1=to_np(inp["b1"][h:h + 1]), b2=to_np(inp["b2"][h:h + 1]))
    for key in ("dq", "dk", "dv"):
        assert errors(got[key][b:b + 1, h:h + 1], ref[key])["rel_l2"] <= LONG_BACKWARD, key


def test_mixed_precision_gradients_carry_agent_features_as_two_terms_hold_them():
    """The mixed-precision backward pass keeps V_A in fp32 (the second region of its workspace) and reads it as two bf16 terms, good to
    2^-17 = 8e-6.  444 slabs fill 148 SMs, so that a block sums 3136 tokens, which must not lose that; the values have a mean, so rounding does not average out."""
    w = Workload("mixed", 444, 1, 56, 56, 64, 7, "bf16", False, False, 1.0, seed=33)
    g = torch.Generator(device="cuda")
    g.manual_seed(w.seed)
    q, k, v, go = (torch.randn((w.batch, 1, w.tokens, 64), generator=g, device="cuda").to(torch.bfloat16) for _ in range(4))
    v += 1
    mod = make_module(w)
    ws = mod.backward_workspace(56, 56, 49)
    mod.backward(q, k, v, go, 56, 56, 49, workspace=ws)
    size = w.slabs * 49 * 64 * 4
    va = ws[size:2 * size].view(torch.float32).view(w.slabs, 49, 64)
    for s in (0, w.slabs - 1):
        a = q[s, 0].view(7, 8, 7, 8, 64).double().mean(dim=(1, 3)).view(49, 64).to(torch.bfloat16).double()
        ref = torch.softmax(a @ k[s, 0].double().T / 8, dim=1) @ v[s, 0].double()
        assert float((va[s] - ref).norm() / ref.norm()) <= 8e-6 / 4


@pytest.mark.parametrize("pool", [4, 7])
def test_fp32_forward_of_values_at_the_end_of_the_range(pool):
    """fp32 reaches half a bf16 step past the largest bf16: such a value must not become infinite when it is split into bf16 terms."""
    w = Workload("range", 1, 2, 14, 14, 64, pool, "f32", True, True, 1.0, seed=34)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    inp["v"][0, 0, 5, 7] = torch.finfo(torch.float32).max
    inp["v"][0, 0, 90, 9] = -torch.finfo(torch.float32).max
    dev = {k: to_dev(v) for k, v in inp.items()}
    out = make_module(w).forward(dev["q"], dev["k"], dev["v"], 14, 14, w.agents, b1=dev["b1"], b2=dev["b2"], dwc_weight=dev["dwc"])
    ref = oracle_forward(w, inp)
    for ch in (7, 9):
        assert_close(out[:, :1, :, ch] * 1e-38, ref[:, :1, :, ch] * 1e-38, "f32", f"channel {ch}")
    rest = [c for c in range(64) if c not in (7, 9)]
    assert_close(out[:, :, :, rest], ref[:, :, :, rest], "f32", "the others")


@pytest.mark.parametrize("case", [(14, 14, 64, 7), (20, 21, 24, 5), (40, 41, 64, 16)], ids=["short", "padded_channels", "two_row_blocks"])
def test_fp32_forward_of_an_infinite_value(case):
    """An infinite value makes its own channel infinite (NaN where infinities of both signs meet) and touches no other."""
    H, W, d, pool = case
    w = Workload("infinite", 1, 2, H, W, d, pool, "f32", True, True, 1.0, seed=35)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    clean = oracle_forward(w, inp)
    t1, t2 = 2 * W + 2, (H - 3) * W + 5
    inp["v"][0, 0, t1, 7] = float("inf")
    inp["v"][0, 0, t1, 9] = -float("inf")
    inp["v"][0, 0, t1, 11] = float("inf")
    inp["v"][0, 0, t2, 11] = -float("inf")
    dev = {k: to_dev(v) for k, v in inp.items()}
    out = make_module(w).forward(dev["q"], dev["k"], dev["v"], H, W, w.agents, b1=dev["b1"], b2=dev["b2"], dwc_weight=dev["dwc"])
    rest = [c for c in range(d) if c not in (7, 9, 11)]
    assert_close(out[:, :, :, rest], clean[:, :, :, rest], "f32", "the other channels")
    assert_close(out[:, 1], clean[:, 1], "f32", "the other head")
    far = [t for t in range(w.tokens) if abs(t // W - t1 // W) > 1]        # (beside the value the depthwise term adds an infinity of its own)
    assert torch.equal(out[0, 0, far, 7], torch.full((len(far),), float("inf"), device="cuda"))
    assert torch.equal(out[0, 0, far, 9], torch.full((len(far),), -float("inf"), device="cuda"))
    assert bool(torch.isnan(out[0, 0, :, 11]).all())
