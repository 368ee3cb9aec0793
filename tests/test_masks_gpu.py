"""Biases that remove keys and agents (-inf, or the type's lowest value) in whole blocks, against the fp64 oracle."""
import pytest
import torch

from paper_2312_08874_b200 import AA_PATH_AUTO, AA_PATH_QUEUE, AA_PATH_SIMT, Workload, make_inputs
from paper_2312_08874_b200.workloads import TORCH_DTYPE
from tests.parity_util import assert_close, gpu_forward, make_module, oracle_forward
from tests.test_backward_gpu import check, run_both, tensor_core_path

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H  W   d   pool dtype  path
    (1, 2, 20, 20, 64, 7, "f32", AA_PATH_AUTO),       # terms: the first block of 32 agents closed, 17 open
    (1, 1, 32, 33, 32, 9, "f32", AA_PATH_AUTO),       # terms: two blocks closed
    (1, 1, 20, 20, 64, 7, "f32", AA_PATH_SIMT),       # CUDA cores
    (2, 2, 14, 14, 64, 7, "bf16", AA_PATH_AUTO),      # register tiles, one kernel
    (1, 1, 40, 41, 32, 13, "f16", AA_PATH_AUTO),      # register tiles, two row blocks, unaligned bias rows
    (1, 2, 32, 32, 64, 7, "bf16", AA_PATH_AUTO),      # streaming kernels
    (1, 2, 14, 14, 64, 7, "bf16", AA_PATH_QUEUE),     # task queue
    (1, 1, 64, 96, 64, 16, "bf16", AA_PATH_AUTO),     # tensor memory: every agent group of a step closed
    (1, 1, 96, 96, 40, 12, "f16", AA_PATH_AUTO),      # the same, half-filled blocks
    (48, 1, 14, 14, 64, 7, "f32", AA_PATH_AUTO),      # terms, a warp for all agents of 16 tokens (the first two shapes have two)
    (2, 2, 50, 50, 32, 9, "f32", AA_PATH_AUTO),       # the same, two blocks closed
]
IDS = [f"{c[6]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}_path{c[7]}" for c in SHAPES]


def masked(case, value):
    B, heads, H, W, d, pool, dtype, _ = case
    w = Workload("mask", B, heads, H, W, d, pool, dtype, True, True, 1.0, seed=600 + H * W + d)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    low = float("-inf") if value == "inf" else torch.finfo(TORCH_DTYPE[dtype]).min
    n, N = w.agents, w.tokens
    inp["b1"][:, :, :N // 3] = low                        # no agent looks at the first third of the grid
    inp["b1"][0, 3, :N - 24] = low                        # one sees the last 24 tokens only
    inp["b2"][:, ::2, :min(n - 1, max(n * 2 // 3, 32))] = low    # every other token listens to the last agents only
    inp["b2"][:, 1::2, n // 2:] = low
    return w, inp


@pytest.mark.parametrize("value", ["inf", "lowest"])
@pytest.mark.parametrize("case", SHAPES, ids=IDS)
def test_masked_forward_matches_oracle(case, value):
    w, inp = masked(case, value)
    out = gpu_forward(make_module(w, path=case[7]), w, inp)
    assert_close(out, oracle_forward(w, inp), w.dtype, f"{case} {value}")


BACKWARD = [
    (1, 2, 20, 20, 64, 7, "f32", AA_PATH_AUTO),
    (1, 1, 24, 24, 64, 12, "bf16", AA_PATH_AUTO),
    (2, 2, 14, 14, 64, 7, "bf16", AA_PATH_AUTO),
    (2, 1, 14, 14, 64, 7, "bf16", AA_PATH_SIMT),
    # agent values on tensor memory: halves of a row, tiles and whole runs without a key
    (1, 1, 61, 83, 64, 7, "bf16", AA_PATH_AUTO),      # two rows per agent, N odd: B1 by token rows
    (1, 1, 61, 83, 64, 7, "f16", AA_PATH_AUTO),
    (1, 2, 40, 40, 64, 7, "bf16", AA_PATH_AUTO),      # B1 by agent rows
    (1, 1, 40, 41, 40, 7, "bf16", AA_PATH_AUTO),      # the same with three terms
    (1, 1, 105, 79, 64, 11, "bf16", AA_PATH_AUTO),    # one block of 128 rows
    (2, 1, 64, 43, 64, 13, "bf16", AA_PATH_AUTO),     # two
]


@pytest.mark.parametrize("value", ["inf", "lowest"])
@pytest.mark.parametrize("case", BACKWARD, ids=[f"{c[6]}_{c[2]}x{c[3]}_d{c[4]}_p{c[5]}_path{c[7]}" for c in BACKWARD])
def test_masked_backward_matches_oracle(case, value):
    w, inp = masked(case, value)
    _, got, ref = run_both(w, inp, path=case[7])
    check(got, ref, f"{case} {value}", tc=tensor_core_path(w, case[7]))
