"""Calls on host buffers that are cut into parts, against the same call on device tensors and the fp64 oracle."""
import pytest
import torch

from paper_2312_08874_b200 import Workload, make_inputs
from tests.parity_util import assert_close, make_module, oracle_forward

pytestmark = pytest.mark.gpu

SHAPES = [
    # batch heads H  W   d   pool dtype  bias  dwc
    (11, 2, 56, 56, 64, 7, "bf16", True, True),      # four parts of 6, 3, 1 and 1 batch entries
    (1, 5, 73, 75, 64, 5, "f16", True, True),        # parts by heads, their biases at odd offsets
    (5, 1, 60, 61, 32, 4, "f32", False, True),       # fp32, fewer parts than entries
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"B{c[0]}h{c[1]}_{c[2]}x{c[3]}_d{c[4]}_{c[6]}" for c in SHAPES])
def test_split_host_call_matches_oracle(case):
    B, heads, H, W, d, pool, dtype, bias, dwc = case
    w = Workload("host", B, heads, H, W, d, pool, dtype, bias, dwc, 1.0, seed=900 + H * W)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    pin = {k: (None if v is None else v.pin_memory()) for k, v in inp.items()}
    args = (w.grid_h, w.grid_w, w.agents)
    ops = dict(b1=pin["b1"], b2=pin["b2"], dwc_weight=pin["dwc"])
    out = mod.forward_host(pin["q"], pin["k"], pin["v"], *args, **ops)
    assert mod.last_launch_count() > 3, "expected several parts"
    slabs = [(0, 0), (B - 1, heads - 1), (B // 2, heads // 2)]
    for (b, h), ref in zip(slabs, oracle_forward(w, inp, slabs=slabs)):
        assert_close(out[b:b + 1, h:h + 1], ref, dtype, f"{case} slab {(b, h)}")
    # on a stream of the caller's, twice in flight with a staging buffer each
    lanes = [(torch.cuda.Stream(), torch.empty(mod.staging_bytes(*args), dtype=torch.uint8, device="cuda"), torch.empty_like(out).pin_memory()) for _ in range(2)]
    for s, stg, o in lanes + lanes:
        mod.forward_host(pin["q"], pin["k"], pin["v"], *args, **ops, out=o, stream=s, synchronize=False, staging=stg)
    torch.cuda.synchronize()
    assert all(torch.equal(o, out) for _, _, o in lanes)
    assert mod.query_status() == 0


def test_split_host_calls_on_different_streams_do_not_wait_for_one_another():
    w = Workload("host", 8, 2, 56, 56, 64, 7, "bf16", True, True, 1.0, seed=901)
    inp = make_inputs(w, bias_std=0.5, dwc_std=0.2)
    mod = make_module(w)
    pin = {k: v.pin_memory() for k, v in inp.items()}
    args = (pin["q"], pin["k"], pin["v"], w.grid_h, w.grid_w, w.agents)
    ops = dict(b1=pin["b1"], b2=pin["b2"], dwc_weight=pin["dwc"])
    want = mod.forward_host(*args, **ops)
    assert mod.last_launch_count() > 3, "expected several parts"
    lanes = [(torch.cuda.Stream(), torch.empty(mod.staging_bytes(w.grid_h, w.grid_w, w.agents), dtype=torch.uint8, device="cuda"), torch.empty_like(want).pin_memory())
             for _ in range(6)]

    def call(s, stg, o):
        mod.forward_host(*args, **ops, out=o, stream=s, synchronize=False, staging=stg)

    busy, idle = lanes[:2]
    for lane in (idle, busy, busy):                        # both streams have called before
        call(*lane)
    torch.cuda.synchronize()
    with torch.cuda.stream(busy[0]):
        torch.cuda._sleep(1_000_000_000)                   # half a second of work before its call
    call(*busy)
    assert mod.last_launch_count() > 3, "expected several parts"
    ended = torch.cuda.Event()
    ended.record(busy[0])
    call(*idle)
    assert mod.last_launch_count() == 3, "beside a call in flight: one piece"
    idle[0].synchronize()
    assert not ended.query(), "the call on the idle stream waited for the busy one"
    # more streams at work than the handle keeps copy streams for
    for s, _, _ in lanes:
        with torch.cuda.stream(s):
            torch.cuda._sleep(2_000_000)
    for lane in lanes + lanes:
        call(*lane)
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for _, _, o in lanes) and mod.query_status() == 0
