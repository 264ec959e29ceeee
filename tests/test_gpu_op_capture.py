"""Operator calls that were captured into a CUDA graph: results and status words are those of the latest replay."""
import numpy as np
import pytest

from vla_synth.gen import round_to_bf16

pytestmark = pytest.mark.gpu


def _rand(rng, shape, scale=1.0):
    import torch
    return torch.from_numpy(round_to_bf16((scale * rng.standard_normal(shape)).astype(np.float32))).cuda().to(torch.bfloat16)


def test_a_captured_call_reports_on_its_latest_replay():
    """Two graphs of the same calls, one captured with the operand loads switched off (its bounded waits run out on every replay)."""
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(8)
    a, w = _rand(rng, (50, 256)), _rand(rng, (256, 256), 0.1)
    scratch = torch.empty(api.op_attention_scratch_bytes(50, 4, 64), dtype=torch.uint8, device="cuda")

    def calls(stream=None):
        x = api.op_linear(a, w, out_bf16=True, stream=stream)
        return x, api.op_attention(x, x, x, 4, 4, 64, scratch=scratch, stream=stream)

    def status():
        return api.op_status(api.OP_LINEAR), api.op_status(api.OP_ATTENTION, scratch)

    want = calls()
    assert status() == (api.VLA_OK, api.VLA_OK)
    side = torch.cuda.Stream()
    graphs = []
    try:
        for drop in (False, True):
            api.debug_op_fault(drop, wait_limit_ns=1_000_000 if drop else 0)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                out = calls(side)
            graphs.append((g, out))
    finally:
        api.debug_op_fault(False)
    good, bad = graphs
    for _ in range(2):
        bad[0].replay()
        assert status() == (api.VLA_ERR_TIMEOUT, api.VLA_ERR_TIMEOUT)
        good[0].replay()
        assert status() == (api.VLA_OK, api.VLA_OK)
        assert all(torch.equal(x, y) for x, y in zip(good[1], want))
        bad[0].replay()
        again = calls()
        assert status() == (api.VLA_OK, api.VLA_OK)
        assert all(torch.equal(x, y) for x, y in zip(again, want))
