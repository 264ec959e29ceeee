"""The linear layer's tiles of two SMs (csrc/op_linear_pair.cuh) at their edges: token tiles whose second half is ragged or empty,
widths between 128 and 256 and their remainders, K that ends inside a block, every activation, both result types, stores of
eight, two and one feature; and a call whose operand loads never come."""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(2077, 4944, 712), (1747, 2064, 2288), (4645, 3040, 1000), (7744, 2824, 472), (2936, 1496, 1160), (5125, 440, 2048),
          (978, 14489, 792), (3000, 4902, 520), (129, 16384, 4096),
          (294, 8512, 2952), (452, 6648, 6024), (3261, 392, 1424), (823, 2105, 2000), (3104, 592, 1992), (729, 3139, 3160),       # (fp32: K in two and four parts)
          (300, 5144, 4264), (983, 1626, 3912), (326, 5053, 4064), (935, 1456, 3616), (453, 3482, 3024), (929, 1601, 4064)]      # (bf16 too)


@pytest.mark.parametrize("m,n,k", SHAPES)
@pytest.mark.parametrize("act", [0, 1, 2])
def test_against_64_bit_sums(m, n, k, act):
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(m + act)
    a = torch.randn(m, k, device="cuda", generator=g).to(torch.bfloat16)
    w = (k ** -0.5 * torch.randn(n, k, device="cuda", generator=g)).to(torch.bfloat16)
    ref = a.double() @ w.double().T
    sums = 2.0 ** -23 * (k / 16 + 2) * float(ref.abs().max())          # a unit in the last place per 16 products
    if act:
        ref = torch.nn.functional.gelu(ref, approximate="tanh") if act == 1 else torch.nn.functional.silu(ref)
        sums = 2 * sums + 2.0 ** -10 * float(ref.abs().max())          # (the activations' approximations)
    assert float((api.op_linear(a, w, act=act).double() - ref).abs().max()) <= sums
    assert bool(((api.op_linear(a, w, act=act, out_bf16=True).double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 2 * sums).all())
    assert api.op_status(api.OP_LINEAR) == api.VLA_OK


def test_calls_that_follow_one_another_and_a_wait_that_runs_out():
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(0)
    a = torch.randn(2048, 4096, device="cuda", generator=g).to(torch.bfloat16)
    w = (4096 ** -0.5 * torch.randn(4096, 4096, device="cuda", generator=g)).to(torch.bfloat16)
    x = a
    for i in range(12):                                                # tiles of two SMs and of one in turn, each reading the last result
        x = api.op_linear(x if i % 2 else x[:64].repeat(32, 1), w, out_bf16=True)
        y = api.op_linear(x[:64], w, out_bf16=True)
    assert torch.equal(api.op_linear(x[:64].contiguous(), w, out_bf16=True), y)
    good = api.op_linear(a, w, out_bf16=True)
    api.debug_op_fault(True, 2_000_000)
    try:
        api.op_linear(a, w, out_bf16=True)
        assert api.op_status(api.OP_LINEAR) == api.VLA_ERR_TIMEOUT
    finally:
        api.debug_op_fault(False)
    assert torch.equal(api.op_linear(a, w, out_bf16=True), good) and api.op_status(api.OP_LINEAR) == api.VLA_OK


def test_what_starts_behind_a_call_finds_its_own_barriers():
    """Calls whose CTAs take the shared memory of the CTAs before them at once (each starts while the one in front ends): tiles of two SMs
    whose k-blocks are few more than the stages and not, tiles of one SM, attention of one to eight blocks a CTA.  An arrival that came
    after its CTA's end would land on one of their barriers."""
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(3)

    def rand(rows, cols, s):
        return (s * torch.randn(rows, cols, device="cuda", generator=g)).to(torch.bfloat16)
    linear = [(rand(m, k, 1.0), rand(n, k, k ** -0.5), f32) for m, n, k, f32 in
              ((2048, 16384, 64, False), (1747, 2064, 2288, False), (64, 4096, 720, False), (294, 8512, 2952, True), (3000, 4902, 520, True))]
    attn = [(rand(tq, hq * hd, 1.0), rand(tkv, hkv * hd, 1.0), rand(tkv, hkv * hd, 1.0), hq, hkv, hd) for tq, tkv, hq, hkv, hd in
            ((87, 956, 36, 12, 128), (1024, 1024, 12, 12, 64), (51, 867, 8, 1, 256), (300, 64, 16, 16, 128))]
    calls = [lambda a=a, w=w, f=f: api.op_linear(a, w, out_bf16=not f) for a, w, f in linear] + [lambda x=x: api.op_attention(*x) for x in attn]
    want = [f() for f in calls]
    torch.cuda.synchronize()
    for i in range(40):
        order = torch.randperm(len(calls), generator=torch.Generator().manual_seed(i)).tolist()
        got = [calls[j]() for j in order]
        assert all(torch.equal(x, want[j]) for x, j in zip(got, order)), i
    assert api.op_status(api.OP_LINEAR) == api.VLA_OK


def test_captured_calls_follow_their_inputs():
    """Tiles of two SMs and attention over clusters of three CTAs in one graph: a replay computes from what the inputs hold then."""
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(1)
    a = torch.randn(1747, 2288, device="cuda", generator=g).to(torch.bfloat16)
    w = (2288 ** -0.5 * torch.randn(2064, 2288, device="cuda", generator=g)).to(torch.bfloat16)
    q, k, v = (torch.randn(n, 36 * 128, device="cuda", generator=g).to(torch.bfloat16)[:, :c].contiguous() for n, c in ((87, 4608), (956, 1536), (956, 1536)))
    scratch = torch.empty(api.op_attention_scratch_bytes(956, 12, 128), dtype=torch.uint8, device="cuda")

    def calls(stream=None):
        return (api.op_linear(a, w, act=1, out_bf16=True, stream=stream), api.op_linear(a, w, stream=stream),
                api.op_attention(q, k, v, 36, 12, 128, scratch=scratch, stream=stream))
    calls()
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        out = calls(side)
    for _ in range(2):
        for x in (a, q, k):
            x.copy_(x.flip(0))
        want = calls()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(out, want))
    assert api.op_status(api.OP_LINEAR) == api.VLA_OK and api.op_status(api.OP_ATTENTION, scratch) == api.VLA_OK
