"""The linear layer's result rows: widths and addresses that allow stores of eight features, of two, or of one, give the same
values, and nothing outside the result is written."""
import numpy as np
import pytest

from oracle import vla_oracle as O
from vla_synth.gen import round_to_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k", [(50, 136), (300, 64)])
@pytest.mark.parametrize("n", [1, 2, 24, 28, 30, 33, 260, 514, 1001])
def test_widths_and_addresses(m, n, k):
    import torch
    from paper_2609_22335_b200 import api
    lib = api.load_library()
    rng = np.random.default_rng(m + n)
    a = round_to_bf16(rng.standard_normal((m, k)).astype(np.float32))
    w = round_to_bf16((k ** -0.5 * rng.standard_normal((n, k))).astype(np.float32))
    ref = O.linear(a.astype(np.float64), w.astype(np.float64))
    da, dw = (torch.from_numpy(x).cuda().to(torch.bfloat16) for x in (a, w))
    for off in (0, 1, 2, 4):                                 # elements the result starts behind an aligned address
        o32 = torch.full((m * n + 16,), 7.0, dtype=torch.float32, device="cuda")
        o16 = torch.full((m * n + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
        rc = lib.vla_op_linear(da.data_ptr(), dw.data_ptr(), o32.data_ptr() + 4 * off, o16.data_ptr() + 2 * off, m, n, k, 0, None)
        assert rc == api.VLA_OK and api.op_status(api.OP_LINEAR) == api.VLA_OK
        got = o32[off:off + m * n].reshape(m, n)
        assert np.abs(got.cpu().numpy() - ref).max() <= 2.0 ** -23 * (k / 16 + 2) * np.abs(ref).max()    # a unit in the last place per 16 products
        assert torch.equal(o16[off:off + m * n].reshape(m, n), got.to(torch.bfloat16))
        for o in (o32, o16):
            assert (o[:off] == 7).all() and (o[off + m * n:] == 7).all()


@pytest.mark.parametrize("m,n,k", [
    (129, 4833, 64), (129, 4790, 64), (129, 5925, 64), (129, 7154, 64),               # widths 48, 80, 96, 112
    (300, 6284, 72), (4000, 578, 64), (300, 8038, 64), (4000, 733, 72), (4000, 784, 72), (800, 4388, 72), (4000, 923, 72),   # 144 .. 240
    (129, 4756, 1992),                                                                # (fp32: tiles of two SMs)
    (288, 11008, 4096), (572, 6298, 1616), (257, 2370, 2056)])                        # K shared by two and four CTAs, for fp32 results only
def test_widths_that_are_no_power_of_two(m, n, k):
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(n)
    a = torch.randn(m, k, device="cuda", generator=g).to(torch.bfloat16)
    w = (k ** -0.5 * torch.randn(n, k, device="cuda", generator=g)).to(torch.bfloat16)
    ref = a.double() @ w.double().T
    sums = 2.0 ** -23 * (k / 16 + 2) * float(ref.abs().max())          # a unit in the last place per 16 products
    assert float((api.op_linear(a, w).double() - ref).abs().max()) <= sums
    assert bool(((api.op_linear(a, w, out_bf16=True).double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 2 * sums).all())
