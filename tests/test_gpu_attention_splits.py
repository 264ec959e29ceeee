"""Stand-alone attention whose keys are shared by clusters of two to eight CTAs: every split, heads folded and not, each number of
score buffers, a last block of one key, causal tiles some of whose CTAs have no key to look at, and values that only a common
maximum keeps in range."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tq,tkv,hq,hkv,hd,causal", [
    (1024, 1024, 12, 12, 64, False), (725, 687, 12, 12, 128, False), (87, 956, 36, 12, 128, False), (1538, 457, 5, 5, 128, False),
    (339, 1208, 8, 4, 64, False), (1456, 1546, 2, 2, 64, False), (88, 1623, 12, 12, 64, False), (28, 864, 16, 16, 80, False),
    (51, 867, 8, 1, 256, False), (51, 833, 8, 1, 256, False), (300, 1025, 4, 4, 32, False), (70, 1985, 3, 1, 192, False), (9, 2048, 1, 1, 16, False),
    (691, 691, 3, 1, 128, True), (1918, 1918, 4, 4, 256, True), (556, 556, 5, 5, 128, True), (65, 65, 1, 1, 64, True), (513, 513, 2, 2, 96, True)])
@pytest.mark.parametrize("scale", [1.5, 12.0])
def test_against_64_bit(tq, tkv, hq, hkv, hd, causal, scale):
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(tq + tkv)

    def rand(rows, cols, s):
        return (s * torch.randn(rows, cols, device="cuda", generator=g)).to(torch.bfloat16)
    q, k, v = rand(tq, hq * hd, scale), rand(tkv, hkv * hd, 1.5), rand(tkv, hkv * hd, 1.0)
    got = api.op_attention(q, k, v, hq, hkv, hd, causal=causal)
    qs, ks, vs = (x.double().view(x.shape[0], -1, hd).transpose(0, 1) for x in (q, k, v))
    ks, vs = (x.repeat_interleave(hq // hkv, 0) for x in (ks, vs))
    s = qs @ ks.transpose(1, 2) / hd ** 0.5
    if causal:
        s = s.masked_fill(torch.ones(tq, tkv, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = (s.softmax(-1) @ vs).transpose(0, 1).reshape(tq, hq * hd)
    err = float((got.double() - ref).norm() / ref.norm())
    # probabilities and results are rounded to bf16 (2^-9 each, at most), exponentials to 2^-11 or so: a little under 2^-8 together
    assert err <= 2.0 ** -8, err
    assert torch.isfinite(got.float()).all()
    assert torch.equal(got, api.op_attention(q, k, v, hq, hkv, hd, causal=causal))


@pytest.mark.parametrize("tq,tkv,hq,hkv,hd", [
    (1024, 512, 48, 48, 64), (90, 900, 4, 4, 64), (51, 867, 8, 1, 256), (87, 956, 36, 12, 128), (9, 300, 4, 2, 64)])
def test_nan_is_not_lost(tq, tkv, hq, hkv, hd):
    """A row whose scores are NaN is NaN whether its keys are split or not, and where only some of the parts hold a NaN; others are as without it."""
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(tq)
    q, k, v = ((torch.randn(n, h * hd, device="cuda", generator=g)).to(torch.bfloat16) for n, h in ((tq, hq), (tkv, hkv), (tkv, hkv)))
    clean = api.op_attention(q, k, v, hq, hkv, hd).view(tq, hq, hd)
    bad = q.clone()
    bad.view(tq, hq, hd)[tq // 2, hq - 1] = float("nan")
    got = api.op_attention(bad, k, v, hq, hkv, hd).view(tq, hq, hd)
    assert torch.isnan(got[tq // 2, hq - 1]).all()
    keep = torch.ones(tq, hq, dtype=torch.bool, device="cuda")
    keep[tq // 2, hq - 1] = False
    assert torch.equal(got[keep], clean[keep])
    for keys in (slice(0, 64), slice(0, tkv // 2), slice(tkv - 1, tkv)):
        bad = k.clone()
        bad.view(tkv, hkv, hd)[keys, 0] = float("nan")
        got = api.op_attention(q, bad, v, hq, hkv, hd).view(tq, hq, hd)
        assert torch.isnan(got[:, :hq // hkv]).all(), keys
        assert torch.equal(got[:, hq // hkv:], clean[:, hq // hkv:])
