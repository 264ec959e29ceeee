"""Stand-alone attention is as close to 64 bits as probabilities of one bf16 number are with the keys in powers of two of parts that
fill the chip, however many parts the call's plan takes."""
import pytest

pytestmark = pytest.mark.gpu


def _emulated(q, k, v, causal, parts):
    """64-bit attention but for what such a kernel rounds: probabilities (relative to a running maximum that may lag by 2^8, one per part
    of the keys) and results to bf16.  [heads, tokens, head dim]."""
    import torch
    s = q @ k.transpose(1, 2) * (1.4426950408889634 / q.shape[-1] ** 0.5)
    if causal:
        s = s.masked_fill(torch.ones(s.shape[1:], dtype=torch.bool, device=s.device).triu(1), float("-inf"))
    blocks, done = -(-s.shape[2] // 64), []
    for r in range(parts):
        m = torch.full(s.shape[:2], float("-inf"), dtype=torch.double, device=s.device)
        l, o = torch.zeros_like(m), torch.zeros(q.shape[0], q.shape[1], v.shape[-1], dtype=torch.double, device=s.device)
        for b in range(blocks * r // parts, blocks * (r + 1) // parts):
            x = s[:, :, 64 * b:64 * b + 64]
            top = x.max(-1).values
            new = torch.where((m > float("-inf")) & (top - m <= 8), m, torch.maximum(m, top))
            alpha = torch.where(m > float("-inf"), torch.exp2(m - new), torch.zeros_like(m))
            p = torch.exp2(x - torch.where(new > float("-inf"), new, torch.zeros_like(new))[..., None])
            l = l * alpha + p.sum(-1)
            o = o * alpha[..., None] + p.to(torch.bfloat16).double() @ v[:, 64 * b:64 * b + 64]
            m = new
        done.append((m, l, o))
    top = torch.stack([m for m, _, _ in done]).max(0).values
    w = [torch.exp2(m - top) for m, _, _ in done]
    out = sum(f[..., None] * o for f, (_, _, o) in zip(w, done)) / sum(f * l for f, (_, l, _) in zip(w, done))[..., None]
    return out.to(torch.bfloat16).double(), s


# (tokens, keys, heads, KV heads, head width, causal, parts): powers of two up to two CTAs per SM (one above a width of 128)
@pytest.mark.parametrize("tq,tkv,hq,hkv,hd,causal,parts", [
    (87, 956, 36, 12, 128, False, 8), (725, 687, 12, 12, 128, False, 4), (51, 867, 8, 1, 256, False, 8), (1070, 120, 4, 4, 128, False, 2),
    (95, 309, 48, 16, 128, False, 4), (346, 524, 4, 4, 80, False, 8), (1, 128, 8, 8, 128, False, 2), (319, 640, 8, 4, 128, False, 8),
    (420, 420, 16, 2, 64, True, 4), (435, 230, 36, 12, 80, False, 2), (1024, 1024, 12, 12, 64, False, 2), (1813, 1813, 4, 4, 64, True, 4),
    (3, 120, 40, 5, 256, False, 2), (450, 450, 64, 32, 128, True, 1)])
def test_no_further_from_64_bits(tq, tkv, hq, hkv, hd, causal, parts):
    import torch
    from paper_2609_22335_b200 import api
    g = torch.Generator(device="cuda").manual_seed(tq + tkv)

    def rand(rows, cols, s):
        return (s * torch.randn(rows, cols, device="cuda", generator=g)).to(torch.bfloat16)
    q, k, v = rand(tq, hq * hd, 1.5), rand(tkv, hkv * hd, 1.5), rand(tkv, hkv * hd, 1.0)
    got = api.op_attention(q, k, v, hq, hkv, hd, causal=causal).double().view(tq, hq, hd).transpose(0, 1)
    qs, ks, vs = (x.double().view(x.shape[0], -1, hd).transpose(0, 1) for x in (q, k, v))
    ks, vs = (x.repeat_interleave(hq // hkv, 0) for x in (ks, vs))
    emulated, s = _emulated(qs, ks, vs, causal, parts)
    ref = (s * 0.6931471805599453).softmax(-1) @ vs
    err, bound = (float((x - ref).norm() / ref.norm()) for x in (got, emulated))
    print(f"rel-L2 {err:.4g}, {parts} parts of one-term probabilities {bound:.4g}")
    # both hold the same roundings of some thousand to a million results: their norms differ by less than 2 %
    assert err <= 1.02 * bound, (err, bound)
