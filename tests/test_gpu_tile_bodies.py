"""The engine's GEMM and attention tile bodies, operator by operator, against the CPU oracle (fp64) on the same
bf16-representable inputs: the stand-alone operators are kernels of their own and say nothing about these.  Both epilogues of
the GEMM tile, gated rows, addends under the accumulators and behind the product; attention over one and two key segments, folded heads, causal and
suffix masks; and the waits inside the bodies, which run out and are reported."""
import numpy as np
import pytest

from oracle import vla_oracle as O
from vla_synth.gen import round_to_bf16

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda().to(torch.bfloat16)


def _rand(rng, shape, scale=1.0):
    return round_to_bf16((scale * rng.standard_normal(shape)).astype(np.float32))


def _engine_rows(w):
    """Weight rows as the engine keeps them: padded to a multiple of 32 and reordered within each 32."""
    rows = -(-w.shape[0] // 32) * 32
    p = np.arange(32)
    feature = 8 * ((p >> 1) & 3) + 2 * (p >> 3) + (p & 1)
    padded = np.zeros((rows, w.shape[1]), w.dtype)
    padded[:w.shape[0]] = w
    return padded.reshape(-1, 32, w.shape[1])[:, feature].reshape(rows, w.shape[1])


def _act(act, x):
    return [x, O.gelu_tanh(x), O.silu(x)][act]


def _check(got, ref, bf16):
    """fp32 sums of exact bf16 products; activations use hardware approximations (~2^-11 relative); bf16 rows are rounded once."""
    got = got.float().cpu().numpy().astype(np.float64)
    tol = (2e-3 + (2 ** -8 if bf16 else 0)) * np.abs(ref).max() + 1e-5
    assert np.max(np.abs(got - ref)) <= tol, (np.max(np.abs(got - ref)), tol)
    assert np.linalg.norm(got - ref) <= (2.0 ** -8 if bf16 else 1e-3) * np.linalg.norm(ref)


GEMM_SHAPES = [(1, 7, 8), (9, 128, 64), (51, 720, 1024), (64, 264, 192), (65, 256, 192), (176, 960, 2560), (288, 300, 1000),
               (1024, 384, 768), (257, 129, 72)]


@pytest.mark.parametrize("m,n,k", GEMM_SHAPES)
@pytest.mark.parametrize("act", [0, 1, 2])
def test_gemm_tile_general_epilogue(m, n, k, act):
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(m * 1000 + n + k)
    a, w = _rand(rng, (m, k)), _rand(rng, (n, k), 0.05)
    ref = _act(act, O.linear(a.astype(np.float64), w.astype(np.float64)))
    o32, o16 = api.debug_tile_linear(_dev(a), _dev(w), n, act=act, out16=True)
    _check(o32, ref, False)
    _check(o16, ref, True)


@pytest.mark.parametrize("m,n,k", [(m, -(-n // 8) * 8, k) for m, n, k in GEMM_SHAPES])
def test_gemm_tile_straight_epilogue(m, n, k):
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(m * 1000 + n + k)
    a, w = _rand(rng, (m, k)), _rand(rng, (n, k), 0.05)
    ref = O.linear(a.astype(np.float64), w.astype(np.float64))
    da, dw = _dev(a), _dev(_engine_rows(w))
    _check(api.debug_tile_linear(da, dw, n, fast=True)[0], ref, False)
    o32, o16 = api.debug_tile_linear(da, dw, n, fast=True, out16=True)
    _check(o32, ref, False)
    _check(o16, ref, True)
    _check(api.debug_tile_linear(da, dw, n, act=1, fast=True, out32=False, out16=True)[1], _act(1, ref), True)


@pytest.mark.parametrize("m,n,k", [(1, 8, 8), (9, 136, 64), (50, 2048, 720), (65, 100, 192), (130, 516, 256)])
@pytest.mark.parametrize("act", [1, 2])
@pytest.mark.parametrize("fast", [False, True])
def test_gemm_tile_gated(m, n, k, act, fast):
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(m + n + k)
    a, gate, up = _rand(rng, (m, k)), _rand(rng, (n, k), k ** -0.5), _rand(rng, (n, k), k ** -0.5)
    w = np.stack([gate, up], axis=1).reshape(2 * n, k)
    a64 = a.astype(np.float64)
    ref = _act(act, O.linear(a64, gate.astype(np.float64))) * O.linear(a64, up.astype(np.float64))
    got = api.debug_tile_linear(_dev(a), _dev(_engine_rows(w) if fast else w), n, act=act, gated=True, fast=fast, out32=False, out16=True)[1]
    _check(got, ref, True)


@pytest.mark.parametrize("m,n,k", [(1, 8, 64), (50, 720, 960), (64, 136, 2048), (1024, 768, 3072), (129, 72, 64)])
@pytest.mark.parametrize("scale", [1.0, 64.0])
@pytest.mark.parametrize("fast", [False, True])
def test_gemm_tile_addend(m, n, k, scale, fast):
    """out = a w^T + x: both epilogues add behind the product.  An fp32 sum of k products of two bf16 values next to an addend of up to
    `scale` times their size: every step may lose one unit in the last place of the larger, 2^-23 of it, and the tensor core adds 16
    products a step; the straight epilogue's single rounding is what test_gemm_tile_residual_is_rounded_once holds it to."""
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(m + n + k)
    a, w = _rand(rng, (m, k)), _rand(rng, (n, k), k ** -0.5)
    x = (scale * rng.standard_normal((m, n))).astype(np.float32)
    ref = O.linear(a.astype(np.float64), w.astype(np.float64)) + x
    got = api.debug_tile_linear(_dev(a), _dev(_engine_rows(w) if fast else w), n, x=torch.from_numpy(x).cuda(), fast=fast)[0]
    err = np.abs(got.cpu().numpy() - ref)
    print(f"addend {scale:g} x product, k = {k}, {'straight' if fast else 'general'} epilogue: rel-L2 {np.linalg.norm(err) / np.linalg.norm(ref):.3g}")
    assert err.max() <= 2.0 ** -23 * (k / 16 + 2) * np.abs(ref).max()


ADDEND_SHAPES = [(1, 8, 64), (17, 136, 64), (50, 720, 960), (64, 136, 2048), (65, 40, 192), (129, 72, 64), (300, 384, 512), (1024, 768, 3072)]


def _f32(rng, shape, scale=1.0):
    return (scale * rng.standard_normal(shape)).astype(np.float32)


@pytest.mark.parametrize("m,n,k", ADDEND_SHAPES)
@pytest.mark.parametrize("scale", [1.0, 64.0])
@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("mirror", [False, True])
def test_gemm_tile_residual_is_rounded_once(m, n, k, scale, in_place, mirror):
    """x + a w^T with the straight epilogue, into rows of its own and in place, alone and with the bf16 mirror and the sums of squares that the
    next norm reads.  The product's sums are exact to a unit in the last place per 16 products at the product's own size, however large x is,
    and the one addition behind them rounds by half a unit of the result; the mirror is the fp32 rows' rounding, and a partial sum of 128
    squares (32 in a lane, two exchanges, all positive) loses at most 36 half units."""
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(m + n + k)
    a, w, x = _rand(rng, (m, k)), _rand(rng, (n, k), k ** -0.5), _f32(rng, (m, n), scale)
    product = O.linear(a.astype(np.float64), w.astype(np.float64))
    ref = product + x
    o32, o16, ss = api.debug_tile_addends(_dev(a), _dev(_engine_rows(w)), n, x=torch.from_numpy(x).cuda(), out16=mirror, ss=mirror, in_place=in_place)
    got = o32.cpu().numpy().astype(np.float64)
    assert (np.abs(got - ref) <= 2.0 ** -23 * (k / 16 + 2) * np.abs(product).max() + 2.0 ** -24 * np.abs(ref)).all()
    if mirror:
        assert torch.equal(o16, o32.to(torch.bfloat16))
        squares = np.add.reduceat(got ** 2, np.arange(0, n, 128), axis=1)
        assert (np.abs(ss.cpu().numpy() - squares) <= 36 * 2.0 ** -24 * squares).all()


@pytest.mark.parametrize("m,n,k", ADDEND_SHAPES)
@pytest.mark.parametrize("terms", ["b", "v", "t", "u", "bv", "tu", "bvtu"])
def test_gemm_tile_addends_under_the_accumulators(m, n, k, terms):
    """Bias, broadcast vector and tables lie in the accumulators before the first MMA: alone, together, and with residual rows behind the
    product.  The sums then start from them: a unit in the last place of the largest partial sum per 16 products and per addend."""
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(m + n + k + len(terms))
    a, w, x = _rand(rng, (m, k)), _rand(rng, (n, k), k ** -0.5), _f32(rng, (m, n), 4.0)
    under = {"b": _f32(rng, n), "v": _f32(rng, n), "t": _f32(rng, (m, n)), "u": _f32(rng, (m, n))}
    names = {"b": "bias", "v": "vec", "t": "tab", "u": "tab2"}
    args = {names[t]: torch.from_numpy(under[t]).cuda() for t in terms}
    product = O.linear(a.astype(np.float64), w.astype(np.float64))
    added = sum(under[t].astype(np.float64) for t in terms)
    ref = product + added
    sums = 2.0 ** -23 * (k / 16 + 2 + len(terms)) * (np.abs(product).max() + np.abs(added).max())
    da, dw = _dev(a), _dev(_engine_rows(w))
    o32, o16, ss = api.debug_tile_addends(da, dw, n, out16=True, ss=True, **args)
    got = o32.cpu().numpy().astype(np.float64)
    assert (np.abs(got - ref) <= sums).all()
    assert torch.equal(o16, o32.to(torch.bfloat16))
    squares = np.add.reduceat(got ** 2, np.arange(0, n, 128), axis=1)
    assert (np.abs(ss.cpu().numpy() - squares) <= 36 * 2.0 ** -24 * squares).all()
    assert torch.equal(api.debug_tile_addends(da, dw, n, out32=False, out16=True, **args)[1], o16)
    both = api.debug_tile_addends(da, dw, n, x=torch.from_numpy(x).cuda(), **args)[0].cpu().numpy()
    assert (np.abs(both - (ref + x)) <= sums + 2.0 ** -24 * np.abs(ref + x)).all()
    if terms == "b":
        _check(api.debug_tile_addends(da, dw, n, act=1, out32=False, out16=True, **args)[1], _act(1, ref), True)


ATTENTION_SHAPES = [
    (9, 80, 4, 4, 64, False), (50, 226, 15, 5, 64, False), (1024, 1024, 12, 12, 64, False), (17, 17, 16, 16, 64, False),
    (96, 96, 16, 8, 128, False), (300, 300, 8, 1, 256, False), (288, 288, 4, 4, 128, True), (130, 130, 2, 2, 32, True),
    (1, 1, 1, 1, 16, False), (256, 193, 3, 3, 80, False), (200, 200, 2, 2, 64, True), (129, 129, 1, 1, 256, True),
    (51, 867, 8, 1, 256, False), (9, 80, 4, 2, 64, False), (17, 40, 6, 1, 64, False), (30, 30, 4, 2, 32, True),
    (64, 100, 6, 3, 128, False)]


def _check_attention(got, ref):
    """P is rounded to bf16 before P V and the output is bf16: 2^-8 relative each."""
    got = got.float().cpu().numpy().astype(np.float64).reshape(ref.shape)
    assert np.max(np.abs(got - ref)) <= 2e-2 * max(1.0, np.abs(ref).max())
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1e-2


@pytest.mark.parametrize("tq,tkv,hq,hkv,hd,causal", ATTENTION_SHAPES)
def test_attention_tile(tq, tkv, hq, hkv, hd, causal):
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(tq * 7 + tkv + hd)
    q, k, v = _rand(rng, (tq, hq, hd), 1.5), _rand(rng, (tkv, hkv, hd), 1.5), _rand(rng, (tkv, hkv, hd))
    ref = O.attention(q.astype(np.float64), k.astype(np.float64), v.astype(np.float64), causal=causal)
    _check_attention(api.debug_tile_attention(_dev(q.reshape(tq, -1)), _dev(k.reshape(tkv, -1)), _dev(v.reshape(tkv, -1)), hq, hkv, hd,
                                              causal=causal), ref)


@pytest.mark.parametrize("tq,t0,t1,hq,hkv,hd,sfx", [
    (50, 176, 50, 15, 5, 64, 0), (51, 816, 51, 8, 1, 256, 0), (1, 1, 1, 1, 1, 16, 0), (64, 64, 65, 4, 4, 64, 0), (130, 63, 130, 2, 1, 80, 0),
    (50, 176, 50, 15, 5, 64, 1), (51, 100, 51, 8, 1, 256, 2), (130, 63, 130, 2, 2, 80, 70)])
def test_attention_tile_two_segments_and_suffix_mask(tq, t0, t1, hq, hkv, hd, sfx):
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(tq + t0 + t1 + sfx)
    q, k, v = _rand(rng, (tq, hq, hd), 1.5), _rand(rng, (t0 + t1, hkv, hd), 1.5), _rand(rng, (t0 + t1, hkv, hd))
    visible = np.ones((tq, t0 + t1), bool)
    if sfx:
        visible[:sfx, t0 + sfx:] = False
    ref = O.attention(q.astype(np.float64), k.astype(np.float64), v.astype(np.float64), visible=visible)
    seg = lambda x, lo, hi: _dev(x[lo:hi].reshape(hi - lo, -1))
    got = api.debug_tile_attention(_dev(q.reshape(tq, -1)), seg(k, 0, t0), seg(v, 0, t0), hq, hkv, hd, k1=seg(k, t0, t0 + t1), v1=seg(v, t0, t0 + t1), sfx=sfx)
    _check_attention(got, ref)


def test_waits_inside_the_tile_bodies_run_out_and_are_reported():
    """With the operand loads switched off the consumers' bounded waits run out, the node returns and says so; switched back on,
    the same calls are correct."""
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(2)
    a, w = _rand(rng, (40, 192)), _rand(rng, (96, 192), 0.1)
    q, k, v = _rand(rng, (20, 2, 64)), _rand(rng, (200, 2, 64)), _rand(rng, (200, 2, 64))
    linear = lambda: api.debug_tile_linear(_dev(a), _dev(_engine_rows(w)), 96, fast=True)[0]
    attention = lambda: api.debug_tile_attention(_dev(q.reshape(20, -1)), _dev(k.reshape(200, -1)), _dev(v.reshape(200, -1)), 2, 2, 64)
    api.debug_op_fault(True, wait_limit_ns=1_000_000)        # 1 ms
    try:
        for call in (linear, attention):
            with pytest.raises(api.VlaError) as e:
                call()
            assert e.value.code == api.VLA_ERR_TIMEOUT
    finally:
        api.debug_op_fault(False)
    _check(linear(), O.linear(a.astype(np.float64), w.astype(np.float64)), False)
    _check_attention(attention(), O.attention(q.astype(np.float64), k.astype(np.float64), v.astype(np.float64)))


def test_hooks_refuse_what_the_straight_epilogue_cannot_take():
    import torch
    from paper_2609_22335_b200 import api
    lib = api.load_library()
    t = torch.zeros(64, 64, dtype=torch.bfloat16, device="cuda").data_ptr()
    o = torch.zeros(64, 64, dtype=torch.float32, device="cuda").data_ptr()
    bad = api.VLA_ERR_INVALID
    assert lib.vla_debug_tile_linear(t, t, None, o, None, 64, 60, 64, 0, 0, 1) == bad        # width
    assert lib.vla_debug_tile_linear(t, t, None, o + 16, None, 8, 64, 64, 0, 0, 1) == bad    # rows of fp32 that are not 32-byte aligned
    assert lib.vla_debug_tile_linear(t, t, o, o, None, 64, 64, 64, 1, 0, 1) == bad           # activation behind an addend
    assert lib.vla_debug_tile_linear(t, t, o, None, t, 64, 64, 64, 0, 0, 1) == bad           # addend without fp32 rows
    assert lib.vla_debug_tile_linear(t, t, None, o, None, 64, 64, 64, 0, 1, 0) == bad        # gated rows are bf16
    assert lib.vla_debug_tile_addends(t, t, None, o, o, None, None, None, t, None, 64, 64, 64, 1) == bad     # activation behind a broadcast vector
    assert lib.vla_debug_tile_addends(t, t, None, o + 4, None, None, None, o, None, None, 8, 64, 64, 0) == bad    # bias that is not 16-byte aligned
    assert lib.vla_debug_tile_addends(t, t, None, None, None, None, None, o, None, o, 64, 64, 64, 0) == bad  # sums of squares without the mirror
    assert lib.vla_debug_tile_attention(t, t, t, None, None, t, 64, 64, 8, 1, 1, 64, 0, 0) == bad    # a second segment without its keys
    assert lib.vla_debug_tile_attention(t, t, t, None, None, t, 32, 64, 0, 1, 1, 64, 1, 0) == bad    # causal needs tq == t0
