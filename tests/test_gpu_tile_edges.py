"""Shapes at the edges of the kernels' dispatch rules, against the CPU oracle: the linear layer's tile heights and widths, split
K over a cluster and more tiles than the chip holds at once; attention's key blocks dealt out over a cluster; GEMM tiles on
either side of 64 tokens, widths that are no multiple of 32, and the one-feature-wide remains of a tile in the engine; calls
that start behind one another's last tiles."""
import numpy as np
import pytest

from oracle import vla_oracle as O
from vla_synth.configs import CFG1, CFG2, CFG4, mini
from vla_synth.gen import make_weights, frame_inputs, round_to_bf16

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda().to(torch.bfloat16)


def _rand(rng, shape, scale=1.0):
    return round_to_bf16((scale * rng.standard_normal(shape)).astype(np.float32))


@pytest.mark.parametrize("m,n,k", [
    (16, 16, 8), (17, 33, 8), (63, 31, 64), (64, 32, 72), (65, 40, 128),      # one k-block; heights around 64; widths around 32
    (50, 720, 2048), (50, 721, 2048), (1, 16, 4096), (128, 128, 8192),        # few tiles, long K: a cluster shares it
    (129, 257, 1024), (300, 1000, 264), (2500, 1032, 136), (9000, 520, 64),            # remainders; several tiles to a block
    (4100, 2500, 136), (7000, 1801, 72)])                                     # widths between 128 and 256
@pytest.mark.parametrize("act,bf16", [(0, False), (1, True), (2, False)])
def test_linear_at_tile_edges(m, n, k, act, bf16):
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(m + 3 * n + k)
    a, w = _rand(rng, (m, k)), _rand(rng, (n, k), k ** -0.5)
    ref = O.linear(a.astype(np.float64), w.astype(np.float64))
    ref = [ref, O.gelu_tanh(ref), O.silu(ref)][act]
    got = api.op_linear(_dev(a), _dev(w), act=act, out_bf16=bf16)
    torch.cuda.synchronize()
    got = got.float().cpu().numpy().astype(np.float64)
    tol = (2e-3 + (2 ** -8 if bf16 else 0)) * np.abs(ref).max() + 1e-5
    assert np.max(np.abs(got - ref)) <= tol, (np.max(np.abs(got - ref)), tol)


@pytest.mark.parametrize("tq,tkv,hq,hkv,hd,causal", [
    (1, 64, 1, 1, 64, False), (1, 65, 1, 1, 16, False), (3, 2000, 2, 2, 64, False),       # one row; keys split over a cluster
    (51, 867, 8, 1, 256, False), (128, 513, 2, 1, 256, False), (129, 129, 1, 1, 256, True),
    (127, 127, 3, 3, 80, True), (640, 640, 2, 2, 128, True), (200, 1025, 16, 4, 80, False), (1500, 1500, 20, 20, 64, True)])
def test_attention_at_block_edges(tq, tkv, hq, hkv, hd, causal):
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(tq + tkv + hd)
    q, k, v = _rand(rng, (tq, hq, hd), 1.5), _rand(rng, (tkv, hkv, hd), 1.5), _rand(rng, (tkv, hkv, hd))
    ref = O.attention(q.astype(np.float64), k.astype(np.float64), v.astype(np.float64), causal=causal).reshape(tq, -1)
    dq, dk, dv = _dev(q.reshape(tq, -1)), _dev(k.reshape(tkv, -1)), _dev(v.reshape(tkv, -1))
    got = api.op_attention(dq, dk, dv, hq, hkv, hd, causal=causal)
    out = torch.empty_like(dq)
    try:
        api.op_attention_static(dq, dk, dv, out, hq, hkv, hd, causal=causal)
    except api.VlaError:                                     # more scratch than the fixed array holds
        out = got
    torch.cuda.synchronize()
    assert torch.equal(out, got)
    err = np.abs(got.float().cpu().numpy() - ref)
    assert err.max() <= 2e-2 * max(1.0, np.abs(ref).max()), err.max()
    assert np.linalg.norm(err) / np.linalg.norm(ref) < 1e-2


@pytest.mark.parametrize("t,hq,hd", [(1500, 20, 64), (640, 2, 128)])
def test_attention_repeats_itself(t, hq, hd):
    """Causal masks put a tile's warps a block apart; the last P V must be waited for all the same."""
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(t)
    q, k, v = (_dev(_rand(rng, (t, hq * hd), 1.5)) for _ in range(3))
    first = api.op_attention(q, k, v, hq, hq, hd, causal=True)
    for _ in range(200):
        assert torch.equal(api.op_attention(q, k, v, hq, hq, hd, causal=True), first)


@pytest.mark.parametrize("m,n", [(1, 64), (50, 256), (300, 1024)])
def test_calls_that_follow_one_another_see_each_others_results(m, n):
    """A call's kernel sets up while the previous one still runs; what it reads must be that one's finished output."""
    import torch
    from paper_2609_22335_b200 import api
    rng = np.random.default_rng(n)
    w = _dev(_rand(rng, (n, n), n ** -0.5))
    x0 = _dev(_rand(rng, (m, n)))

    def chain(wait):
        x = x0
        for _ in range(12):
            x = api.op_linear(x, w, act=0, out_bf16=True)
            if wait:
                torch.cuda.synchronize()
            x = api.op_attention(x, x, x, n // 64, n // 64, 64)
            if wait:
                torch.cuda.synchronize()
            x = x * 2.0                                      # another library's kernel in between
        torch.cuda.synchronize()
        return x

    want = chain(True)
    for _ in range(3):
        assert torch.equal(chain(False), want)


SMALL2 = dict(img=128, vis_layers=1, llm_layers=2, act_layers=2, n_steps=2, vocab=2048, n_streams=1, n_frames=2)
SMALL4 = dict(n_cam=1, img=112, vis_layers=1, llm_layers=2, act_layers=2, mlp=1024, n_steps=2, vocab=2048, n_streams=1, n_frames=2)
ENGINE = {
    # head tiles on either side of 64 and of 128 tokens, and of one token
    "tokens1": mini(CFG4, horizon=1, **SMALL4),
    "tokens63": mini(CFG2, horizon=63, **SMALL2),
    "tokens64": mini(CFG2, horizon=64, **SMALL2),
    "tokens65": mini(CFG2, horizon=65, **SMALL2),
    "tokens129": mini(CFG2, horizon=129, **SMALL2),
    # widths that leave a ragged last group of 32 or of 128 features, gated and plain, with and without rotary rows
    "widths2": mini(CFG2, mlp=1000, act_mlp=264, vis_mlp=808, act_dim=33, **SMALL2),
    "widths4": mini(CFG4, **{**SMALL4, "mlp": 520}, act_mlp=136, act_dim=7),
    "widths1": mini(CFG1, mlp=72, act_mlp=200, act_dim=1, n_streams=1, n_frames=2),
}


@pytest.mark.parametrize("key", list(ENGINE))
def test_engine_at_tile_edges(key):
    from paper_2609_22335_b200 import Engine
    m = ENGINE[key]
    w = make_weights(m, seed=0)
    frames = [[frame_inputs(m, r, n, seed=3) for n in range(m.n_frames)] for r in range(m.n_streams)]
    outs = []
    for mode in ("serial", "cosched"):
        eng = Engine(m, mode=mode, n_streams=m.n_streams)
        try:
            eng.load_weights(w)
            outs.append(eng.run(frames))
        finally:
            eng.close()
    for r in range(m.n_streams):
        for n in range(m.n_frames):
            assert np.array_equal(outs[0][r][n], outs[1][r][n])
            ref = O.action_chunk(m, w, frames[r][n], np.float32)
            assert np.linalg.norm(outs[0][r][n] - ref) <= 1e-2 * np.linalg.norm(ref)
            assert np.max(np.abs(outs[0][r][n] - ref)) <= 3e-2 * max(1.0, float(np.sqrt(np.mean(ref * ref))))
