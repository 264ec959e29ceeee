"""What a program that uses this package has it do: the cases whose speed counts.

Two kinds of use.  A robot fleet's server keeps one ``Engine`` per model and streams frames through it
(``kind = "engine"``): one frame of one robot, where every microsecond of the chain of small dependent steps is
reaction time, up to a full set of request streams, where throughput counts.  And a program that wants the kernels
without the frame pipeline calls the operators on its own tensors (``kind = "linear"`` and ``"attention"``).

Model shapes are the repository's five workloads; operator shapes are the contractions of those workloads.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2609_22335_b200 import Engine, api
from paper_2609_22335_b200.workload_math import chunk_work
from vla_synth.configs import get_config, is_gain, weight_shapes

DEVICE = "cuda:0"


def listed():
    return [
        # The tiny workload, one frame: nothing but launches, hand-overs and host calls.
        {"name": "tiny_frame", "kind": "engine", "model": "cfg1", "streams": 1, "frames": 1, "inputs": "pageable"},
        # One robot waiting for its next actions: camera frames in page-locked buffers, one frame in flight.
        {"name": "smolvla_frame", "kind": "engine", "model": "cfg2", "streams": 1, "frames": 1, "inputs": "pinned"},
        # A few robots whose frames arrive as ordinary numpy arrays, two frames in flight each.
        {"name": "smolvla_few", "kind": "engine", "model": "cfg2", "streams": 4, "frames": 3, "inputs": "pageable"},
        # The benchmark's full load: 32 robots, frames already on the GPU.
        {"name": "smolvla_fleet", "kind": "engine", "model": "cfg2", "streams": 32, "frames": 4, "inputs": "device"},
        # Wide decoder layers before a diffusion transformer with adaptive norms and cross attention.
        {"name": "gr00t_streams", "kind": "engine", "model": "cfg3", "streams": 8, "frames": 3, "inputs": "device"},
        # Long prefix with rotary positions and one shared KV head of width 256.
        {"name": "pi0_streams", "kind": "engine", "model": "cfg4", "streams": 4, "frames": 2, "inputs": "pinned"},
        # One frame of the 7B model: its weights are read once for 288 tokens.
        {"name": "cogact_frame", "kind": "engine", "model": "cfg5", "streams": 1, "frames": 1, "inputs": "device"},
        # An action head's projection (50 action tokens): one pass over a small weight matrix.
        {"name": "linear_head", "kind": "linear", "m": 50, "n": 2048, "k": 720, "act": 0, "bf16": True},
        # A vision encoder's MLP over a batch of eight views.
        {"name": "linear_vision", "kind": "linear", "m": 8192, "n": 3072, "k": 768, "act": 1, "bf16": True},
        # A 7B decoder's gate projection over one prefix, fp32 result.
        {"name": "linear_prefix", "kind": "linear", "m": 288, "n": 11008, "k": 4096, "act": 2, "bf16": False},
        # A vision encoder layer's attention over one 1024-token view.
        {"name": "attention_vision", "kind": "attention", "tq": 1024, "tkv": 1024, "hq": 12, "hkv": 12, "hd": 64,
         "causal": False, "static": False},
        # An action head's joint attention: 51 queries, one shared KV head, ragged key count, no scratch of its own.
        {"name": "attention_head", "kind": "attention", "tq": 51, "tkv": 867, "hq": 8, "hkv": 1, "hd": 256,
         "causal": False, "static": True},
    ]


# ---------------------------------------------------------------- further cases of the same ranges
def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    most = work(listed()[3])["flops"]
    while True:
        kind = rng.choice(["engine", "engine", "linear", "attention"])
        if kind == "engine":
            model = rng.choice(["cfg1", "cfg2", "cfg3", "cfg4", "cfg5"])
            case = {"kind": kind, "model": model, "streams": _log_int(rng, 1, get_config(model).n_streams),
                    "frames": rng.randint(1, 6), "inputs": rng.choice(["pageable", "pinned", "device"])}
        elif kind == "linear":
            case = {"kind": kind, "m": _log_int(rng, 1, 8192), "n": _log_int(rng, 7, 16384), "k": 8 * _log_int(rng, 8, 1536),
                    "act": rng.choice([0, 0, 1, 2]), "bf16": rng.random() < 0.7}
        else:
            hd = rng.choice([32, 64, 64, 80, 128, 128, 256])
            hkv = rng.choice([1, 2, 4, 5, 8, 12, 16, 32])
            hq = hkv * rng.choice([1, 1, 2, 3, 8])
            tq, tkv = _log_int(rng, 1, 2048), _log_int(rng, 1, 2048)
            causal = rng.random() < 0.25
            tkv = tq if causal else tkv
            case = {"kind": kind, "tq": tq, "tkv": tkv, "hq": hq, "hkv": hkv, "hd": hd, "causal": causal,
                    "static": rng.random() < 0.3 and 2 * hkv * hd * (tkv + 63) <= 4 << 20}
            if hq > 64:
                continue
        if work(case)["flops"] <= most and all({k: v for k, v in c.items() if k != "name"} != case for c in listed()):
            return case


# ---------------------------------------------------------------- what a program has in hand before the call
class _Weights:
    """A weight table of the package's form: N(0, 0.02) matrices cut from one pool of random values, unit gains."""

    def __init__(self, m):
        self.shapes = weight_shapes(m)
        g = torch.Generator(device=DEVICE).manual_seed(1)
        n = max(int(np.prod(s)) for s in self.shapes.values())
        self.pool = (0.02 * torch.randn(n + (1 << 20), device=DEVICE, generator=g)).to(torch.bfloat16).float().cpu().numpy()
        self.at = {name: (7919 * 64 * i) % (1 << 20) for i, name in enumerate(self.shapes)}

    def names(self):
        return list(self.shapes)

    def __getitem__(self, name):
        shape = self.shapes[name]
        if is_gain(name):
            return np.ones(shape, dtype=np.float32)
        return self.pool[self.at[name]:self.at[name] + int(np.prod(shape))].reshape(shape)


@functools.lru_cache(maxsize=None)
def _engine(model):
    """The server's engine of one model: made once, kept for as long as the program runs."""
    m = get_config(model)
    eng = Engine(m, mode="cosched", device=DEVICE)
    eng.load_weights(_Weights(m))
    return eng


def _frame(m, g, inputs):
    f = {"image": torch.rand(m.n_cam, 3, m.img, m.img, device=DEVICE, generator=g),
         "text": torch.randint(0, m.vocab, (m.n_text,), device=DEVICE, generator=g, dtype=torch.int32),
         "state": torch.randn(m.state_dim, device=DEVICE, generator=g) if m.state_dim > 0 else None,
         "noise": torch.randn(m.horizon, m.act_dim, device=DEVICE, generator=g)}
    if inputs == "device":
        return f
    f = {k: None if v is None else v.cpu() for k, v in f.items()}
    if inputs == "pinned":
        f = {k: None if v is None else v.pin_memory() for k, v in f.items()}
    return {k: None if v is None else v.numpy() for k, v in f.items()}


def prepare(case, seed):
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    if case["kind"] == "engine":
        m = get_config(case["model"])
        frames = [[_frame(m, g, case["inputs"]) for _ in range(case["frames"])] for _ in range(case["streams"])]
        return {"case": case, "engine": _engine(case["model"]), "frames": frames}

    def rand(rows, cols, scale):
        return (scale * torch.randn(rows, cols, device=DEVICE, generator=g)).to(torch.bfloat16)
    if case["kind"] == "linear":
        return {"case": case, "a": rand(case["m"], case["k"], 1.0), "w": rand(case["n"], case["k"], 0.02)}
    tq, tkv, hq, hkv, hd = (case[k] for k in ("tq", "tkv", "hq", "hkv", "hd"))
    s = {"case": case, "q": rand(tq, hq * hd, 1.5), "k": rand(tkv, hkv * hd, 1.5), "v": rand(tkv, hkv * hd, 1.0)}
    if case["static"]:
        s["out"] = torch.empty_like(s["q"])
    else:
        s["scratch"] = torch.empty(api.op_attention_scratch_bytes(tkv, hkv, hd), dtype=torch.uint8, device=DEVICE)
    return s


# ---------------------------------------------------------------- one pass
def _serve_resident(eng, frames):
    """Frames that are on the GPU already: submitted as fast as the rings accept, chunks taken as they finish."""
    n = len(frames[0])
    out = np.empty((len(frames), n) + eng.chunk_shape, dtype=np.float32)
    sent, done = [0] * len(frames), [0] * len(frames)
    left = len(frames) * n
    while left:
        for r, fs in enumerate(frames):
            while sent[r] < n:
                f = fs[sent[r]]
                ptrs = [None if f[k] is None else f[k].data_ptr() for k in ("image", "text", "state", "noise")]
                if eng.submit_ptrs(r, *ptrs, device=True) == api.VLA_ERR_BUSY:
                    break
                sent[r] += 1
            while done[r] < sent[r] and eng.poll(r, out[r, done[r]]) is not None:
                done[r] += 1
                left -= 1
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "engine":
        if case["inputs"] == "device":
            return _serve_resident(state["engine"], state["frames"])
        return np.array(state["engine"].run(state["frames"]))
    if case["kind"] == "linear":
        return api.op_linear(state["a"], state["w"], act=case["act"], out_bf16=case["bf16"])
    if case["static"]:
        return api.op_attention_static(state["q"], state["k"], state["v"], state["out"], case["hq"], case["hkv"], case["hd"],
                                       causal=case["causal"])
    return api.op_attention(state["q"], state["k"], state["v"], case["hq"], case["hkv"], case["hd"], causal=case["causal"],
                            scratch=state["scratch"])


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["kind"] == "engine":
        m = get_config(case["model"])
        w, chunks = chunk_work(m), case["streams"] * case["frames"]
        frame = 4 * (m.n_cam * 3 * m.img * m.img + m.n_text + m.state_dim + 2 * m.horizon * m.act_dim)   # inputs and the chunk
        return {"bytes": 2 * (w["vlm_params"] + w["head_params"]) + chunks * frame, "flops": chunks * w["flops"]}
    if case["kind"] == "linear":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2 * (m * k + n * k) + (2 if case["bf16"] else 4) * m * n, "flops": 2 * m * n * k}
    tq, tkv, hq, hkv, hd = (case[k] for k in ("tq", "tkv", "hq", "hkv", "hd"))
    pairs = tq * (tq + 1) // 2 if case["causal"] else tq * tkv
    return {"bytes": 2 * hd * (2 * tq * hq + 2 * tkv * hkv), "flops": 4 * pairs * hq * hd}


def tolerance(case):
    if case["kind"] == "engine":
        return {"rel": 1e-2, "max": 1e-1}      # bf16 operands through tens of layers, fp32 sums and chunks
    if case["kind"] == "linear":
        if case["bf16"]:
            return {"rel": 5e-3, "max": 3e-2}  # the result's own rounding to bf16
        # fp32 sums of exact products; an activation may use the hardware's approximations (about 2^-11)
        return {"rel": 1e-5 if case["act"] == 0 else 1e-3}
    return {"rel": 1e-2, "max": 1e-1}          # bf16 probabilities and results
