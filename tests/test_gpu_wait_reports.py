"""A device-side wait that runs out inside a tile reaches the host as VLA_ERR_TIMEOUT.  The failure is made on the host (a
dependency count raised while nothing is in flight); the wait is bounded, the kernel returns and the context can be closed."""
import time

import pytest

from vla_synth.configs import CFG1
from vla_synth.gen import make_weights, frame_inputs

pytestmark = pytest.mark.gpu


def _head_gemm(node):
    return node["phase"] == 1 and node["n_pred"] > 0 and node["name"].endswith("L1.w2")


def _emit(node):
    return node["op"] == 8


@pytest.mark.parametrize("which", [_head_gemm, _emit])
def test_tile_that_waits_for_its_release_in_vain_is_reported_while_other_streams_run(which):
    """The stalled node's tile was queued before its release and waits on its worker.  Its own wait
    tells the host, whether or not the idle watchdog has something to say beside the frames of another stream; and the frame it
    belongs to is never handed out, not even when that tile is the one that publishes it."""
    from paper_2609_22335_b200 import Engine, api
    eng = Engine(CFG1, mode="cosched", n_streams=2, wait_limit_ns=200_000_000)            # 0.2 s
    try:
        eng.load_weights(make_weights(CFG1, seed=0))
        eng.run([[frame_inputs(CFG1, r, n, seed=0) for n in range(4)] for r in range(2)])     # everything is loaded and warm
        eng.wait_idle()
        victim = next(i for i, n in enumerate(eng.program_info()) if which(n))
        eng.bump_dependency(0, 0, victim, 1)
        frame = frame_inputs(CFG1, 0, 0, seed=0)
        assert eng.submit(0, frame) == api.VLA_OK
        code, t0 = None, time.time()
        while code is None and time.time() - t0 < 5.0:
            try:
                eng.submit(1, frame)                         # (VLA_ERR_BUSY: the ring is full)
                eng.poll(1)
                assert eng.poll(0) is None
            except api.VlaError as e:
                code = e.code
        assert code == api.VLA_ERR_TIMEOUT and "wait ran out" in eng.last_error()
    finally:
        eng.close()
