"""Two contexts in one process do not undo one another's set-up."""
import numpy as np
import pytest

from vla_synth.configs import CFG1, CFG4, mini
from vla_synth.gen import make_weights, frame_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["serial", "two_stream"])
def test_context_of_a_small_model_leaves_the_one_of_a_wide_model_usable(mode):
    """Head-dimension-256 attention tiles take more shared memory per block than any tile of the small model."""
    from paper_2609_22335_b200 import Engine
    wide = mini(CFG4, n_cam=1, img=112, vis_layers=1, llm_layers=2, act_layers=2, mlp=1024, n_steps=2, vocab=2048, n_streams=1, n_frames=1)
    frames = [[frame_inputs(wide, 0, 0, seed=4)]]
    got, engines = [], []
    try:
        for with_other in (False, True):
            engines.append(Engine(wide, mode=mode, n_streams=1))
            engines[-1].load_weights(make_weights(wide, seed=0))
            if with_other:
                engines.append(Engine(CFG1, mode=mode, n_streams=1))
            got.append(engines[with_other].run(frames)[0][0])
    finally:
        for e in engines:
            e.close()
    assert np.array_equal(got[0], got[1])
