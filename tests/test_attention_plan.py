"""The launch plan of the stand-alone attention (csrc/attention_plan.h, compiled for the host): whatever the shape, the cluster's exchange
fits its shared memory, the score buffers and the output fit tensor memory, and a split into fewer parts than the precision asks for
takes its probabilities in two terms."""
import ctypes as C
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
B200 = [0, 148, 74, 45, 33, 26, 22, 15, 15], [0, 296, 148, 93, 71, 56, 45, 37, 33]            # clusters of one CTA per SM, and of two


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    out = tmp_path_factory.mktemp("plan") / "libattention_plan.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-x", "c++", os.path.join(HERE, "attention_plan_host_shim.cc"),
                    "-o", str(out)], check=True)
    lib = C.CDLL(str(out))

    def call(tiles, tkv, hs, causal=False, sms=148, room=B200):
        o = (C.c_int * 7)()
        lib.attention_plan_host(tiles, tkv, hs, int(causal), sms, (C.c_int * 9)(*room[0]), (C.c_int * 9)(*room[1]), o)
        return dict(zip(("split", "stages", "smem", "tmem_cols", "s_bufs", "terms", "min_parts"), o))
    return call


def _old_parts(tiles, tkv, hs, sms, smem):
    """Powers of two up to the chip's CTAs: the parts that the operator's precision is stated for."""
    s, per_sm = 1, 2 if hs <= 128 else 1
    while s < 8 and tiles * s * 2 <= per_sm * sms and -(-tkv // 64) >= 2 * s and -(-(hs // 16) // (2 * s)) * 2 * s * 8192 <= smem:
        s *= 2
    return s


def test_every_plan_is_one_the_kernel_can_run(plan):
    rnd = random.Random(4)
    shapes = [(t, n, hs) for t in (1, 4, 96, 148, 149, 5000) for n in (1, 64, 65, 867, 100000) for hs in (16, 64, 80, 128, 144, 192, 256)]
    shapes += [(int(2 ** rnd.uniform(0, 11)), int(2 ** rnd.uniform(0, 12)), 16 * rnd.randint(1, 16)) for _ in range(3000)]
    two = 0
    for tiles, tkv, hs in shapes:
        for sms, room in ((148, B200), (132, ([0, 132, 66, 40, 32, 24, 18, 16, 16], [0, 264, 132, 84, 64, 48, 40, 32, 32])),
                          (7, ([0, 7, 3, 2, 1, 1, 1, 1, 0], [0, 14, 7, 4, 3, 2, 2, 2, 1])), (148, ([0] * 9, [0] * 9))):
            p = plan(tiles, tkv, hs, tiles % 2 == 1, sms, room)
            assert 1 <= p["split"] <= min(8, -(-tkv // 64)) and 2 <= p["stages"] <= 4
            boxes = -(-hs // 64)
            assert p["smem"] == boxes * (16384 + p["stages"] * 16384) <= (104 if hs <= 128 else 208) * 1024
            if p["split"] > 1:
                assert -(-(hs // 16) // p["split"]) * p["split"] * 8192 <= p["smem"]
            assert 2 <= p["s_bufs"] <= 3 and p["s_bufs"] * 64 + hs <= p["tmem_cols"] == (256 if hs <= 128 else 512)
            assert p["min_parts"] == _old_parts(tiles, tkv, hs, sms, p["smem"])
            assert p["terms"] == (1 if p["split"] >= p["min_parts"] else 2)
            assert p["split"] <= 2 or sms == 7 or room[0][8] > 0             # clusters of unknown number are not used
            two += p["terms"] == 2
    assert two > 500


def test_splits_that_fill_the_chip(plan):
    """Clusters of three and more get two CTAs an SM; causal tiles are short but for the last ones; and a split that is not worth its meeting."""
    splits = [plan(*a)["split"] for a in ((60, 1908, 64), (60, 1813, 64, True), (384, 687, 80, True), (384, 987, 64, True), (440, 1345, 64, True),
                                          (960, 1264, 64), (96, 1024, 64), (72, 687, 128), (36, 956, 128), (4, 867, 256))]
    assert splits == [4, 4, 1, 1, 1, 1, 2, 2, 3, 8]
