"""The tile plan of the stand-alone linear layer (csrc/linear_plan.h, compiled for the host): whatever the shape, the tiles cover
the result, the stages fit half an SM, and a split's partial sums fit the stages and its clusters the chip."""
import ctypes as C
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    out = tmp_path_factory.mktemp("plan") / "libplan_host.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-x", "c++", os.path.join(HERE, "linear_plan_host_shim.cc"),
                    "-o", str(out)], check=True)
    lib = C.CDLL(str(out))

    def call(m, n, k, f32=False, sms=148):
        o = (C.c_int * 6)()
        lib.linear_plan_host(m, n, k, int(f32), sms, o)
        return dict(zip(("bm", "bn", "ks", "tiles_m", "tiles", "stages"), o))

    def pair(m, n, k, f32=False, sms=148):
        o = (C.c_int * 5)()
        lib.linear_pair_plan_host(m, n, k, int(f32), sms, o)
        return list(o)
    call.pair = pair
    return call


def test_every_plan_is_one_the_kernel_can_run(plan):
    rnd = random.Random(3)
    shapes = [(m, n, k) for m in (1, 16, 17, 64, 127, 128, 129, 100000) for n in (1, 7, 16, 255, 256, 257, 70000) for k in (8, 64, 72, 4096, 20000)]
    shapes += [(int(2 ** rnd.uniform(0, 14)), int(2 ** rnd.uniform(0, 15)), 8 * int(2 ** rnd.uniform(0, 11))) for _ in range(3000)]
    for m, n, k in shapes:
        for sms, f32 in ((148, False), (148, True), (132, False), (7, False), (7, True)):
            p = plan(m, n, k, f32, sms)
            bm, bn, ks, stages = p["bm"], p["bn"], p["ks"], p["stages"]
            assert bm % 16 == 0 and 16 <= bm <= 128 and p["tiles_m"] * bm >= m > (p["tiles_m"] - 1) * bm
            assert bn % 16 == 0 and 16 <= bn <= 256 and p["tiles"] == p["tiles_m"] * -(-n // bn)
            stage = (bm + bn) * 128
            assert 2 <= stages <= 12 and stages * stage + max(0, 16384 - stage) <= 110 * 1024
            assert ks in (1, 2, 4, 8)
            if ks > 1:
                assert bn in (32, 64, 128, 256) and bn % (32 * ks) == 0 and -(-k // 64) >= 2 * ks and p["tiles"] * ks <= 2 * sms
                assert 128 * (bn // ks) * (ks - 1) * 4 <= stages * stage


def test_widths_that_fill_the_chip(plan):
    """Shapes where a power of two leaves a second CTA to a few SMs, or a second round to a few CTAs."""
    pairs = [(p["bn"], p["ks"]) for p in (plan(3455, 1392, 8448), plan(1441, 4360, 6256), plan(653, 7782, 2248), plan(452, 6648, 6024),
                                          plan(8192, 3072, 768), plan(50, 2048, 720))]
    assert pairs == [(144, 1), (192, 1), (160, 1), (192, 1), (240, 1), (16, 1)]


def test_fp32_results_keep_their_split(plan):
    """Sums are split where they are long and the chip has room, whatever a width without a split would gain."""
    for shape, ks in (((288, 11008, 4096), 2), ((452, 6648, 6024), 2), ((938, 1352, 6144), 4), ((91, 9152, 1344), 4), ((8192, 3072, 768), 1)):
        assert plan(*shape, f32=True)["ks"] == ks


def test_a_call_goes_where_it_is_faster(plan):
    """Shapes that a plan which took clusters of four for one CTA per SM, their late ones for a whole wave, and a pair's k-block for 350 cycles
    sent to two-SM tiles or a wider split at up to 1.5 times the time; and ones that gain from two SMs."""
    def choice(*shape):
        pair = plan.pair(*shape)[1]
        p = plan(*shape)
        return (pair or p["bn"], p["ks"], pair > 0)
    for shape, best in (((948, 786, 6656, False), (128, 4, False)), ((719, 1056, 5472, False), (128, 4, False)), ((286, 2435, 4640, False), (128, 4, False)),
                        ((4390, 149, 6736, True), (128, 4, False)), ((1215, 810, 10616, True), (128, 4, False)), ((931, 1072, 11040, True), (128, 4, False)),
                        ((4917, 1076, 7296, True), (160, 1, False)), ((360, 10776, 5888, False), (112, 1, False)),
                        ((489, 4487, 2928, True), (128, 4, True)), ((983, 1626, 3912, False), (128, 2, True)), ((4096, 4096, 4096, False), (240, 1, True))):
        assert choice(*shape) == best, shape


def test_every_plan_of_two_sm_tiles_is_one_the_kernel_can_run(plan):
    rnd = random.Random(5)
    shapes = [(m, n, k) for m in (1, 128, 129, 256, 257, 100000) for n in (7, 112, 113, 255, 257, 70000) for k in (8, 72, 4096, 20000)]
    shapes += [(int(2 ** rnd.uniform(6, 14)), int(2 ** rnd.uniform(4, 15)), 8 * int(2 ** rnd.uniform(0, 11))) for _ in range(3000)]
    used = 0
    for m, n, k in shapes:
        for sms, f32 in ((148, False), (148, True), (132, False), (7, True), (1, False)):
            bm, bn, tiles_m, tiles, stages = plan.pair(m, n, k, f32, sms)
            if bn == 0:
                continue
            used += 1
            parts = plan(m, n, k, f32, sms)["ks"]              # accumulators in the 512 columns of tensor memory
            assert m > 128 and sms > 1 and parts * bn <= 512 and -(-k // 64) >= parts
            assert bm % 16 == 0 and 16 <= bm <= 128 and tiles_m * 2 * bm >= m > (tiles_m - 1) * 2 * bm
            assert bn % 16 == 0 and 128 <= bn <= 256 and tiles == tiles_m * -(-n // bn)
            stage = (bm + bn // 2) * 128                       # whole 1024-byte swizzle groups, and the MMA reads 128 rows of tokens
            assert bm * 128 % 1024 == 0 and stage % 1024 == 0
            assert 2 <= stages <= 12 and (stages - 1) * stage + max(stage, 16384) <= 224 * 1024
    assert used > 1000


def test_the_gpu_tests_reach_what_they_are_for(plan):
    """The shapes of the tests of two-SM tiles go to them, with K in one, two and four parts for both result types, stores of eight, two and
    one feature, and widths that end inside 32 columns; those of the exchange between CTAs go to that."""
    from test_gpu_linear_pair import SHAPES
    reached = set()
    for m, n, k in SHAPES:
        for f32 in (False, True):
            width = plan.pair(m, n, k, f32)[1]
            assert width > 0 or (m, n, k, f32) in ((3261, 392, 1424, False), (326, 5053, 4064, True))
            if width:
                reached.add((f32, plan(m, n, k, f32)["ks"], 8 if n % 8 == 0 else 2 if n % 2 == 0 else 1))
                reached.add((f32, width % 32))
    assert reached >= {(False, p, v) for p in (1, 2, 4) for v in (8, 2, 1)} | {(True, 1, v) for v in (8, 2, 1)} | {(True, 2, 8), (True, 2, 1), (True, 4, 8), (True, 4, 1)}
    assert reached >= {(f32, w) for f32 in (False, True) for w in (0, 16)}
    for shape, ks in (((288, 11008, 4096), 2), ((572, 6298, 1616), 2), ((257, 2370, 2056), 4)):
        assert plan(*shape, f32=True)["ks"] == ks and plan(*shape, f32=True)["bn"] == (256 if ks == 2 else 128) and plan.pair(*shape, True)[1] == 0
