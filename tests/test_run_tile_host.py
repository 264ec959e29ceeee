"""Which body runs a tile (csrc/run_tile.cuh, compiled for the host with stand-ins for the bodies): every operation its own,
and an operation that the kernel does not have none at all -- it is recorded as an error."""
import ctypes as C
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
GEMM, RMSNORM, ATTN, PATCHIFY, EMBED, ADDROWS, TIMEEMB, EMIT, EMIT_PART = 0, 1, 2, 3, 4, 6, 7, 8, 9
BAD_OP = 5


@pytest.fixture(scope="module")
def run_tile(tmp_path_factory):
    out = tmp_path_factory.mktemp("run_tile") / "librun_tile.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-x", "c++", os.path.join(HERE, "run_tile_host_shim.cc"),
                    "-o", str(out)], check=True)
    lib = C.CDLL(str(out))

    def call(load_time, op):
        err = C.c_uint(0)
        return lib.run_tile_host(int(load_time), op, C.byref(err)), err.value
    return call


@pytest.mark.parametrize("load_time", [False, True])
def test_every_operation_runs_its_own_body(run_tile, load_time):
    for op in (GEMM, RMSNORM, ATTN, PATCHIFY, EMBED, ADDROWS, EMIT, EMIT_PART):
        assert run_tile(load_time, op) == (op, 0)


def test_load_time_operation_is_an_error_in_the_persistent_kernel(run_tile):
    assert run_tile(True, TIMEEMB) == (TIMEEMB, 0)
    assert run_tile(False, TIMEEMB) == (-1, BAD_OP)


@pytest.mark.parametrize("load_time", [False, True])
def test_unknown_operation_is_an_error(run_tile, load_time):
    for op in (5, 10, -1):
        assert run_tile(load_time, op) == (-1, BAD_OP)
