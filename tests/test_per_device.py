"""What the operators look up once per GPU (csrc/per_device.h, compiled for the host): first calls from several threads each get a whole
record, one of them is kept, and a look-up that failed is tried again."""
import ctypes as C
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_first_calls_from_several_threads(tmp_path):
    out = tmp_path / "libper_device.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-shared", "-fPIC", "-x", "c++", os.path.join(HERE, "per_device_host_shim.cc"),
                    "-o", str(out)], check=True)
    lib = C.CDLL(str(out))
    lib.per_device_first_calls.restype = C.c_longlong

    def first_calls(dev, n, fail=0):
        got = (C.c_longlong * n)()
        return lib.per_device_first_calls(dev, n, fail, got), list(got)
    for dev in range(32):
        kept, got = first_calls(dev, 8)
        assert 1 <= kept <= 8 and kept in got and all(1 <= x <= 8 for x in got)
        later, got = first_calls(dev, 8)
        assert later == kept and got == [kept] * 8
    kept, got = first_calls(32, 4, fail=4)
    assert kept == 0 and got == [0] * 4                      # nothing is kept of a look-up that failed ...
    kept, got = first_calls(32, 4, fail=1)
    assert got.count(0) <= 1 and kept in got and kept > 0    # ... and the next call tries again
    for dev in (-1, 64):
        assert first_calls(dev, 2) == (0, [0, 0])
