"""Automatic split of the FP64 stage kernel (csrc/rlb_schedule.h) on the host: the choice is that of handing every work
item to the slot that comes free first, for handles of equal and of uneven tubes around all multiples of the slots, and
it takes a small part of the time."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("sched") / "libsched.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-o", out,
                    os.path.join(HERE, "cpu_src", "schedule_check.cpp")], check=True)
    fn = ctypes.CDLL(out).schedule_eval
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_longlong, ctypes.c_void_p, ctypes.c_void_p]

    def run(rows, tiles, slots=456):
        r, t = np.asarray(rows, dtype=np.float64), np.asarray(tiles, dtype=np.int64)
        o, us = np.zeros(2, dtype=np.int32), np.zeros(2)
        fn(r.ctypes.data, t.ctypes.data, r.size, slots, o.ctypes.data, us.ctypes.data)
        return int(o[0]), int(o[1]), us

    return run


@pytest.mark.parametrize("rows", [12, 96, 384, 3072])
def test_equal_tiles(choose, rows):
    for n in [1, 2, 57, 58, 100, 228, 229] + [456 * k + d for k in range(1, 9) for d in (-1, 0, 1, 4, 150)]:
        got, ref, _ = choose([rows], [n])
        assert got == ref, (n, rows, got, ref)


def test_uneven_tubes(choose):
    rng = np.random.default_rng(11)
    for _ in range(150):
        k = int(rng.integers(2, 40))
        rows = np.sort(rng.integers(12, 700, k))[::-1]
        tiles = np.maximum(1, np.exp(rng.uniform(0, np.log(3600 / k), k)).astype(np.int64))
        slots = int(rng.choice([1, 7, 152, 456]))
        got, ref, _ = choose(rows, tiles, slots)
        assert got == ref, (rows, tiles, slots)


def test_time_below_eight_waves(choose):
    """A handle just below 8 waves of equal tiles: the queue of single slots takes some ms in every handle's creation."""
    got, ref, us = choose([384], [3647])
    assert got == ref and us[0] <= 0.1 * us[1], us
