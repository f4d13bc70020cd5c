"""The end of a block of the generated lane kernel, where warps meet once a
turn and their last zones are packed into fewer warps (block_done), run on
the host with one fibre per thread (tests/host/block_tail.cpp).  Warps run
ahead of one another as far as the barriers let them, in many orders, with
zones that end at once (what an expired budget or an attempt limit does) and
zones that run on."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def run_block(tmp_path_factory):
    gxx = shutil.which(os.environ.get("CXX", "g++"))
    if gxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("host") / "libblocktail.so")
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic",
                           "-I", os.path.join(ROOT, "include"),
                           os.path.join(HERE, "host", "block_tail.cpp"), "-o", out])
    fn = C.CDLL(out).run_block
    fn.argtypes = [C.c_int, C.c_longlong, C.c_void_p, C.c_void_p]

    def run(warps, zone_turns, order):
        t = np.ascontiguousarray(zone_turns, np.int32)
        o = np.ascontiguousarray(order, np.int32)
        return fn(32 * warps, t.size, t.ctypes.data, o.ctypes.data)

    return run


@pytest.mark.parametrize("warps", [1, 2, 3, 5, 8])
def test_warps_agree_on_the_last_zones_in_any_order(run_block, warps):
    rng = np.random.default_rng(warps)
    for trial in range(40):
        zones = int(rng.integers(1, 32 * warps * 2 + 1))
        # whole warps of zones that end together, at different turns
        turns = rng.integers(1, 6, zones)
        turns[: 32 * warps] = np.repeat(rng.integers(1, 6, warps), 32)[: min(zones, 32 * warps)]
        if trial % 2:
            turns = np.where(rng.random(zones) < 0.2, rng.integers(1, 30, zones), turns)
        order = rng.permutation(warps)
        assert run_block(warps, turns, order) == 0, (trial, zones, order)
