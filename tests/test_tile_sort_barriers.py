"""The sort of a tile's keys gives the same whichever of the CTA's warps is ahead (on the host: tile_sort_host.cpp)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
TILE, WARPS = 2_048, 8


@pytest.fixture(scope="module")
def host_sort(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("tile_sort") / "tile_sort_host.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-fno-strict-aliasing", "-Wno-unknown-pragmas", "-shared", "-fPIC",
                           os.path.join(HERE, "tile_sort_host.cpp"), "-o", out])
    return ctypes.CDLL(out).tile_sort_host


@pytest.mark.parametrize("order", [range(WARPS), range(WARPS)[::-1], [4, 5, 6, 7, 0, 1, 2, 3], [1, 0, 3, 2, 5, 4, 7, 6]], ids=str)
@pytest.mark.parametrize("tokens", [1, 8, 9, 255, 256, 257, 300, 512, 513, 1_024, 1_025, 2_047, 2_048])
def test_every_order_of_the_warps(host_sort, tokens, order):
    K, topic_bits = 20_000, 15
    rng = np.random.default_rng(tokens)
    z = rng.integers(0, K, tokens).astype(np.uint32)
    off = np.concatenate([[0], np.sort(rng.integers(0, tokens + 1, 40)), [tokens]]).astype(np.int32)
    warps = np.array(order, np.int32)
    registers, shared, in_range = np.zeros(TILE, np.uint32), np.zeros(TILE, np.uint32), ctypes.c_int()
    p = [ctypes.c_void_p(a.ctypes.data) for a in (z, off, warps, registers, shared)]
    assert host_sort(p[0], p[1], off.size - 1, topic_bits, K, p[2], p[3], p[4], ctypes.byref(in_range)) == 0
    want = np.full(TILE, 0xFFFFFFFF, np.uint32)
    want[:tokens] = np.sort(np.repeat(np.arange(off.size - 1, dtype=np.uint32), np.diff(off)) << topic_bits | z)
    assert np.array_equal(registers, want) and np.array_equal(shared, want)
    assert in_range.value == 1
