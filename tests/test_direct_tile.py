"""The direct sum's launch rule (csrc/sg_direct_tile.h, host arithmetic, compiled
here) on the sizes of test_gpu_direct_shapes.py: every kernel instance is reached, each with
rows of one and of several target chunks, with a full and a partly filled last one, so
that a change of the rule's costs cannot drop an instance from the tests; and its
shapes stay within what the kernel takes, over its whole range of grids."""
import ctypes
import os
import subprocess

import pytest

import test_gpu_direct_shapes as shapes

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2506_10812_gb300", "csrc")
SOURCE = """#include "sg_direct_tile.h"
extern "C" void tile(int nr, int nphi, int f64, int *o)
{
    const sg::DirectTile t = sg::direct_tile(nr, nphi, f64 != 0);
    o[0] = t.KT, o[1] = t.W, o[2] = t.S, o[3] = t.nchunk;
}
"""


@pytest.fixture(scope="module")
def tile(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile")
    (d / "tile.cpp").write_text(SOURCE)
    lib = str(d / "tile.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(d / "tile.cpp"), "-o", lib])
    fn = ctypes.CDLL(lib).tile

    def call(nr, nphi, f64):
        o = (ctypes.c_int * 4)()
        fn(nr, nphi, int(f64), o)
        return tuple(o)
    return call


def kind(tile, nr, nphi, f64):
    KT, W, _, nchunk = tile(nr, nphi, f64)
    return KT, nchunk > 1, nphi % (32 * W * KT) != 0


def test_sizes_reach_every_instance(tile):
    both = [(several, part) for several in (False, True) for part in (False, True)]
    got = {kind(tile, nr, nphi, False) for nr, nphi in shapes.F32}
    assert got >= {(KT, *b) for KT in (2, 4) for b in both}
    got = {kind(tile, nr, nphi, True) for nr, nphi in shapes.F64}
    assert got >= {(2, False, True), (2, True, False), (2, True, True), (1, True, False), (1, True, True)}


def test_shapes_are_launchable(tile):
    for f64 in (False, True):
        for nr in (1, 2, 3, 7, 8, 100, 1024, 1 << 21):
            for nphi in (8, 9, 31, 33, 255, 257, 1000, 4096, 1 << 23):
                if nr * nphi > 1 << 24:
                    continue
                KT, W, S, nchunk = tile(nr, nphi, f64)
                assert KT in ((1, 2) if f64 else (1, 2, 4)) and 1 <= W <= 8 and S in (1, 2, 4, 8) and S <= nr
                assert (nchunk - 1) * 32 * W * KT < nphi <= nchunk * 32 * W * KT
                assert nr * nchunk * S < 1 << 31
