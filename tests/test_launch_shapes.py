"""Launch shapes against the buffers they fill, over the grids a mesh
descriptor may have: the mixed 3D sensitivity writes one partial sum per
block, and its grid must fit the partial sums' buffer and the grid limits.

The shapes are enumerated from the accepted descriptors (a coarsest grid of at
most 2048 nodes, up to ten levels) up to two billion elements, more than any
workspace on this GPU allows (about 500 bytes an element)."""

import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_00385_gb300", "csrc")

SRC = """
#include "launch_shapes.h"
extern "C" int chunk(int x, int y, int z) { return topo::sensitivity_chunk(x, y, z); }
extern "C" long long blocks(int x, int y, int z, int c) { return topo::sensitivity_blocks(x, y, z, c); }
extern "C" long long partials() { return topo::PARTIALS; }
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("shapes")
    (d / "s.cpp").write_text(SRC)
    so = str(d / "s.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "s.cpp"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)
    lib.blocks.restype = lib.partials.restype = ctypes.c_longlong
    return lib


def _grids():
    side = [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 16, 20, 31, 63, 100, 255, 340, 511]
    for levels in range(2, 11):
        f = 2 ** (levels - 1)
        for a in side:
            for b in side:
                for c in side:
                    if (a + 1) * (b + 1) * (c + 1) <= 2048 and f ** 3 * a * b * c <= 2e9:
                        yield f * a, f * b, f * c


def test_sensitivity_partial_sums_fit(shapes):
    cap = shapes.partials()
    assert cap == 608 * 16 * 16
    many = 0
    for x, y, z in _grids():
        zc = shapes.chunk(x, y, z)
        n = shapes.blocks(x, y, z, zc)
        assert 1 <= zc and 1 <= n <= cap, (x, y, z, zc, n)
        assert (y + 3) // 4 <= 65535 and (z + zc - 1) // zc <= 65535
        many += shapes.blocks(x, y, z, 16) > cap
    assert many > 0                                   # (704 x 704 x 704 is one)
    assert shapes.blocks(704, 704, 704, 16) == 170368
    assert shapes.chunk(192, 96, 96) == 8 and shapes.chunk(320, 160, 160) == 16
