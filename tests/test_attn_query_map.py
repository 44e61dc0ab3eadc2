"""The query fetch of the tensor-core attention, address by address on the CPU: every entry of every tile gets its own row, and no tile
reads behind the room its buffer has.  The map and its coordinates are the kernel's own (csrc/q_tile.cuh), compiled for the host."""
import ctypes
import itertools
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_19201_b200", "csrc")
SHIM = """
#include "q_tile.cuh"
extern "C" void tile_map(int rows, int H, int G, int hd, QTileMap *m) { *m = q_tile_map(rows, H, G, hd); }
extern "C" void tile_start(int G, int row, int *c) { q_tile_start(G, row, c[0], c[1]); }
extern "C" int tile_room(int rows) { return q_tile_room(rows); }
"""


class Map(ctypes.Structure):
    _fields_ = [("dims", ctypes.c_ulonglong * 5), ("strides", ctypes.c_ulonglong * 4), ("box", ctypes.c_uint * 5)]


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    d = tmp_path_factory.mktemp("q_tile")
    src, lib = os.path.join(d, "shim.cpp"), os.path.join(d, "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


def tile_rows(shim, m, G, first_head, row):
    """The 128 rows of a tile in the order the copy leaves them, each the byte offset of its first column, -1 where it is outside the map."""
    c = (ctypes.c_int * 2)()
    shim.tile_start(G, row, c)
    at = [s + np.arange(b) for s, b in zip((first_head, c[0], 0, c[1]), m.box[1:])]
    grid = np.meshgrid(*reversed(at), indexing="ij")[::-1]
    inside = np.logical_and.reduce([(0 <= g) & (g < n) for g, n in zip(grid, m.dims[1:])])
    return np.where(inside, sum(g * s for g, s in zip(grid, m.strides)), -1).ravel()


# rows per sequence and sequences of a call: prompts (one sequence, up to the whole buffer) and decode rounds (at most 256 rows)
CALLS = [(n, 1) for n in (1, 2, 3, 7, 8, 61, 64, 65, 100, 249, 250, 255, 256, 257, 271, 272)] + [(1, 8), (7, 8), (31, 8), (32, 8), (61, 4), (64, 4), (85, 3), (127, 2), (128, 2)]


@pytest.mark.parametrize("G", [1, 2, 4, 8, 16, 32, 64])
@pytest.mark.parametrize("hd,hkv", [(64, 2), (128, 1), (256, 3)])
def test_tiles(shim, G, hd, hkv):
    H = G * hkv
    for n, batch in CALLS:
        XR = max(256, (n * batch + 15) // 16 * 16)
        m = Map()
        shim.tile_map(XR, H, G, hd, ctypes.byref(m))
        part = hd * 2
        room = shim.tile_room(XR) * H * 2 * part
        # what a tensor map takes: extents, 16-byte strides, a box of 128 rows of 128 bytes
        assert all(d >= 1 for d in m.dims) and all(s % 16 == 0 for s in m.strides) and all(1 <= b <= 256 for b in m.box)
        assert m.box[0] == 64 and m.box[1] * m.box[2] * m.box[3] * m.box[4] == 128
        n_rt = (n * G + 63) // 64
        for b, kvh, rt in itertools.product(range(batch), range(hkv), sorted({0, 1, *range(n_rt - 9, n_rt)} & set(range(n_rt)))):
            got = tile_rows(shim, m, G, kvh * G, b * n + rt * 64 // G)
            end = int(got.max()) + part
            assert end <= room, f"{n} rows x {batch}: a tile reads {end - room} bytes behind its buffer"
            assert batch > 1 or end <= XR * H * 2 * part                     # a prompt's: nothing behind its rows
            e = np.arange(min(64, n * G - rt * 64))
            want = ((b * n + (rt * 64 + e) // G) * H + kvh * G + (rt * 64 + e) % G) * 2 * part
            at = e // 8 * 16 + e % 8
            assert (got[at] == want).all() and (got[at + 8] == want + part).all()
