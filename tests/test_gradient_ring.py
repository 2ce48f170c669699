"""The data gradients' shared-memory slots: all interleavings of a block's copying and issuing threads (no GPU)."""
import os
import subprocess

import pytest

from paper_2012_09849_b200 import build as hb


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    hb.build()
    exe = str(tmp_path_factory.mktemp("ring") / "walk")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-I", os.path.join(hb.PKG, "csrc"), "-I", os.path.join(hb.ROOT, "include"),
                           "-I", cuda, os.path.join(os.path.dirname(__file__), "x3_ring_walk.cpp"), "-o", exe, "-L", hb.PKG, "-l:libhts.so",
                           "-Wl,-rpath," + hb.PKG])
    return lambda *args: subprocess.run([exe, *map(str, args)], capture_output=True, text=True)


# M tiles, N tiles, first tile and blocks: one tile; tiles of one N tile; a tile of each N tile; several of each; N tiles left out
TILES = [(1, 1, 0, 1), (2, 1, 0, 1), (1, 2, 0, 1), (2, 2, 0, 2), (3, 2, 1, 2), (2, 2, 0, 1), (1, 3, 0, 2)]


# (64-row chunks, taps, width of the grid): the dense layer, the third and the second convolution of 84 x 84 and 72 x 96 frames, one
# whose taps just share an entry, and grids too wide for that
@pytest.mark.parametrize("tiles", TILES)
@pytest.mark.parametrize("layer", [(8, 1, 1), (1, 9, 9), (1, 9, 10), (1, 9, 51), (1, 9, 60), (1, 4, 10), (1, 4, 12), (1, 4, 103), (1, 4, 130)])
def test_no_slot_is_overwritten_and_everyone_ends(walk, layer, tiles):
    done = walk(*layer, *tiles)
    assert done.returncode == 0, done.stdout
