"""Work items of the batched form: whatever launch shape is set or tuned, a small
batch's items leave every resident block two (creation, the tuner's candidates and a
given shape go through one rule), and a large batch's are of the size asked for."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def tile(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    (d / "h.cpp").write_text('#include "hrm_tiles.h"\n'
                             'extern "C" long tile(long most, long cells, long blocks) { return hrm::cell_tile(most, cells, blocks); }')
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(ROOT, "paper_2208_04488_gb300", "csrc"),
                    str(d / "h.cpp"), "-o", str(d / "h.so")], check=True)
    f = ctypes.CDLL(str(d / "h.so")).tile
    f.restype, f.argtypes = ctypes.c_long, [ctypes.c_long] * 3
    return f


@pytest.mark.parametrize("cells", [1, 127, 9000, 24 * 6000, 1 << 20, 11_350_000, 1 << 33])
@pytest.mark.parametrize("blocks", [152, 456, 912])
@pytest.mark.parametrize("most", [256, 1024, 4096, 16384])
def test_items_feed_every_block(tile, most, cells, blocks):
    t = tile(most, cells, blocks)
    assert 1 <= t <= most and t % 128 == 0
    if t > 128:  # (128 cells are what a block takes at a time)
        assert (t - 128) * 2 * blocks < cells
    if cells >= 2 * blocks * most:
        assert t == most


def test_default_can_be_set_again(tile):
    """24 instances of 6000 cells: the default shape (4096) and all candidates give the item that creation gives."""
    assert {tile(most, 24 * 6000, 912) for most in (1024, 4096, 16384)} == {128}
