"""The tiled fp32 passes where their last tile is partly empty: the narrow tile at d = 64 (up to 32
slots; the statistics and the deslice), and last tiles of 1 to 9 slots and of half a tile, whose
warps and products past the slots are left out; and grids of several waves (59,000 points), which
take the instantiations with more resident blocks.  Oracle and bars of test_simt_tiles_gpu.
"""
import pytest

from test_simt_tiles_gpu import test_tile_edges as check

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 2, 64, 1, "f32"), (1, 127, 2, 64, 15, "bf16"), (2, 128, 1, 64, 16, "f32"), (1, 129, 3, 64, 17, "f32"),
          (2, 300, 2, 64, 31, "bf16"), (1, 300, 2, 64, 33, "f32"), (1, 200, 2, 32, 8, "f32"), (1, 200, 2, 32, 72, "f32"),
          (1, 200, 2, 16, 73, "f32"), (2, 257, 1, 16, 96, "bf16"), (1, 129, 2, 64, 97, "f32"), (1, 129, 2, 16, 17, "f32"),
          (1, 59001, 1, 16, 17, "f32"), (1, 59001, 1, 16, 65, "bf16"), (4, 15000, 1, 32, 20, "f32")]


@pytest.mark.parametrize("fused", [True, False], ids=["fused", "separate"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B{}N{}H{}d{}G{}{}".format(*s))
def test_partly_empty_tiles(lib, shape, fused):
    check(lib, shape, fused)
