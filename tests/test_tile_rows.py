"""Tiles of the CUDA-core in-place pass (host arithmetic)."""
import pytest

from paper_2601_17261_b200 import binding as B

BLOCK_0P6B = [(1024, 2048), (1024, 1024), (1024, 1024), (2048, 1024), (1024, 3072), (1024, 3072), (3072, 1024)]
BLOCK_8B = [(4096, 4096), (4096, 1024), (4096, 1024), (4096, 4096), (4096, 12288), (4096, 12288), (12288, 4096)]


def layers_of(shapes, r, f32=True, pair=False):
    out, at = [], 1 << 32
    for i, (d_in, d_out) in enumerate(shapes):
        out.append(B.agzo_layer(at, d_in, at if pair else None, d_in, None, 0, 256, d_in, B.AGZO_F32 if f32 else B.AGZO_BF16, 0, d_out,
                                d_in, 0, r, i, 0))
        at += 4 * d_in * d_out + 4096 & -256
    return out


@pytest.mark.parametrize("r", [1, 4, 8, 16, 24])
@pytest.mark.parametrize("shapes", [BLOCK_0P6B * 2, BLOCK_8B * 4, [(1024, 1024)] * 8])
def test_a_layer_element_by_element_leaves_the_others_their_tiles(shapes, r):
    odd = [(1001, 1001)]
    both = B.agzo_debug_tile_rows(layers_of(shapes + odd, r))
    assert both == (B.agzo_debug_tile_rows(layers_of(shapes, r))[0], B.agzo_debug_tile_rows(layers_of(odd, r))[1])
    assert both[1] <= 32


def test_lists_that_memory_bounds():
    # heights measured as the best ones, or within 2 % of them; by the rounds alone these lists got others
    assert [B.agzo_debug_tile_rows(layers_of(BLOCK_0P6B * 2, r))[0] for r in (1, 2, 3, 4)] == [32] * 4
    assert B.agzo_debug_tile_rows(layers_of(BLOCK_8B * 4, 4))[0] == 32
    assert B.agzo_debug_tile_rows(layers_of([(2048, 2048)] * 24, 2))[0] == 32
    assert B.agzo_debug_tile_rows(layers_of([(1024, 1024)] * 30, 1, f32=False))[0] > 64
    assert B.agzo_debug_tile_rows(layers_of(BLOCK_8B, 2, f32=False))[0] == 128
    # strips of which a fifth is empty stay with the rounds, and so does a list of 60 MB
    assert B.agzo_debug_tile_rows(layers_of([(1640, 1640)] * 20, 4))[0] > 64
    assert B.agzo_debug_tile_rows(layers_of(BLOCK_0P6B, 4))[0] > 64


def test_large_16_bit_lists_of_ranks_3_and_4_keep_the_tallest_tiles():
    # their set-up is what the power cap takes from the pass: with it active 128 rows are 2 to 3 % slower than 256
    for blocks in (BLOCK_8B * 10, BLOCK_0P6B * 56):
        assert [B.agzo_debug_tile_rows(layers_of(blocks, r, f32=False))[0] for r in (1, 2, 3, 4)] == [128, 128, 256, 256]
