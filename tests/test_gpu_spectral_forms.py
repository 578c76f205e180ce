"""FP32 boxes of 2^20 cells and more that the spectral solve takes in its small
form: the check of test_spectral_lengths (residual below the tolerance within
the iterations that the contrast allows) on lines where the two forms' plans have
as many stages, save one or two, and save one of a long line off whole words."""
import pytest

from test_spectral_lengths import test_solve_in_boxes_of_every_length as solve

BOXES = [(512, 64, 32), (64, 64, 512), (16, 512, 128), (125, 128, 70), (343, 64, 48), (64, 175, 98), (128, 81, 128),
         (375, 64, 48), (162, 128, 64)]


# FP64 lines of 96, by their plan, along each axis
FP64_96 = [(96, 32, 32), (32, 96, 32), (30, 32, 96), (96, 96, 96)]

# FP64 boxes of fewer tiles of 32 lines than SMs: 8 or 16 lines a tile, rows of fewer cells than that, odd rows
FP64_TILES = [(32, 32, 192), (16, 64, 64), (64, 75, 64), (6, 10, 150), (15, 40, 32), (64, 64, 64), (8, 8, 8)]


@pytest.mark.gpu
@pytest.mark.parametrize("box", BOXES)
def test_small_form_of_large_boxes(lbeh, box):
    assert box[0] * box[1] * box[2] >= 1 << 20
    solve(lbeh, "fp32", box)


@pytest.mark.gpu
@pytest.mark.parametrize("box", FP64_96)
def test_fp64_lines_of_96(lbeh, box):
    solve(lbeh, "fp64", box)


@pytest.mark.gpu
@pytest.mark.parametrize("box", FP64_TILES)
def test_fp64_tiles(lbeh, box):
    solve(lbeh, "fp64", box)
