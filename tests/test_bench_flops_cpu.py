"""The matrix work that bench.py credits to the separable kernels, against their layouts: M = 128
rows and K = 16 per MMA, two FLOP per multiply-add."""
import bench


def test_separable_degridder_flop_follow_its_tile():
    # one tile: 128 visibilities (rows), every (polarisation, y, re/im) column, K = (x, cos/sin) for
    # hi x hi, hi x lo, lo x hi and the w remainder
    for L in (32, 24, 16):
        assert bench.SEP_DEGRID_TILE == 128
        assert bench.sep_degrid_flop_per_tile(L) == 2 * 128 * (4 * L * 2) * (2 * L) * 4


def test_separable_gridder_flop_follow_its_group():
    # one group of 8 visibilities (K = 16): A hi against 6 L rows of B, A lo against 2 L
    for L in (32, 24, 16):
        assert bench.sep_grid_flop_per_group(L) == 2 * 128 * 16 * 8 * L
