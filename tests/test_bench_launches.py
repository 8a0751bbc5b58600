"""bench.launches_per_step on the grids whose transforms are the library's own, and at the sizes whose vector work
is one kernel: per iteration spread, transforms (three kernels, or the product between cuFFT's), gather, pairs and
vectors (one kernel up to 16,384 slots, else three)."""
import bench


def test_own_transforms():
    for grid in ((24, 24, 24), (64, 64, 64), (50, 64, 80), (96, 96, 96), (28, 32, 40), (10, 10, 10)):
        assert bench.own_transforms(grid), grid
    for grid in ((100, 100, 100), (224, 224, 224), (22, 20, 20), (26, 64, 64), (256, 256, 8)):
        assert not bench.own_transforms(grid), grid


def test_kernels_per_iteration():
    def per(n, grid):
        return bench.launches_per_step(5, n, 0.0, 0, grid) - bench.launches_per_step(4, n, 0.0, 0, grid)

    assert per(96000, (100, 100, 100)) == 7
    assert per(23558, (64, 64, 64)) == 9
    assert per(16384, (54, 54, 54)) == 7 and per(16385, (54, 54, 54)) == 9
    assert per(648, (24, 24, 24)) == 7 and per(648, (22, 22, 22)) == 5


def test_whole_step():
    # load, lists, spread, 3, gather, pairs, assemble | guess, spread, 3, gather, pairs, residual, direction,
    # condition, 8 x 7, unsort | dipoles, spread, 3, derivatives twice, energy, pairs, atoms, frames, unsort
    assert bench.launches_per_step(8, 640, 0.0, 0, (24, 24, 24)) == 9 + (1 + 6 + 3 + 56 + 1) + 12
    # one more for the padding of a ragged last block, and for the blocks' boxes from eight blocks an SM on
    assert bench.launches_per_step(8, 648, 0.0, 0, (24, 24, 24)) - bench.launches_per_step(8, 640, 0.0, 0, (24, 24, 24)) == 1
    a, b = (bench.launches_per_step(8, 32 * k, 0.0, 0, (100, 100, 100)) for k in (1216, 1215))
    assert a - b == 1
