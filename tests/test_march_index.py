"""The row-marching kernels' vertical bookkeeping, restated on the CPU.

Going down the rows of a strip, a level's state holds source rows i0 and
i1 = min(i0 + 1, H_l - 1); the next source row, min(i1 + 1, H_l - 1), is
staged ahead.  A row on which i0 grows moves the state by one source row.
The scheme needs i0 to grow by at most one per row, for every image height,
level and starting row, with i0 as the kernels' fp32 bilinear_tap gives it.
"""
import numpy as np
import pytest

from test_staging_coverage import level_size, tap32


def _i0(H, l):
    Hl = level_size(H, l)
    ratio = np.float32(Hl / H)
    i0, i1, _ = tap32(np.arange(H), ratio, Hl)
    return i0, i1, Hl


HEIGHTS = list(range(1, 300)) + [512, 683, 1080, 1361, 2160, 8191, 65535, 65536]


@pytest.mark.parametrize("L", [2, 4, 7, 8, 12])
def test_source_row_moves_by_at_most_one(L):
    for H in HEIGHTS:
        for l in range(1, L):
            i0, _, _ = _i0(H, l)
            step = np.diff(i0)
            assert step.size == 0 or (step.min() >= 0 and step.max() <= 1), (H, l)


@pytest.mark.parametrize("H", [1, 2, 3, 5, 31, 32, 33, 64, 65, 135, 257, 1080])
def test_marched_rows_are_the_defined_ones(H):
    for l in range(1, 8):
        i0, i1, Hl = _i0(H, l)
        for start in {0, 1, H // 3, H - 1} & set(range(H)):
            up, low = i0[start], i1[start]
            staged = min(low + 1, Hl - 1)
            for y in range(start, H):
                if y > start and i0[y] != i0[y - 1]:
                    up, low = low, staged
                    staged = min(staged + 1, Hl - 1)
                assert (up, low) == (i0[y], i1[y]), (H, l, start, y)
