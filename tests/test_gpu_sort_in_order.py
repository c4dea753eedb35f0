"""The tile sort on arrays that are in order, whose warps add all of a bin's
particles at once: whole warps and ragged last ones, bins of less and of more
than a warp, table slots that several bins claim, and order that breaks off."""
import numpy as np
import pytest

from test_gpu_sort import _run

pytestmark = pytest.mark.gpu

SHAPES = {1: (1000, 1, 1), 2: (203, 97, 1), 3: (41, 33, 30)}


@pytest.mark.parametrize("n", [(1 << 17) + 1, (1 << 18) + 33, (1 << 19) + 2047, (1 << 19) + 31])
@pytest.mark.parametrize("dim", [1, 2, 3])
def test_cells_in_order(dim, n):
    cells = int(np.prod(SHAPES[dim]))
    _run(dim, SHAPES[dim], n, lambda rs, k: np.sort(rs.integers(0, cells, k)), seed=n % 1000 + dim)


@pytest.mark.parametrize("n", [300_000, 600_011])
def test_many_small_bins_in_order(n):
    # 2 x 2 tiles: 16,384 bins of 18 or 37 particles, some 60 to 110 to a chunk of the table's 1024 slots
    def cells(rs, k):
        x, y = np.arange(65536) % 256, np.arange(65536) // 256
        order = np.argsort((y // 2 * 128 + x // 2) * 4, kind="stable")  # tile by tile
        return order[np.sort(rs.integers(0, 65536, k))]

    _run(2, (256, 256, 1), n, cells, seed=n % 100, tile=[2, 2])


def test_order_in_parts_of_a_chunk():
    # 700 particles of one cell, then 500 anywhere, over and over: warps of both forms in a block
    def cells(rs, k):
        c = rs.integers(0, 65536, k)
        at = np.arange(k)
        return np.where(at % 1200 < 700, at // 1200 * 37 % 65536, c)

    _run(2, (256, 256, 1), 600_000, cells, seed=9)
