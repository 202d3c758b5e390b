"""The window rule of test_window_geometry.py at the size that the 2D tile kernel has now (768
nodes for a chunk of 512 slots; that file's 2,048 were those of chunks of 2,048), the cut to
the capacity taken more often: the same chunks, wide boxes that are cut in both directions,
and what a sorted chunk of 512 slots keeps inside."""
import numpy as np
import pytest

import test_window_geometry as geo


@pytest.fixture(autouse=True)
def _size(monkeypatch):
    monkeypatch.setattr(geo, "K_WIN", 768)


@pytest.mark.parametrize("nx,ny", [(1024, 1024), (256, 48), (64, 40), (2, 9), (4096, 8), (383, 5), (768, 3)])
def test_window_nodes_are_the_cells_nodes(nx, ny):
    geo.test_window_nodes_are_the_cells_nodes(nx, ny)


@pytest.mark.parametrize("width,height", [(700, 1), (380, 3), (100, 20), (20, 100), (1000, 9), (3, 300)])
def test_boxes_beyond_the_capacity_are_cut(width, height):
    nx, ny = 1024, 512
    cells = ((100 + np.arange(height))[:, None] * nx + (900 + np.arange(width)) % nx).ravel()
    ww, wx0, wy0, wh = geo.window(cells, nx, ny, int(cells[len(cells) // 2]))
    assert ww <= 384 and ww * wh <= 768 and wh >= 2
    # what is taken is taken right; the others (all of them where the box is wider than half the
    # capacity: two rows of nodes hold no cell of the chunk's) go to global memory
    assert geo.check_chunk(cells, nx, ny) < cells.size


def test_a_sorted_chunk_with_drift_is_taken_whole():
    """512 slots sorted at 32 particles per cell (16 cells of a row), each cell then moved by up
    to 8 cells in x and y: the window holds the nodes of every cell and of every cell one more
    step can reach."""
    nx, ny = 1024, 1024
    rng = np.random.default_rng(5)
    cells = 500 * nx + 700 + np.repeat(np.arange(16), 32)
    cy, cx = np.divmod(cells, nx)
    cx = cx + rng.integers(-8, 9, cells.size)
    cy = cy + rng.integers(-8, 9, cells.size)
    geo.check_chunk(cy * nx + cx, nx, ny, expect_all=True)
