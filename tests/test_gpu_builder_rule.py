"""GPU test of the builder's choice between the bit matrix and the way without it:
graphs whose nodes see little for their number take the latter, shown by the
number of launches, and both ways give the same CSR.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vga():
    from paper_2604_08374_gb300 import build
    build.build()
    import paper_2604_08374_gb300 as v
    return v


def _noise():  # views of about 5 cells
    return (np.random.default_rng(3).random((310, 310)) < 0.35).astype(np.uint8)


def _rooms():  # rooms of 16 x 16 cells in a column-major comb of doors
    grid = np.zeros((271, 271), np.uint8)
    grid[16::17, :] = 1
    grid[:, 16::17] = 1
    at = np.arange(16) * 17 + 3
    grid[16::17, at] = 0
    grid[at[:, None], np.arange(16, 271, 17)[None, :]] = 0
    return grid


def _build(vga, obst, nodes, order):
    vga.vga_set_visibility_sweep_limits(0, nodes)
    try:
        vga.vga_profile_reset()
        with vga.vga_visibility_build(obst, order=order) as g:
            return vga.vga_profile_read()["kernel_launches"], g.copy_csr()
    finally:
        vga.vga_set_visibility_sweep_limits(0, 0)


@pytest.mark.parametrize("order", ["raster", "hilbert"])
@pytest.mark.parametrize("grid,matrix", [(_noise, False), (_rooms, True)])
def test_matrix_where_the_nodes_see_enough(vga, grid, matrix, order):
    obst = grid()
    assert vga.vga_visibility_count(obst) > 50_000
    launches, csr = _build(vga, obst, 0, order)
    without, same = _build(vga, obst, 1 << 20, order)
    assert all(np.array_equal(x, y) for x, y in zip(csr, same))
    assert (launches != without) == matrix
