"""The visibility builder where the device's memory is nearly all taken: its bit
matrix (N^2 / 8 bytes) is far larger than the graph of a plan of rooms, and a
build that finds room for the matrix but not for what goes with it takes the
way without the matrix instead of failing.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
MB = 1 << 20


@pytest.fixture(scope="module")
def vga():
    from paper_2604_08374_gb300 import build
    build.build()
    import paper_2604_08374_gb300 as v
    return v


def _rooms(count, size):
    """count x count rooms of size x size cells, joined by one-cell doors."""
    side = count * (size + 1) - 1
    grid = np.zeros((side, side), np.uint8)
    grid[size::size + 1, :] = 1
    grid[:, size::size + 1] = 1
    at = np.arange(count) * (size + 1) + size // 2
    grid[size::size + 1, at] = 0
    grid[at[:, None], np.arange(size, side, size + 1)[None, :]] = 0
    return grid


def _csr(vga, obst):
    with vga.vga_visibility_build(obst) as g:
        off, b, _ = g.copy_csr()
    return off, b


def test_matrix_with_no_room_beside_it(vga):
    obst = _rooms(12, 20)
    n = vga.vga_visibility_count(obst)
    pitch = -(-n // 512) * 16
    matrix = 128 * pitch * pitch
    want = _csr(vga, obst)
    vga.vga_set_visibility_sweep_limits(0, 1 << 20)  # the way without the matrix: its kernels loaded, the same graph
    try:
        assert all(np.array_equal(x, y) for x, y in zip(_csr(vga, obst), want))
    finally:
        vga.vga_set_visibility_sweep_limits(0, 0)
    for over in range(0, 13):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        hold = torch.empty(free - matrix - over * MB, dtype=torch.uint8, device="cuda")
        try:
            got = _csr(vga, obst)
        finally:
            del hold
            torch.cuda.empty_cache()
        assert all(np.array_equal(x, y) for x, y in zip(got, want)), over
