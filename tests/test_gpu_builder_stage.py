"""GPU parity of the visibility builder's way without the bit matrix where its
stage is sized by a sample of the sources (above 256 MB of bound, some 16,000
nodes), and where the stage then fills up and the lists left out are swept again.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vga():
    from paper_2604_08374_gb300 import build
    build.build()
    import paper_2604_08374_gb300 as v
    return v


def _uneven():
    """27,000 cells, a hall in one corner and closets elsewhere: lists of very different lengths."""
    grid = workloads.rectangles_until(190, 190, (1, 3), 26_000, seed=8)
    grid[:70, :70] = 0
    return grid


@pytest.mark.parametrize("cap,nodes", [(0, 1 << 20), (0, 1), (47, 1 << 20)], ids=["sampled", "global", "full"])
@pytest.mark.parametrize("order", ["raster", "hilbert"])
def test_sampled_stage_gives_the_matrix_graph(vga, cap, nodes, order):
    obst = _uneven()
    assert vga.vga_visibility_count(obst) > 17_000
    with vga.vga_visibility_build(obst, order=order) as g:
        want = g.copy_csr()
    vga.vga_set_visibility_sweep_limits(cap, nodes)
    try:
        with vga.vga_visibility_build(obst, order=order) as g:
            got = g.copy_csr()
    finally:
        vga.vga_set_visibility_sweep_limits(0, 0)
    assert all(np.array_equal(x, y) for x, y in zip(got, want))
