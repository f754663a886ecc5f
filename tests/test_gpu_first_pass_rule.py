"""GPU test of the rule for the first pass's scatter: whole groups of nodes where
nodes see much, one by one where they see little (csrc/vga_common.cuh,
group_scatter_pays); either way the oracle's registers.
"""
import pytest

import oracle
import workloads
from test_gpu_codes import _components, _corridor, check, vga  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _graph(name):
    if name == "rooms":  # 6,084 cells, a few hundred neighbours each
        return oracle.build_graph(_corridor(19, 18))[:2] + (None,)
    if name == "site":  # 2,500 cells, half of them neighbours
        return oracle.build_graph(workloads.rectangles_until(53, 53, (2, 10), 2500, seed=4))[:2] + (None,)
    return _components([1500, 1024])  # complete graphs


@pytest.mark.parametrize("name,p,grouped", [("rooms", 8, 0), ("rooms", 10, 0), ("site", 8, 1), ("site", 12, 0),
                                            ("components", 8, 1), ("components", 13, 0)])
def test_first_pass_by_degree(vga, name, p, grouped):  # noqa: F811
    off, b, comp = _graph(name)
    check(vga, off, b, comp, p, 1, 5, 8)
    with vga.vga_graph_load(off, b, comp) as g:
        assert grouped == (g.n_edges >= g.n_nodes * (768 + (1 << p) // 4))
        assert g.n_nodes >= 8 * torch.cuda.get_device_properties(0).multi_processor_count
        md, ball = (torch.empty(g.n_nodes, dtype=torch.float64, device="cuda") for _ in range(2))
        vga.vga_profile_reset()
        vga.vga_profile_enable(True)
        try:
            vga.hyperball_run_dev(g, p, 1, 5, md, ball)
            prof = vga.vga_profile_read()
        finally:
            vga.vga_profile_enable(False)
        assert prof["first_pass_launches"] == 1 and prof["first_pass_grouped"] == grouped
