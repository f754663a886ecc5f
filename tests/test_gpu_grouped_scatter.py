"""GPU parity of the first pass's grouped scatter (csrc/first_pass.cuh) on graphs
that take it in single analyses and in batches: two groups of four nodes an SM
at least, and a mean degree from which it pays.  The key widths' edges, both
register formats and table schemes, groups of fewer than four nodes, nodes
without edges, and register indices with several keys of a rho of 16 or more,
whose largest one is searched among a node's ids.
"""
import numpy as np
import pytest

import oracle
from test_gpu_codes import _components, check, vga  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _grouped(vga, g, p, bits=8, **kw):  # noqa: F811
    """First passes by whole groups in one profiled run."""
    md = torch.empty(g.n_nodes, dtype=torch.float64, device="cuda")
    vga.vga_profile_reset()
    vga.vga_profile_enable(True)
    try:
        vga.hyperball_run_dev(g, p, 1, 1, md, None, register_bits=0 if bits == 8 else bits, **kw)
        return vga.vga_profile_read()["first_pass_grouped"]
    finally:
        vga.vga_profile_enable(False)


def _graph(p):
    """Complete graphs of the degree that p asks for, a triangle and single nodes: n is 3 mod 4."""
    size = 776 + (1 << p) // 4
    sizes = [size] * max(1, -(-1300 // size)) + [3, 1, 1]
    sizes[0] += (3 - sum(sizes)) % 4
    return _components(sizes)


@pytest.mark.parametrize("p,bits,levels,d", [(5, 8, 0, 2), (6, 4, 3, 2), (8, 8, 3, 2), (9, 4, 5, 1), (10, 8, 5, 2),
                                             (12, 8, 3, 1), (12, 4, 0, 1), (13, 8, 0, 1), (13, 4, 3, 1)])
def test_grouped_scatter_matches_the_oracle(vga, p, bits, levels, d):  # noqa: F811
    off, b, comp = _graph(p)
    with vga.vga_graph_load(off, b, comp) as g:
        assert g.n_nodes % 4 == 3
        assert _grouped(vga, g, p, bits, table_levels=levels) == 1
    check(vga, off, b, comp, p, d, 11, bits, table_levels=levels)


# Two nodes of one register index with different rho >= 16, in one of two complete graphs of 900 or one in each.
LARGE = [(5, 225456128, (1253, 1507)), (5, 193564672, (794, 1488)), (7, 2460184576, (1092, 1269)),
         (7, 269475840, (143, 1446))]


@pytest.mark.parametrize("p,seed,nodes", LARGE)
@pytest.mark.parametrize("levels", [5, 3])
def test_several_large_rho_of_one_index(vga, p, seed, nodes, levels):  # noqa: F811
    off, b, comp = _components([900, 900])
    regs = oracle.hll_init(1800, p, seed)[list(nodes)]
    j = regs.argmax(1)
    assert j[0] == j[1] and regs.max(1).min() >= 16 and len(set(regs.max(1).tolist())) == 2
    check(vga, off, b, comp, p, 2, seed, 8, table_levels=levels)
    ref = oracle.hyperball(off, b, p, 2, seed=seed, comp_size=comp)
    with vga.vga_graph_load(off, b, comp) as g:
        assert _grouped(vga, g, p, table_levels=levels) == 1
        md, ball = (torch.empty(1800, dtype=torch.float64, device="cuda") for _ in range(2))
        vga.hyperball_run_batch([dict(graph=g, p=p, d=2, seed=seed, mean_depth=md, ball=ball)])
        assert np.array_equal(md.cpu().numpy(), ref["mean_depth"]) and np.array_equal(ball.cpu().numpy(), ref["ball"])
