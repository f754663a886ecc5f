"""GPU test of runs whose workspace has no room for the code passes' arrays
(csrc/codes.cuh): a workspace of the bytes that the byte union takes, such as
one sized for a larger graph, and a server whose budget is that small.  They run
over bytes with the same results; a byte less is refused.
"""
import ctypes as C

import numpy as np
import pytest

import oracle
from test_gpu_codes import _components, graph, vga  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _up(x):
    return (x + 255) // 256 * 256


def _least(vga, g, p):  # noqa: F811
    """The workspace without window, full marks and list (a piece: 16 registers)."""
    n, m = g.n_nodes, 1 << p
    pieces = n * m // 16
    entries = max(n, pieces) if pieces <= 1 << 16 else n
    return vga.hyperball_workspace_bytes(g, p) - _up(10 * m) - _up(n) - _up(8 * entries)


def _run(vga, g, p, size):  # noqa: F811
    n = g.n_nodes
    md, ball = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    ws = torch.full((size + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    at, it = -ws.data_ptr() % 256, C.c_int()
    status = vga.lib().hyperball_run_dev(g.handle, p, 0, 3, 0, md.data_ptr(), ball.data_ptr(), C.byref(it),
                                         ws.data_ptr() + at, size, None, None)
    assert bool((ws[at + size:] == 0xA5).all())
    return status, md.cpu().numpy(), ball.cpu().numpy(), it.value


def _same(got, ref):
    assert got[0] == 0 and got[3] == ref["iterations"]
    assert np.array_equal(got[1], ref["mean_depth"], equal_nan=True) and np.array_equal(got[2], ref["ball"])


@pytest.mark.parametrize("name,p", [("tiny", 7), ("corridor", 10), ("rect60", 10), ("components", 9)])
def test_workspace_without_room_for_codes(vga, name, p):  # noqa: F811
    off, b, comp = graph(name)
    ref = oracle.hyperball(off, b, p, 0, seed=3, comp_size=comp)
    with vga.vga_graph_load(off, b, comp) as g:
        least = _least(vga, g, p)
        _same(_run(vga, g, p, least), ref)
        _same(_run(vga, g, p, vga.hyperball_workspace_bytes(g, p) - 1), ref)
        assert _run(vga, g, p, least - 1)[0] == vga.VGA_EINVAL


def test_workspace_of_a_larger_graph(vga):  # noqa: F811
    # at p = 8 a graph of 4,096 nodes lists all its pieces, one of 4,097 one a node
    off, b, comp = _components([64] * 64)
    ref = oracle.hyperball(off, b, 8, 0, seed=3, comp_size=comp)
    with vga.vga_graph_load(*_components([64] * 64 + [1])) as larger:
        size = vga.hyperball_workspace_bytes(larger, 8)
    with vga.vga_graph_load(off, b, comp) as g:
        _same(_run(vga, g, 8, size), ref)


def test_server_budget_without_room_for_codes(vga):  # noqa: F811
    off, b, comp = graph("rect60")
    ref = oracle.hyperball(off, b, 10, 3, seed=3, comp_size=comp)
    with vga.vga_graph_load(off, b, comp) as g:
        budget = _up(_least(vga, g, 10)) + _up(16 * g.n_nodes)
        with vga.Server(hbm_budget_bytes=budget, solo_nodes=1) as server:
            done = server.wait(server.submit(g, 10, 3, 3))
        assert done["iterations"] == ref["iterations"]
        assert np.array_equal(done["mean_depth"], ref["mean_depth"]) and np.array_equal(done["ball"], ref["ball"])
        with vga.Server(hbm_budget_bytes=budget - 256, solo_nodes=1) as server:
            with pytest.raises(vga.VgaError):
                server.submit(g, 10, 3, 3)
