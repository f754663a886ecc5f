"""GPU parity of the estimator where a node's registers are all 1: their exact
harmonic sum is then m 2^(64 - p) = 2^64 and no longer fits 64 bits, which a lane
reaches alone where a node's registers are 16 bytes (p = 4, or p = 5 packed).
"""
import numpy as np
import pytest

import oracle
from test_gpu_codes import check, vga  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SEED = 9


def _graph(p):
    """A complete graph of nodes with register indices 0 .. m - 1 and a rho of 1, the others without edges."""
    n, m = 64 << p, 1 << p
    regs = oracle.hll_init(n, p, SEED)
    members = [int(np.flatnonzero(regs[:, j] == 1)[0]) for j in range(m)]
    row_ptr, lists = np.zeros(n + 1, np.uint64), []
    for v in range(n):
        if v in members:
            lists.append(np.array(sorted(set(members) - {v}), np.uint32))
        row_ptr[v + 1] = row_ptr[v] + (m - 1 if v in members else 0)
    off, b = oracle.csr_encode(row_ptr, np.concatenate(lists))
    after = oracle.hyperball(off, b, p, 1, seed=SEED, trace=1)
    assert (after["regs"][1][members] == 1).all() and np.isfinite(after["c"][1]).all()
    return off, b


@pytest.mark.parametrize("p,bits,mode", [(4, 8, 0), (4, 8, 1), (5, 4, 0), (5, 8, 0), (6, 4, 0), (8, 8, 0)])
def test_registers_all_one(vga, p, bits, mode):  # noqa: F811
    off, b = _graph(p)
    check(vga, off, b, None, p, 3, SEED, bits, union_mode=mode)


def test_registers_all_one_in_a_batch(vga):  # noqa: F811
    off, b = _graph(4)
    ref = oracle.hyperball(off, b, 4, 3, seed=SEED)
    with vga.vga_graph_load(off, b) as g:
        md, ball = (torch.empty(g.n_nodes, dtype=torch.float64, device="cuda") for _ in range(2))
        its = vga.hyperball_run_batch([dict(graph=g, p=4, d=3, seed=SEED, mean_depth=md, ball=ball)])
        assert its == [ref["iterations"]]
        assert np.array_equal(md.cpu().numpy(), ref["mean_depth"]) and np.array_equal(ball.cpu().numpy(), ref["ball"])
