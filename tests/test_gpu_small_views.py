"""GPU test of the code passes (csrc/codes.cuh) on graphs whose nodes see little:
a 4-bit pass that would leave more pieces open than are settled one by one is
left out for the byte union, and one that does so unforeseen is followed by it.
The registers are the oracle's; which kernels ran shows in the number of
launches.
"""
import numpy as np
import pytest

import oracle
from test_gpu_codes import check, vga  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, P = 4200, 8  # more than 65,536 pieces of 16 registers: the list holds one a node


def _band(reach=1, hub=None, hub_reach=0):
    """Node v sees v - reach ... v + reach; with `hub`, that node and the first hub_reach see each other, too."""
    row_ptr, lists = np.zeros(N + 1, np.uint64), []
    for v in range(N):
        ids = set(range(max(0, v - reach), min(N, v + reach + 1)))
        if hub is not None:
            ids |= set(range(hub_reach)) if v == hub else {hub} if v < hub_reach else set()
        lists.append(np.array(sorted(ids - {v}), np.uint32))
        row_ptr[v + 1] = row_ptr[v] + len(lists[v])
    return oracle.csr_encode(row_ptr, np.concatenate(lists))


def _spokes(n, hub, hub_reach):
    """A band of `n` nodes; nodes 100, 101, ... also see every 3rd, 15th, 16th, 120th, ... id (up to 1,334
    runs), and `hub` and the first hub_reach each other."""
    sees = [set(range(max(0, v - 1), min(n, v + 2))) for v in range(n)]
    for k, step in enumerate((3, 15, 16, 17, 120, 130, 140)):
        for u in range(0, n, step):
            sees[100 + k].add(u)
            sees[u].add(100 + k)
    for u in range(hub_reach):
        sees[hub].add(u)
        sees[u].add(hub)
    lists = [np.array(sorted(s - {v}), np.uint32) for v, s in enumerate(sees)]
    row_ptr = np.zeros(n + 1, np.uint64)
    row_ptr[1:] = np.cumsum([len(x) for x in lists])
    return oracle.csr_encode(row_ptr, np.concatenate(lists))


def _large(seed):
    """The nodes and register indices with a rho of 16 or more."""
    return np.nonzero(oracle.hll_init(N, P, seed) >= 16)


def _launches(vga, g, seed, d, **kw):  # noqa: F811
    md, ball = (torch.empty(N, dtype=torch.float64, device="cuda") for _ in range(2))
    counts = []
    for _ in range(2):  # the first run builds the graph's lists
        vga.vga_profile_reset()
        vga.hyperball_run_dev(g, P, d, seed, md, ball, track_changes=1, **kw)
        counts.append(vga.vga_profile_read()["kernel_launches"])
    return counts[1]


@pytest.mark.parametrize("reach", [1, 10])
def test_passes_that_would_leave_much_open_go_over_bytes(vga, reach):  # noqa: F811
    off, b = _band(reach)
    seed = 66772992
    assert len(set(_large(seed)[1] // 16)) == 3  # three pieces of every node start below the window
    check(vga, off, b, None, P, 6, seed, 8)
    with vga.vga_graph_load(off, b) as g:
        over_bytes = _launches(vga, g, seed, 3, slice_bytes=1 << P)
        assert _launches(vga, g, seed, 3) == over_bytes + 1  # the window
        ws = torch.empty(16 << 20, dtype=torch.uint8, device="cuda")
        over_bytes = _launches(vga, g, seed, 3, union_mode=1)
        # below 16 neighbours a node the per-neighbour union gathers no codes at all
        assert _launches(vga, g, seed, 3, union_mode=1, workspace=ws) == over_bytes + (reach == 10)


def _one_large():
    seed = next(s for s in range(0, 1 << 20, 1 << 13) if len(_large(s)[0]) == 1)
    return seed, int(_large(seed)[0][0]), int(_large(seed)[1][0])


def test_open_pieces_within_the_list(vga):  # noqa: F811
    # all but 700 nodes see the one large rho in pass 1
    seed, hub, _ = _one_large()
    off, b = _band(1, hub, 3500)
    check(vga, off, b, None, P, 4, seed, 8, track_changes=1)
    with vga.vga_graph_load(off, b) as g:
        # the window, and the open pieces with nothing behind them
        assert _launches(vga, g, seed, 2) == _launches(vga, g, seed, 2, slice_bytes=1 << P) + 2


def test_pass_that_leaves_more_open_than_foreseen(vga):  # noqa: F811
    # 1,500 nodes below the window after pass 1, and still about all of them after pass 2
    seed, hub, j = _one_large()
    off, b = _band(6, hub, 2600)
    below = [(r[:, j] == 0).sum() for r in oracle.hyperball(off, b, P, 2, seed=seed, trace=2)["regs"]]
    assert below[2] > 1300 and below[1] ** 2 < 600 * below[0]  # the list is good for about 1,170 pieces
    check(vga, off, b, None, P, 4, seed, 8, track_changes=1)
    with vga.vga_graph_load(off, b) as g:
        # as above, and the byte union of the open pairs behind them
        assert _launches(vga, g, seed, 2) == _launches(vga, g, seed, 2, slice_bytes=1 << P) + 4


@pytest.mark.parametrize("hub_reach", [0, 3500], ids=["many", "few"])
@pytest.mark.parametrize("levels", [5, 3])
def test_settling_of_open_pieces(vga, levels, hub_reach):  # noqa: F811
    # all pieces fit the list of a graph this small: 4-bit passes leave up to 4,000
    # open, of nodes with 1 to 1,335 range lookups
    n = 4000
    seed, hub, _ = _one_large()
    off, b = _spokes(n, hub, hub_reach)
    check(vga, off, b, None, P, 5, seed, 8, table_levels=levels)
    ref = oracle.hyperball(off, b, P, 5, seed=seed)
    with vga.vga_graph_load(off, b) as g:
        out = [[torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)] for _ in range(3)]
        jobs = [dict(graph=g, p=P, d=5, seed=seed, mean_depth=md, ball=ball) for md, ball in out]
        assert vga.hyperball_run_batch(jobs) == [ref["iterations"]] * 3
        for md, ball in out:
            assert np.array_equal(md.cpu().numpy(), ref["mean_depth"])
            assert np.array_equal(ball.cpu().numpy(), ref["ball"])


def test_narrow_rows_of_few_go_over_bytes(vga):  # noqa: F811
    # 9,000 nodes of a handful of rows each: no 4-bit pass at p = 9, one at p = 10
    n = 9000
    row_ptr = np.zeros(n + 1, np.uint64)
    lists = [np.array([u for u in range(max(0, v - 9), min(n, v + 10)) if u != v], np.uint32) for v in range(n)]
    row_ptr[1:] = np.cumsum([len(x) for x in lists])
    off, b = oracle.csr_encode(row_ptr, np.concatenate(lists))
    seed = next(s for s in range(0, 1 << 20, 1 << 14)
                if max(oracle.hll_init(n, p, s).max() for p in (9, 10)) < 16)  # the window reaches 0
    with vga.vga_graph_load(off, b) as g:
        md, ball = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))

        def launches(p, **kw):
            for _ in range(2):
                vga.vga_profile_reset()
                it = vga.hyperball_run_dev(g, p, 2, seed, md, ball, track_changes=1, **kw)
            ref = oracle.hyperball(off, b, p, 2, seed=seed)
            assert it == 2 and np.array_equal(md.cpu().numpy(), ref["mean_depth"])
            return vga.vga_profile_read()["kernel_launches"]

        assert launches(9) == launches(9, slice_bytes=512)
        assert launches(10) == launches(10, slice_bytes=1024) + 2  # the window and the (no) open pieces
        jobs = [dict(graph=g, p=p, d=3, seed=seed, mean_depth=torch.empty(n, dtype=torch.float64, device="cuda"),
                     ball=torch.empty(n, dtype=torch.float64, device="cuda")) for p in (9, 10)]
        vga.hyperball_run_batch(jobs)
        for job in jobs:
            ref = oracle.hyperball(off, b, job["p"], 3, seed=seed)
            assert np.array_equal(job["mean_depth"].cpu().numpy(), ref["mean_depth"])


def test_open_slices_after_a_pass_over_many(vga):  # noqa: F811
    # as above with 8 slices of 32 registers: the byte union of the one slice with open pairs
    seed, hub, j = _one_large()
    off, b = _band(6, hub, 2600)
    check(vga, off, b, None, P, 4, seed, 8, track_changes=1, l2_budget_mb=1)
    with vga.vga_graph_load(off, b) as g:
        # bytes: 8 tables and unions; codes: 4 and 4, the window, the open pieces, a table and a union
        assert _launches(vga, g, seed, 2, l2_budget_mb=1) == _launches(vga, g, seed, 2, slice_bytes=32) - 16 + 12
