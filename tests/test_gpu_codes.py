"""GPU parity of the passes that gather register codes (csrc/codes.cuh).

From the second pass on, runs with an automatic slice width gather 4-bit or
1-bit codes of the registers and recompute from the bytes whatever a code pass
leaves open.  Every pass must equal the oracle's registers and estimates bit
for bit: where the codes settle everything, where most pairs stay open
(several components, long corridors), where a register's window does not
reach down to 0 (a rho above 15 on a graph of small balls), in both register
formats, both table schemes, one slice and many, and at the precisions where a
code row is as narrow as it can be.
"""
import ctypes

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vga():
    from paper_2604_08374_gb300 import build
    build.build()
    import paper_2604_08374_gb300 as v
    return v


def _corridor(n_rooms, size):
    """Rooms in a row joined by one-cell doors: a pass reaches one room on."""
    w = n_rooms * (size + 1) - 1
    grid = np.zeros((size, w), np.uint8)
    grid[:, size::size + 1] = 1
    for k in range(n_rooms - 1):
        grid[(k * 3) % size, size + k * (size + 1)] = 0
    return grid


def _components(sizes):
    """Complete graphs side by side: (offsets, bytes, component sizes)."""
    lists, comp, base = [], [], 0
    for s in sizes:
        ids = np.arange(base, base + s, dtype=np.uint32)
        for v in range(s):
            lists.append(np.delete(ids, v))
            comp.append(s)
        base += s
    row_ptr = np.zeros(len(lists) + 1, np.uint64)
    row_ptr[1:] = np.cumsum([len(x) for x in lists])
    off, b = oracle.csr_encode(row_ptr, np.concatenate(lists))
    return off, b, np.array(comp, np.uint32)


_cache = {}


def graph(name):
    if name not in _cache:
        comp = None
        if name == "components":
            off, b, comp = _components([1, 3, 40, 2, 500, 17, 260, 1, 96])
        else:
            obst = {"tiny": lambda: workloads.tiny(1), "corridor": lambda: _corridor(12, 9),
                    "rect60": lambda: workloads.rectangles_until(61, 59, (2, 12), 3100, seed=4),
                    "open": lambda: workloads.open_grid(37, 29)}[name]()
            off, b, _ = oracle.build_graph(obst)
        _cache[name] = (off, b, comp)
    return _cache[name]


def _seed_with_rho_above(n, p, at_least):
    """A hash seed for which some node's rho is at least `at_least`."""
    for seed in range(0, 4000 << 10, 1 << 10):  # (id ^ seed) takes new values for every seed
        if oracle.hll_init(n, p, seed).max() >= at_least:
            return seed
    raise AssertionError("no such seed")


def trace(vga, g, p, d, seed, conv, tuning, max_trace=12):
    """hyperball_run_trace with any tuning field."""
    n, m = g.n_nodes, 1 << p
    md, ball = np.zeros(n), np.zeros(n)
    regs, c = np.zeros((max_trace + 1, n, m), np.uint8), np.zeros((max_trace + 1, n))
    it = ctypes.c_int()
    status = vga.lib().hyperball_run_trace(g.handle, p, d, seed, conv, md.ctypes.data, ball.ctypes.data,
                                           ctypes.byref(it), regs.ctypes.data, c.ctypes.data, max_trace, tuning)
    assert status == 0, vga.lib().vga_last_error()
    return {"iterations": it.value, "regs": regs, "c": c, "mean_depth": md, "ball": ball}


def check(vga, off, b, comp, p, d, seed, bits, conv=0, **kw):
    ref = oracle.hyperball(off, b, p, d, seed=seed, trace=12, reg_bits=bits, conv_mode=conv, comp_size=comp)
    with vga.vga_graph_load(off, b, comp) as g:
        got = trace(vga, g, p, d, seed, conv, vga._tuning(register_bits=0 if bits == 8 else bits, **kw))
    assert got["iterations"] == ref["iterations"]
    for t in range(min(got["iterations"], 12) + 1):
        assert np.array_equal(got["regs"][t], ref["regs"][t]), f"registers differ after pass {t}"
        assert np.array_equal(got["c"][t], ref["c"][t]), f"estimates differ after pass {t}"
    assert np.array_equal(got["mean_depth"], ref["mean_depth"], equal_nan=True)
    assert np.array_equal(got["ball"], ref["ball"])


CASES = [
    # graph, p, d, register bits, table levels, L2 budget (MB; small: many slices)
    ("tiny", 10, 0, 8, 0, 0),
    ("tiny", 10, 3, 4, 3, 0),
    ("tiny", 5, 0, 8, 0, 0),       # one 16-byte row of 4-bit codes, no 1-bit row
    ("tiny", 7, 0, 8, 0, 0),       # the narrowest 1-bit row
    ("tiny", 6, 0, 4, 5, 0),
    ("corridor", 8, 0, 8, 0, 0),   # many passes, most registers open for long
    ("corridor", 10, 0, 4, 3, 1),
    ("rect60", 11, 0, 8, 0, 1),    # 64 slices of 32 bytes: no codes (more than 32)
    ("rect60", 10, 0, 8, 0, 1),    # slices of 64 bytes
    ("rect60", 9, 5, 8, 3, 0),
    ("open", 12, 0, 8, 0, 0),
    ("open", 13, 2, 4, 0, 0),
    ("components", 7, 0, 8, 0, 0),
    ("components", 10, 0, 8, 3, 0),
    ("components", 9, 0, 4, 0, 1),
]


@pytest.mark.parametrize("name,p,d,bits,levels,mb", CASES)
def test_code_passes_match_the_oracle(vga, name, p, d, bits, levels, mb):
    off, b, comp = graph(name)
    check(vga, off, b, comp, p, d, 3, bits, table_levels=levels, l2_budget_mb=mb)


@pytest.mark.parametrize("name,p", [("components", 7), ("corridor", 8), ("tiny", 10)])
def test_windows_that_do_not_reach_zero(vga, name, p):
    # a rho of 17 or more: the 4-bit window of its register starts at 2 or above
    off, b, comp = graph(name)
    check(vga, off, b, comp, p, 0, _seed_with_rho_above(len(off) - 1, p, 17), 8)


@pytest.mark.parametrize("track", [0, 1])
def test_stop_rule_and_tracking(vga, track):
    off, b, comp = graph("corridor")
    check(vga, off, b, comp, 10, 0, 5, 8, conv=1, track_changes=track)
