"""GPU parity of the first pass's grouped scatter (csrc/first_pass.cuh), which
runs with an automatic slice width take while there are at most 2,048 nodes a
register index: every register after every pass equals the oracle's, at the
key widths' edges (p = 12, 13), in both register formats and table schemes, with
groups of fewer than four nodes, without edges, and where several keys of one
register index have a rho of 16 or more, which the scatter has no level for.
"""
import numpy as np
import pytest

import oracle
from test_gpu_codes import check, graph, vga  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,p,d,bits,levels", [
    ("tiny", 5, 1, 8, 0), ("tiny", 12, 2, 8, 3), ("tiny", 13, 1, 8, 0), ("corridor", 9, 2, 8, 5),
    ("corridor", 13, 1, 4, 0), ("rect60", 10, 2, 8, 3), ("rect60", 12, 1, 4, 5), ("open", 11, 1, 8, 3),
    ("components", 6, 1, 4, 0), ("components", 8, 2, 8, 0),
])
def test_first_pass_matches_the_oracle(vga, name, p, d, bits, levels):  # noqa: F811
    off, b, comp = graph(name)
    check(vga, off, b, comp, p, d, 11, bits, table_levels=levels)


def _keys(n, p, seeds):
    """(register index, rho) of every node under each seed: Alg. 1's hash."""
    u = np.uint64
    with np.errstate(over="ignore"):
        x = (np.arange(n, dtype=u)[None, :] ^ seeds[:, None]) + u(0x9E3779B97F4A7C15)
        x = (x ^ (x >> u(30))) * u(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> u(27))) * u(0x94D049BB133111EB)
        x ^= x >> u(31)
        return (x >> u(64 - p)).astype(np.int64), (x << u(p)) < (u(1) << u(49))  # rho >= 16


def _seed_with_two_large(n, p):
    """A seed under which two nodes of one register index have different rho >= 16."""
    for first in range(1, 400_000, 1000):
        seeds = np.arange(first, first + 1000, dtype=np.uint64) << np.uint64(12)
        j, large = _keys(n, p, seeds)
        for s in np.flatnonzero(large.sum(1) >= 2):
            ids = np.flatnonzero(large[s])
            regs = oracle.hll_init(n, p, int(seeds[s]))[ids]
            for reg in np.unique(j[s, ids]):
                rhos = regs[j[s, ids] == reg, reg]
                if rhos.min() >= 16 and len(np.unique(rhos)) > 1:
                    return int(seeds[s])
    raise AssertionError("no such seed")


@pytest.mark.parametrize("name", ["corridor", "components", "open"])
def test_registers_with_several_large_rho(vga, name):  # noqa: F811
    off, b, comp = graph(name)
    check(vga, off, b, comp, 5, 2, _seed_with_two_large(len(off) - 1, 5), 8)
