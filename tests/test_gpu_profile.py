"""GPU test of the profile (vga_profile) beside the code passes: passes of one-bit
codes, which have no fixed bytes, add neither launches nor time to the union's.
"""
import pytest

import oracle
import workloads
from test_gpu_codes import vga  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _profile(vga, g, p, d, **kw):  # noqa: F811
    md = torch.empty(g.n_nodes, dtype=torch.float64, device="cuda")
    vga.vga_profile_reset()
    vga.vga_profile_enable(True)
    try:
        it = vga.hyperball_run_dev(g, p, d, 7, md, None, track_changes=1, **kw)
        return it, vga.vga_profile_read()
    finally:
        vga.vga_profile_enable(False)


def test_one_bit_passes_are_not_union_launches(vga):  # noqa: F811
    # every node sees every other: pass 2 finds all registers at their maximum
    off, b, _ = oracle.build_graph(workloads.open_grid(37, 29))
    with vga.vga_graph_load(off, b) as g:
        it, prof = _profile(vga, g, 10, 2)
        assert it == 2 and prof["first_pass_launches"] == 1
        assert prof["union_launches"] == 0 and prof["union_ms"] == 0.0
        it, prof = _profile(vga, g, 10, 2, slice_bytes=256)  # over bytes: 4 slices
        assert it == 2 and prof["union_launches"] == 4 and prof["union_ms"] > 0.0
