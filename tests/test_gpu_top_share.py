"""GPU test of the choice of one-bit passes (csrc/vga_common.cuh, mostly_at_top):
registers that no node raises do not count as having reached their maximum.  On
a graph of far fewer nodes than registers the second pass gathers 4-bit codes,
which settle it, and in a batch, too, results are the oracle's.
"""
import numpy as np
import pytest

import oracle
import workloads
from test_gpu_codes import check, vga  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bits", [8, 4])
def test_few_nodes_many_registers(vga, bits):  # noqa: F811
    off, b, _ = oracle.build_graph(workloads.rectangles_until(29, 29, (2, 8), 690, seed=1))
    n, p = len(off) - 1, 12
    seed = next(s for s in range(0, 1 << 20, 1 << 12) if oracle.hll_init(n, p, s).max() < 16)
    check(vga, off, b, None, p, 4, seed, bits)
    with vga.vga_graph_load(off, b) as g:
        md, ball = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))

        def launches(**kw):
            for _ in range(2):
                vga.vga_profile_reset()
                vga.hyperball_run_dev(g, p, 2, seed, md, ball, register_bits=0 if bits == 8 else 4, **kw)
            return vga.vga_profile_read()["kernel_launches"]

        # 4,096 registers: 2 slices of 4-bit codes, the open pieces and the window, for 4 (packed 2) byte slices
        assert launches() == launches(slice_bytes=1024) + 2 * 2 + 2 - 2 * bits // 2
        out = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)]
        its = vga.hyperball_run_batch([dict(graph=g, p=p, d=0, seed=seed, mean_depth=out[0], ball=out[1])])
    ref = oracle.hyperball(off, b, p, 0, seed=seed)
    assert its == [ref["iterations"]] and np.array_equal(out[0].cpu().numpy(), ref["mean_depth"])
