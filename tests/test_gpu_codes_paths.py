"""GPU parity of the code passes (csrc/codes.cuh) outside the single-graph
run-aware path: the batched engine, whose one-bit passes are done again in four
bits when they leave too much open, and the per-neighbour union with a
workspace that has room for codes (four bits, one bit only, or none).  Results
equal the oracle's bit for bit.
"""
import ctypes as C

import numpy as np
import pytest

import oracle
from test_gpu_codes import graph

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def vga():
    from paper_2604_08374_gb300 import build
    build.build()
    import paper_2604_08374_gb300 as v
    return v


def _same(got_md, got_ball, got_it, ref):
    assert got_it == ref["iterations"]
    assert np.array_equal(got_md, ref["mean_depth"], equal_nan=True)
    assert np.array_equal(got_ball, ref["ball"])


@pytest.mark.parametrize("use_graph", [True, False])
def test_batched_code_passes(vga, use_graph):
    # p = 6: no codes; 7: the narrowest one-bit rows; 13: four slices
    jobs, refs, keep = [], [], []
    for name, p, d, conv in (("tiny", 6, 0, 0), ("tiny", 7, 0, 0), ("corridor", 8, 0, 0), ("corridor", 10, 0, 1),
                             ("rect60", 12, 0, 0), ("rect60", 9, 4, 0), ("open", 13, 0, 0), ("components", 10, 0, 0),
                             ("components", 7, 2, 0)):
        off, b, comp = graph(name)
        g = vga.vga_graph_load(off, b, comp)
        keep.append(g)
        n = g.n_nodes
        jobs.append(dict(graph=g, p=p, d=d, seed=p, conv_mode=conv,
                         mean_depth=torch.empty(n, dtype=torch.float64, device="cuda"),
                         ball=torch.empty(n, dtype=torch.float64, device="cuda")))
        refs.append(oracle.hyperball(off, b, p, d, seed=p, conv_mode=conv, comp_size=comp))
    its = vga.hyperball_run_batch(jobs, use_graph=use_graph)
    for job, it, ref in zip(jobs, its, refs):
        _same(job["mean_depth"].cpu().numpy(), job["ball"].cpu().numpy(), it, ref)
    for g in keep:
        g.free()


def _up(x):
    return (x + 255) // 256 * 256


@pytest.mark.parametrize("bits", [0, 1, 4])
@pytest.mark.parametrize("name,p,d,conv", [("tiny", 7, 0, 0), ("corridor", 8, 0, 0), ("corridor", 10, 0, 1),
                                           ("rect60", 9, 0, 0), ("open", 12, 0, 0), ("components", 10, 0, 0)])
def test_per_neighbour_codes(vga, name, p, d, conv, bits):
    off, b, comp = graph(name)
    ref = oracle.hyperball(off, b, p, d, seed=2, conv_mode=conv, comp_size=comp)
    m = 1 << p
    with vga.vga_graph_load(off, b, comp) as g:
        n = g.n_nodes
        # the mode's own bytes (slices of 1,024 registers), then the window (and some slack), a
        # byte and a list entry a node, and the codes
        s = max(1, m // 1024)
        size = 2 * _up(n * m) + 3 * _up(8 * n) + _up(8 * (m + 1)) + 256 + _up(4 * n) + _up(s * n) + 2 * _up(4 * n)
        if bits:
            size += _up(16 * m) + _up(n) + _up(8 * n) + n * m * bits // 8
        ws = torch.full((size + 256,), 0xA5, dtype=torch.uint8, device="cuda")
        at = -ws.data_ptr() % 256
        md, ball = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
        it = C.c_int()
        tuning = vga._tuning(union_mode=1, slice_bytes=min(m, 1024))
        st = vga.lib().hyperball_run_dev(g.handle, p, d, 2, conv, md.data_ptr(), ball.data_ptr(), C.byref(it),
                                         ws.data_ptr() + at, size, None, tuning)
        assert st == 0, vga.lib().vga_last_error()
        _same(md.cpu().numpy(), ball.cpu().numpy(), it.value, ref)
        assert bool((ws[at + size:] == 0xA5).all())


@pytest.mark.parametrize("name,p", [("tiny", 7), ("corridor", 8), ("rect60", 10), ("components", 9)])
def test_per_neighbour_codes_of_4bit_registers(vga, name, p):
    off, b, comp = graph(name)
    ref = oracle.hyperball(off, b, p, 0, seed=4, reg_bits=4, comp_size=comp)
    with vga.vga_graph_load(off, b, comp) as g:
        n = g.n_nodes
        md, ball = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
        ws = torch.empty(8 << 20, dtype=torch.uint8, device="cuda")
        assert ws.data_ptr() % 256 == 0
        it = vga.hyperball_run_dev(g, p, 0, 4, md, ball, workspace=ws, union_mode=1, register_bits=4)
        _same(md.cpu().numpy(), ball.cpu().numpy(), it, ref)
