"""The work that users have this framework do, as cases that can be timed.

A case is one call, or one short sequence of calls, of the public entry points
on a seeded obstacle grid (``workloads``): analyses of a resident graph from
the smallest grid to the city, the whole way from a grid or a host CSR to mean
depths, a batch, a burst of served requests, and the entry point that allocates
nothing.  ``listed`` names the cases, ``draw`` gives others of the same ranges,
``prepare`` makes what a program holds before the call, ``run`` is one pass,
``work`` the bytes it cannot do without, and ``exact`` the same outputs in
plain torch: HyperBall by boolean matrix products over the decoded CSR, with
the estimator in float64.
"""
import math

import numpy as np
import torch

import paper_2604_08374_gb300 as vga
import workloads

# Mean degree of the two grid families by free cells (three sites each): the
# edges of a case are counted from it, one byte an edge in the compressed CSR.
_DEGREE = {
    "rects": ((800, 2_000, 5_000, 12_000, 30_000, 42_680, 80_000, 130_000, 236_693),
              (360, 1_170, 2_220, 4_950, 7_980, 9_310, 12_400, 13_800, 16_900)),
    "blocks": ((950, 2_282, 5_200, 12_000, 30_000, 43_500, 80_000, 130_000, 236_693),
               (900, 2_000, 2_770, 5_000, 8_700, 10_600, 14_600, 16_300, 21_000)),
}
_MAX_CELLS = 236_693  # the city workload
_POOL_MAX = 60_000    # largest graph of the served pool


def listed():
    return [
        # the smallest call: one analysis of a 32 x 32 plan (a room, a floor); launches and latency
        dict(name="tiny_d3", op="run", kind="rects", cells=903, p=10, d=3, bits=8, order="raster", site=1),
        # a small site at high precision until nothing changes
        dict(name="small_p12_full", op="run", kind="rects", cells=5_003, p=12, d=0, bits=8, order="raster", site=2),
        # an ordinary district (the paper's 42,705-cell size), depth limit 3
        dict(name="medium_d3", op="run", kind="rects", cells=42_700, p=10, d=3, bits=8, order="raster", site=3),
        # the paper's packed 4-bit registers and Hilbert numbering, unlimited depth, odd size
        dict(name="medium_4bit_full", op="run", kind="blocks", cells=90_001, p=11, d=0, bits=4, order="hilbert", site=4),
        # the headline: a city of 236k cells, p = 10, d = 3
        dict(name="city_d3", op="run", kind="blocks", cells=236_693, p=10, d=3, bits=8, order="raster", site=5),
        # the largest analysis: the city at p = 12, unlimited depth
        dict(name="city_p12_full", op="run", kind="blocks", cells=236_693, p=12, d=0, bits=8, order="raster", site=6),
        # a grid to its compressed visibility graph in host memory, to be kept in a file
        dict(name="build_csr", op="build", kind="rects", cells=9_973, order="raster", site=7),
        # a grid all the way to mean depths and the closed-form metrics, once: city size
        dict(name="analyse_city", op="analyse", kind="blocks", cells=236_693, p=10, d=3, order="raster", site=8),
        # a compressed graph from pinned host memory to host results, once
        dict(name="load_run", op="load", kind="blocks", cells=100_003, p=10, d=3, site=9),
        # a study of many sites: uneven graphs, precisions and depths in one call
        dict(name="batch_64", op="batch", jobs=64, lo=1_000, hi=30_000, site=10),
        # a burst of requests on a resident pool of graphs
        dict(name="serve_burst", op="serve", pool=12, requests=40, lo=1_000, hi=_POOL_MAX, site=11),
        # a caller that may not allocate device memory (per-neighbour union, the paper's stop rule)
        dict(name="noalloc_20k", op="noalloc", kind="rects", cells=20_011, p=10, d=5, site=12),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _draw(rng)
    case["site"] = rng.randint(100, 999)
    return case


def _draw(rng):
    op = rng.choices(("run", "build", "analyse", "load", "batch", "serve", "noalloc"), (6, 1, 2, 2, 1, 1, 1))[0]
    kind = rng.choice(("rects", "blocks"))
    if op == "run":
        return dict(op=op, kind=kind, cells=_log_uniform(rng, 800, _MAX_CELLS), p=rng.choice((8, 9, 10, 11, 12)),
                    d=rng.choice((2, 3, 5, 10, 0)), bits=rng.choice((8, 8, 8, 4)),
                    order=rng.choice(("raster", "raster", "hilbert")))
    if op == "build":
        return dict(op=op, kind=kind, cells=_log_uniform(rng, 800, 30_000), order=rng.choice(("raster", "hilbert")))
    if op == "analyse":
        return dict(op=op, kind=kind, cells=_log_uniform(rng, 800, _MAX_CELLS), p=rng.choice((8, 9, 10)),
                    d=rng.choice((3, 5)), order=rng.choice(("raster", "hilbert")))
    if op == "load":
        return dict(op=op, kind=kind, cells=_log_uniform(rng, 800, 100_003), p=rng.choice((8, 10, 11)),
                    d=rng.choice((3, 5, 0)))
    if op == "batch":
        return dict(op=op, jobs=rng.randint(8, 64), lo=rng.randint(900, 2_000), hi=rng.randint(8_000, 30_000))
    if op == "serve":
        return dict(op=op, pool=rng.randint(4, 12), requests=rng.randint(8, 40), lo=rng.randint(900, 2_000),
                    hi=rng.randint(10_000, _POOL_MAX))
    return dict(op=op, kind=kind, cells=_log_uniform(rng, 800, 30_000), p=rng.choice((8, 9, 10)),
                d=rng.choice((3, 5, 0)))


def _turned(grid, seed):
    """One of the grid's eight rotations and reflections."""
    grid = np.rot90(grid, seed % 4)
    return np.ascontiguousarray(grid[:, ::-1] if seed % 8 >= 4 else grid)


def _grid(case, seed):
    """The case's site, turned by the seed: random rectangles (the medium
    workload's recipe) or urban blocks (the city's, scaled) with about `cells`
    free cells.  Its cells, lists and numbering differ with the seed, the
    number of nodes and edges does not."""
    cells, site = case["cells"], case["site"]
    if case["kind"] == "rects":
        return _turned(workloads.grid_for_free_cells(cells, seed=site), seed)
    side = int(math.ceil(math.sqrt(cells / 0.8755)))
    area = side * side / (workloads.CITY["W"] * workloads.CITY["H"])
    return _turned(workloads.city(seed=site, W=side, H=side, block_free=int(workloads.CITY["block_free"] * area),
                                  n_small=int(round(workloads.CITY["n_small"] * area))), seed)


def _out(n):
    return torch.empty(max(n, 1), dtype=torch.float64, device="cuda")


def _sites(case, seed):
    """Batch: (grid, p, d) of every job."""
    rng = np.random.default_rng(case["site"])
    sizes = np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), case["jobs"])).astype(int)
    return [(_turned(workloads.grid_for_free_cells(int(n), seed=case["site"] * 1000 + i), seed + i), int(rng.choice([8, 10, 12])),
             int(rng.choice([3, 0]))) for i, n in enumerate(sizes)]


def _requests(case, seed):
    """Served burst: the pool's grids and (graph, p, d) of every request."""
    rng = np.random.default_rng(case["site"])
    sizes = np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), case["pool"])).astype(int)
    grids = [_turned(workloads.grid_for_free_cells(int(n), seed=case["site"] * 1000 + i), seed + i) for i, n in enumerate(sizes)]
    reqs = [(int(rng.integers(case["pool"])), int(rng.choice([8, 10, 12])), int(rng.choice([3, 5, 0])))
            for _ in range(case["requests"])]
    return grids, reqs


def prepare(case, seed):
    op, s = case["op"], {"op": case["op"], "case": case, "seed": seed}
    if op == "batch":
        sites = _sites(case, seed)
        graphs = [vga.vga_visibility_build(grid) for grid, _, _ in sites]
        total = sum(g.n_nodes for g in graphs)
        s["md"], s["ball"], s["jobs"], at = _out(total), _out(total), [], 0
        for k, (g, (_, p, d)) in enumerate(zip(graphs, sites)):
            s["jobs"].append(dict(graph=g, p=p, d=d, seed=seed + k, mean_depth=s["md"][at:at + g.n_nodes],
                                  ball=s["ball"][at:at + g.n_nodes]))
            at += g.n_nodes
        s["ws"] = torch.empty(vga.hyperball_batch_workspace_bytes(s["jobs"]), dtype=torch.uint8, device="cuda")
        return s
    if op == "serve":
        grids, s["reqs"] = _requests(case, seed)
        s["graphs"] = [vga.vga_visibility_build(grid) for grid in grids]
        s["server"] = vga.Server(hbm_budget_bytes=16 << 30)
        return s
    grid = _grid(case, seed)
    if op in ("build", "analyse"):
        s["grid"] = grid
        if op == "build":  # host memory for the graph; an edge takes 1 to 2 bytes at these sizes
            n = vga.vga_visibility_count(grid)
            s.update(offsets=np.zeros(n + 1, np.int64), degree=np.zeros(n, np.int32),
                     csr=np.zeros(65_536 + 2 * int(_edges(case["kind"], n)), np.uint8))
        return s
    if op == "load":
        g, cells = vga.vga_visibility_build(grid, return_cells=True)
        offsets, csr, _ = g.copy_csr()
        g.free()
        pinned = torch.empty(len(csr), dtype=torch.uint8, pin_memory=True)
        pinned.numpy()[:] = csr
        s.update(offsets=offsets, csr=pinned.numpy(), keep=pinned, cells=cells, shape=grid.shape)
        return s
    g = vga.vga_visibility_build(grid, order=case.get("order", "raster"))
    s.update(g=g, md=_out(g.n_nodes), ball=_out(g.n_nodes))
    if op == "run":
        s["ws"] = torch.empty(vga.hyperball_workspace_bytes(g, case["p"]), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    op, c = s["op"], s["case"]
    if op == "run":
        it = vga.hyperball_run_dev(s["g"], c["p"], c["d"], s["seed"], s["md"], s["ball"], workspace=s["ws"],
                                   register_bits=0 if c["bits"] == 8 else c["bits"])
        return {"mean_depth": s["md"], "ball": s["ball"], "passes": it}
    if op == "noalloc":
        it = vga.hyperball_run_noalloc(s["g"], c["p"], c["d"], s["seed"], s["md"], s["ball"], conv_mode=1)
        return {"mean_depth": s["md"], "ball": s["ball"], "passes": it}
    if op == "build":
        with vga.vga_visibility_build(s["grid"], order=c["order"]) as g:
            assert g.n_bytes <= s["csr"].size
            status = vga.lib().vga_graph_copy_csr(g.handle, s["offsets"].ctypes.data, s["csr"].ctypes.data,
                                                  s["degree"].ctypes.data)
            assert status == 0, vga.lib().vga_last_error()
        return {"offsets": s["offsets"], "csr": s["csr"], "degree": s["degree"]}
    if op == "analyse":
        with vga.vga_visibility_build(s["grid"], order=c["order"]) as g:
            md, ball = _out(g.n_nodes), _out(g.n_nodes)
            it = vga.hyperball_run_dev(g, c["p"], c["d"], s["seed"], md, ball)
            metrics = vga.vga_metrics(g, md)
            return {"mean_depth": md, "ball": ball, "metrics": metrics, "passes": it, "edges": g.n_edges}
    if op == "load":
        with vga.vga_graph_load(s["offsets"], s["csr"]) as g:
            g.set_cells(s["shape"][1], s["shape"][0], s["cells"])
            md, ball, it = vga.hyperball_run(g, c["p"], c["d"], s["seed"])
        return {"mean_depth": md, "ball": ball, "passes": it}
    if op == "batch":
        its = vga.hyperball_run_batch(s["jobs"], workspace=s["ws"])
        return {"mean_depth": s["md"], "ball": s["ball"], "passes": np.array(its)}
    rids = [s["server"].submit(s["graphs"][k], p, d, s["seed"] + i) for i, (k, p, d) in enumerate(s["reqs"])]
    done = [s["server"].wait(r) for r in rids]
    return {"mean_depth": np.concatenate([r["mean_depth"] for r in done]),
            "ball": np.concatenate([r["ball"] for r in done]), "passes": np.array([r["iterations"] for r in done])}


# ---------------------------------------------------------------------------
# Bytes a pass cannot do without
# ---------------------------------------------------------------------------

def _edges(kind, cells):
    x, y = _DEGREE[kind]
    return cells * math.exp(np.interp(math.log(cells), np.log(x), np.log(y)))


def work(case):
    """The compressed CSR (one byte an edge, 8 an offset) read or written once,
    the grid read and the outputs written once."""
    op = case["op"]
    if op in ("batch", "serve"):
        lo, hi = math.log(case["lo"]), math.log(case["hi"])
        n = case["jobs"] if op == "batch" else case["requests"]
        sizes = [math.exp(lo + (hi - lo) * (k + 0.5) / n) for k in range(n)]
        return {"bytes": sum(_edges("rects", c) + 8 * c + 16 * c for c in sizes), "flops": 0.0}
    cells = case["cells"]
    csr = _edges(case["kind"], cells) + 8 * cells
    if op == "build":
        return {"bytes": 1.15 * cells + 2 * csr + 4 * cells, "flops": 0.0}
    if op == "analyse":
        return {"bytes": 1.15 * cells + csr + 48 * cells, "flops": 0.0}
    return {"bytes": csr + 16 * cells, "flops": 0.0}


# ---------------------------------------------------------------------------
# The same outputs in plain torch
# ---------------------------------------------------------------------------

_EXACT_MACS = 6e15  # multiply-adds of boolean products in bfloat16: about 10 s on the device


def _decode_rows(offsets, csr, r0, r1, n):
    """Rows r0 .. r1 of the 0/1 adjacency matrix with ones on the diagonal."""
    o = torch.from_numpy(offsets[r0:r1 + 1].astype(np.int64)).cuda()
    b = torch.from_numpy(csr[int(offsets[r0]):int(offsets[r1])]).cuda()
    a = torch.zeros(r1 - r0, n, dtype=torch.bfloat16, device="cuda")
    a[torch.arange(r1 - r0, device="cuda"), torch.arange(r0, r1, device="cuda")] = 1
    if b.numel():
        ends = torch.nonzero(b < 128).flatten()                   # last byte of every varint
        starts = torch.cat([ends.new_zeros(1), ends[:-1] + 1])
        val = torch.zeros_like(ends)
        for k in range(5):
            at = starts + k
            more = at <= ends
            val += torch.where(more, (b[at.clamp(max=b.numel() - 1)].long() & 127) << (7 * k), 0)
        row = torch.searchsorted(o[1:] - o[0], starts, right=True)
        run = torch.cumsum(val, 0)
        first = torch.searchsorted(starts, o[:-1] - o[0])         # first varint of every row
        before = torch.cat([run.new_zeros(1), run])[first]        # ids restart in every row
        a[row, run - before[row]] = 1
    return a


def _initial(n, p, seed, bits):
    """Alg. 1's initial counters: SplitMix64 of id ^ seed, top p bits, leading zeros of the rest."""
    u = np.uint64
    with np.errstate(over="ignore"):
        x = (np.arange(n, dtype=np.uint64) ^ u(seed)) + u(0x9E3779B97F4A7C15)
        x = (x ^ (x >> u(30))) * u(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> u(27))) * u(0x94D049BB133111EB)
        x ^= x >> u(31)
        j, w = (x >> u(64 - p)).astype(np.int64), x << u(p)
    rho = np.full(n, 65 - p, np.int64)
    left = np.ones(n, bool)
    for k in range(64 - p):
        hit = left & ((w >> u(63 - k)) & u(1)).astype(bool)
        rho[hit] = k + 1
        left &= ~hit
    regs = torch.zeros(n, 1 << p, dtype=torch.uint8, device="cuda")
    regs[torch.arange(n, device="cuda"), torch.from_numpy(j).cuda()] = \
        torch.from_numpy(np.minimum(rho, 15 if bits == 4 else 99).astype(np.uint8)).cuda()
    return regs


def _estimate(regs, p):
    m = 1 << p
    alpha = {4: 0.673, 5: 0.697, 6: 0.709}.get(p, 0.7213 / (1 + 1.079 / m))
    power = torch.pow(torch.tensor(2.0, dtype=torch.float64, device="cuda"),
                      -torch.arange(256, dtype=torch.float64, device="cuda"))
    z = torch.cat([power[part.int()].sum(1) for part in regs.split(16384)])
    e = alpha * m * m / z
    v = torch.cat([(part == 0).sum(1) for part in regs.split(16384)]).double()
    return torch.where((e <= 2.5 * m) & (v > 0), m * torch.log(m / v.clamp(min=1)), e)


def _hyperball(offsets, csr, p, d, seed, bits=8, conv_mode=0):
    n = len(offsets) - 1
    regs = _initial(n, p, seed, bits)
    c = _estimate(regs, p)
    total, t = torch.zeros_like(c), 0
    chunk = max(1, min(n, int(8e9) // (2 * n)))
    whole = _decode_rows(offsets, csr, 0, n, n) if chunk >= n else None
    while True:
        t += 1
        top, nxt = int(regs.max()), torch.empty_like(regs)
        for r0 in range(0, n, chunk):
            r1 = min(n, r0 + chunk)
            a = whole if whole is not None else _decode_rows(offsets, csr, r0, r1, n)
            acc = torch.zeros(r1 - r0, 1 << p, dtype=torch.uint8, device="cuda")
            for level in range(1, top + 1):
                acc += (a @ (regs >= level).to(torch.bfloat16)) > 0
            nxt[r0:r1] = acc
        new = _estimate(nxt, p)
        total += t * (new - c)
        stop = bool((new - c).max() <= 0.5) if conv_mode else bool((nxt == regs).all())
        regs, c = nxt, new
        if stop or (d > 0 and t >= d):
            break
    md = total / (n - 1) if n > 1 else torch.full_like(total, float("nan"))
    return md, c, t


def _csr_of(grid, order="raster"):
    with vga.vga_visibility_build(grid, order=order) as g:
        offsets, csr, degree = g.copy_csr()
    return offsets, csr, degree


def _macs(n, p, d):
    return float(n) * n * (1 << p) * 18 * (d if 0 < d < 5 else 5)


def _metrics(md, degree, n):
    k = float(n)
    if k > 2:
        ra = 2 * (md - 1) / (k - 2)
        dk = 2 * (k * (math.log2((k + 2) / 3) - 1) + 1) / ((k - 1) * (k - 2))
        hh, pv = dk / ra, (1 - ra).clamp(min=0)
    else:
        hh = pv = torch.full_like(md, float("nan"))
    return torch.stack([hh, torch.log2((md + 2) / 3), pv, md * torch.from_numpy(degree.astype(np.float64)).cuda()], 1)


def exact(case, seed):
    op = case["op"]
    if op == "build":
        return None
    if op in ("batch", "serve"):
        if op == "batch":
            todo = [(grid, p, d) for grid, p, d in _sites(case, seed)]
        else:
            grids, reqs = _requests(case, seed)
            todo = [(grids[k], p, d) for k, p, d in reqs]
        if sum(_macs(int((g == 0).sum()), p, d) for g, p, d in todo) > _EXACT_MACS:
            return None
        got = [_hyperball(*_csr_of(g)[:2], p, d, seed + k) for k, (g, p, d) in enumerate(todo)]
        return {"mean_depth": torch.cat([x[0] for x in got]), "ball": torch.cat([x[1] for x in got]),
                "passes": np.array([x[2] for x in got])}
    if _macs(case["cells"], case["p"], case["d"]) > _EXACT_MACS:
        return None
    offsets, csr, degree = _csr_of(_grid(case, seed), case.get("order", "raster"))
    md, ball, it = _hyperball(offsets, csr, case["p"], case["d"], seed, case.get("bits", 8),
                              1 if op == "noalloc" else 0)
    out = {"mean_depth": md, "ball": ball, "passes": it}
    if op == "analyse":
        out.update(metrics=_metrics(md, degree, len(offsets) - 1), edges=int(degree.astype(np.int64).sum()))
    return out
