"""Kernels at the sizes where they can go wrong: remainders, the edges of
runs, tiles and windows, empty rows and hubs, each against the FP64 oracle.

Tolerances: k-hop lists exact; one step within 1e-4 (FP32 modes) and 1e-12
(FP64) of the largest move; quality figures within 1e-11 relative.
"""
import numpy as np
import pytest

import __graft_entry__
import oracle as O
from paper_1606_02162_gb300 import gila as G
from paper_1606_02162_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {G.GILA_FP32: 1e-4, G.GILA_FP32_COMPENSATED: 1e-4, G.GILA_FP64: 1e-12}


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    import torch
    torch.cuda.set_device(0)


def hub_and_gaps(edges, n, isolated):
    """A hub joined to the first `edges` vertices after it, a path along the
    rest, and `isolated` vertices without edges at the end."""
    a = np.concatenate([np.zeros(edges, dtype=np.int64), np.arange(edges, n - 1)])
    b = np.concatenate([np.arange(1, edges + 1), np.arange(edges + 1, n)])
    return I.csr_from_edges(n + isolated, a, b)


# entries of the adjacency (2 E): below, at and above one run of 256 entries,
# a hub longer than a run, trailing and leading empty rows
@pytest.mark.parametrize("g", [
    hub_and_gaps(5, 20, 0), hub_and_gaps(20, 129, 3), hub_and_gaps(20, 130, 0),
    hub_and_gaps(1000, 1300, 700), I.csr_from_edges(600, [598], [599]), I.csr_from_edges(3, [], []),
], ids=["small", "one_run", "run_and_two", "hub", "last_edge", "no_edges"])
@pytest.mark.parametrize("p", [0, 2, 3])
def test_edge_figures(g, p):
    import torch
    pos = I.uniform_positions(g.n, 11).astype(np.float32).astype(np.float64)
    pos[1] = pos[0]  # an edge (or pair) of length 0
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, 2)
    want = O.metrics(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, d=1.3, p=p)
    for prec, dt in ((G.GILA_FP64, torch.float64), (G.GILA_FP32, torch.float32)):
        with G.Graph.from_inputs(g) as h:
            got = G.gila_layout_metrics(h.handle, G.params(k=2, d=1.3, p=p, precision=prec),
                                        torch.tensor(pos, dtype=dt, device="cuda"))
        for key in ("edge_mean", "edge_std", "edge_cv", "rep_total", "att_total"):
            assert abs(got[key] - want[key]) <= 1e-11 * max(1.0, abs(want[key])), (key, prec)


def mesh_with_tail(rows, cols, extra):
    """A triangulated mesh followed by `extra` vertices without edges."""
    m = I.tri_mesh(rows, cols)
    a, b = m.edge_list()
    return I.csr_from_edges(m.n + extra, a, b)


def unsorted_rows(g):
    """The same graph with every adjacency row in descending order."""
    col = g.col_idx.copy()
    for u in range(g.n):
        col[g.row_ptr[u]:g.row_ptr[u + 1]] = col[g.row_ptr[u]:g.row_ptr[u + 1]][::-1]
    return I.Graph(g.name, g.n, g.row_ptr, col)


# rows of one, two, nine and more steps; a last slice of 1, 31 and 32 rows;
# empty slices; k-hop rows longer than the adjacency's; an unsorted adjacency,
# which the row-per-lane plan refuses
@pytest.mark.parametrize("name,g,k,rows", [
    ("path", I.path(1025), 2, True), ("cycle", I.cycle(2047), 3, True),
    ("grid", I.grid(40, 41), 1, True), ("mesh", I.tri_mesh(61, 67), 3, True),
    ("mesh_k5", I.tri_mesh(100, 90), 5, True), ("tail", mesh_with_tail(50, 64, 100), 2, True),
    ("unsorted", unsorted_rows(I.grid(40, 41)), 2, False), ("short", I.path(33), 2, False),
    ("star", I.star(300), 1, False),
], ids=lambda v: v if isinstance(v, str) else "")
@pytest.mark.parametrize("pq", [(2, 1), (3, 2)], ids=["fr", "p3q2"])
def test_row_per_lane_step(name, g, k, rows, pq):
    import torch
    p, q = pq
    pos = I.uniform_positions(g.n, 21).astype(np.float32).astype(np.float64)
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, k)
    t = 0.3
    _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, t, d=1.2, p=p, q=q)
    for prec in TOL:
        dt = torch.float64 if prec == G.GILA_FP64 else torch.float32
        with G.Graph.from_inputs(g) as h:
            G.gila_graph_tune(h.handle, tiled=1)
            G.gila_profile_enable(h.handle, 2)
            x = torch.tensor(pos, dtype=dt, device="cuda")
            y, disp = torch.empty_like(x), torch.empty_like(x)
            G.gila_layout_step(h.handle, G.params(k=k, d=1.2, p=p, q=q, precision=prec), t, x, y,
                               disp)
            torch.cuda.synchronize()
            kernel = G.gila_profile_read_kernel(h.handle)["name"]
        assert ("row per lane" in kernel) == rows, kernel
        assert torch.equal(y, x + disp)
        assert np.abs(disp.double().cpu().numpy() - want).max() <= TOL[prec] * np.abs(want).max()


# slices of one, a whole and a started 32 rows; graphs below, at and above the
# slices from which a cluster takes one (2048 vertices in FP32, 512 in FP64);
# one beyond FP64's shared memory; empty rows; long rows and an unsorted
# adjacency, which keep the group kernel beside the others
def batch_graphs():
    return [I.csr_from_edges(1, [], []), I.path(31), I.cycle(32), I.grid(3, 11), I.grid(16, 32),
            I.tri_mesh(19, 27), I.random_tree(2016, 3), I.grid(32, 64), I.erdos_renyi(2081, 4.0, 5),
            mesh_with_tail(40, 60, 33), I.grid(100, 100), I.star(300), unsorted_rows(I.grid(9, 9)),
            I.erdos_renyi(5000, 4.0, 9)]


@pytest.mark.parametrize("prec", list(TOL), ids=["fp32", "fp32c", "fp64"])
@pytest.mark.parametrize("pq,sched", [((2, 1), O.SCHED_LINEAR), ((3, 2), O.SCHED_GEOM)],
                         ids=["fr_linear", "p3q2_geometric"])
def test_batch_row_per_lane(prec, pq, sched):
    graphs = batch_graphs()
    p, q = pq
    pos = [I.uniform_positions(g.n, 60 + i).astype(np.float32).astype(np.float64)
           for i, g in enumerate(graphs)]
    off = np.concatenate([[0], np.cumsum([g.n for g in graphs])])
    iters = 4 if prec == G.GILA_FP64 else 1
    prm = G.params(k=2, iters=iters, d=1.2, p=p, q=q, precision=prec,
                   schedule=G.GILA_COOL_LINEAR if sched == O.SCHED_LINEAR else G.GILA_COOL_GEOMETRIC)
    with G.Batch(graphs) as b:
        out = G.gila_layout_batch_run(b.handle, prm, np.concatenate(pos))
        again = G.gila_layout_batch_run(b.handle, prm, np.concatenate(pos))
        G.gila_batch_khop_reset(b.handle)  # the plan is made anew
        rebuilt = G.gila_layout_batch_run(b.handle, prm, np.concatenate(pos))
        G.gila_batch_tune(b.handle, threads=256, ctas_per_sm=8)
        shaped = G.gila_layout_batch_run(b.handle, prm, np.concatenate(pos))
    assert np.array_equal(out, again) and np.array_equal(out, rebuilt) and np.array_equal(out, shaped)
    for i, g in enumerate(graphs):
        krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, 2)
        want = O.run(g.n, g.row_ptr, g.col_idx, krow, kcol, pos[i], iters, d=1.2, p=p, q=q,
                     schedule=sched) - pos[i]
        got = out[off[i]:off[i + 1]] - pos[i]
        scale = np.abs(want).max()
        # FP32: the move is read back as (position + move) - position
        slack = 4 * np.finfo(np.float32).eps * np.abs(pos[i]).max() if prec != G.GILA_FP64 else 0.0
        # FP64: rounding grows over four iterations (1e-9 as for a few iterations)
        tol = 1e-9 if prec == G.GILA_FP64 else TOL[prec]
        assert np.abs(got - want).max() <= tol * max(scale, 1e-300) + slack, (i, g.name, g.n)


# cells (tiles x rows) below, at and above a scan tile of 2048; one tile and
# more tiles than the warps of a block; blocks of a single row (a target above
# the rows) and of the most rows; a hub's tile beside nearly empty ones
@pytest.mark.parametrize("g,k,tune", [
    (I.barabasi_albert(511, 2, 4), 2, dict(tile_vertices=128)),
    (I.barabasi_albert(512, 2, 4), 2, dict(tile_vertices=128)),
    (I.barabasi_albert(4101, 2, 5), 2, dict(tile_vertices=100)),
    (I.barabasi_albert(40, 2, 6), 2, dict(tile_vertices=8, ctas_per_sm=8)),
    (I.random_tree(9001, 7), 1, dict(tile_vertices=9002)),
    (hub_and_gaps(1000, 6000, 50), 2, dict(tile_vertices=512)),
], ids=["511", "512", "42_tiles", "rows_as_blocks", "one_tile", "hub"])
@pytest.mark.parametrize("prec", list(TOL), ids=["fp32", "fp32c", "fp64"])
def test_tile_plan_step(g, k, tune, prec):
    import torch
    pos = I.uniform_positions(g.n, 31).astype(np.float32).astype(np.float64)
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, k)
    _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, 0.4, d=1.1)
    dt = torch.float64 if prec == G.GILA_FP64 else torch.float32
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, tiled=1, **tune)
        G.gila_profile_enable(h.handle, 2)
        x = torch.tensor(pos, dtype=dt, device="cuda")
        y, disp = torch.empty_like(x), torch.empty_like(x)
        G.gila_layout_step(h.handle, G.params(k=k, d=1.1, precision=prec), 0.4, x, y, disp)
        torch.cuda.synchronize()
        assert G.gila_profile_read_kernel(h.handle)["name"] == "blocked_kernel"
    assert np.abs(disp.double().cpu().numpy() - want).max() <= TOL[prec] * np.abs(want).max()


# weighted tiles: one tile and many, a last tile of one to three vertices (the
# weights' tail behind the bulk copy), zero weights; other exponents stay with
# the plain kernel; weights set, cleared and set again on one graph
@pytest.mark.parametrize("n,tv", [(1001, 4), (1002, 100), (1003, 1000), (4097, 512), (900, 900)])
@pytest.mark.parametrize("prec", list(TOL), ids=["fp32", "fp32c", "fp64"])
def test_weighted_tiles(n, tv, prec):
    import torch
    g = I.barabasi_albert(n, 2, 8)
    pos = I.uniform_positions(g.n, 41).astype(np.float32).astype(np.float64)
    w = 1.0 + np.random.default_rng(n).integers(0, 5, g.n)
    w[::7] = 0.0
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, 2)
    dt = torch.float64 if prec == G.GILA_FP64 else torch.float32
    x = torch.tensor(pos, dtype=dt, device="cuda")
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, tiled=1, tile_vertices=tv)
        G.gila_profile_enable(h.handle, 2)
        for wt, p, q, kernel in ((w, 2, 1, "blocked_kernel"), (w, 3, 2, "iteration_kernel"),
                                 (None, 2, 1, "blocked_kernel"), (w[::-1], 2, 1, "blocked_kernel"),
                                 (w, 2, 1, "blocked_kernel")):
            G.gila_graph_set_repulsion_weights(h.handle, wt)
            _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, 0.4, d=1.1, p=p, q=q,
                             wt=None if wt is None else np.ascontiguousarray(wt))
            y, disp = torch.empty_like(x), torch.empty_like(x)
            G.gila_layout_step(h.handle, G.params(k=2, d=1.1, p=p, q=q, precision=prec), 0.4, x, y,
                               disp)
            torch.cuda.synchronize()
            assert G.gila_profile_read_kernel(h.handle)["name"].startswith(kernel)
            got = disp.double().cpu().numpy()
            assert np.abs(got - want).max() <= TOL[prec] * np.abs(want).max()


# balls stored as bitmaps: words below and above a warp's turn of 64, a last
# turn of one word, one to four 16-byte words a thread in the radius-3 unions
# (dense Chung-Lu), and sparse balls of many words (Barabasi-Albert)
@pytest.mark.parametrize("g,k", [
    (I.chung_lu(2049, 2.3, 8.0, 8196, 1), 3), (I.chung_lu(6001, 2.3, 8.0, 24004, 2), 3),
    (I.chung_lu(33000, 2.3, 8.0, 132000, 3), 3), (I.chung_lu(70001, 2.3, 8.0, 280004, 4), 3),
    (I.barabasi_albert_fast(40000, 3, 5), 2), (I.star(3000), 2),
], ids=["cl2049", "cl6001", "cl33000", "cl70001", "ba40000", "star"])
def test_khop_rows_from_bitmaps(g, k):
    deg = np.diff(g.row_ptr)
    sel = np.unique(np.concatenate([np.argsort(-deg)[:20], np.linspace(0, g.n - 1, 150).astype(int)]))
    want_counts, want = O.khop_rows(g.n, g.row_ptr, g.col_idx, k, sel)
    with G.Graph.from_inputs(g) as h:
        G.gila_build_khop(h.handle, k)
        counts, cols = G.gila_khop_export_rows(h.handle, sel)
    assert np.array_equal(counts, want_counts) and np.array_equal(cols, want)


@pytest.mark.parametrize("name,g,tune", [
    ("plain", I.grid(20, 21), {}), ("tiles", I.barabasi_albert(3000, 2, 3), dict(tiled=1, tile_vertices=500)),
    ("rows", I.tri_mesh(40, 50), dict(tiled=1)),
], ids=["plain", "tiles", "rows"])
def test_stream_capture(name, g, tune):
    """Iterations captured into a CUDA graph replay to the same placement."""
    import torch
    x0 = torch.tensor(I.uniform_positions(g.n, 51), dtype=torch.float32, device="cuda")
    prm = G.params(k=2, iters=6, t0=0.3)
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, **tune) if tune else None
        x = x0.clone()
        G.gila_layout_run_device(h.handle, prm, x)  # lists and plan
        torch.cuda.synchronize()
        want = x.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            G.gila_graph_set_stream(h.handle)
            G.gila_layout_run_device(h.handle, prm, x)
        for _ in range(2):
            x.copy_(x0)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(x, want)
        G.gila_graph_set_stream(h.handle)
