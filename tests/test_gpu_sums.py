"""The sums of the force kernels: orders of additions that results rely on,
and the accuracy each mode promises."""
import os

import numpy as np
import pytest

import __graft_entry__
import oracle as O
from paper_1606_02162_gb300 import gila as G
from paper_1606_02162_gb300 import inputs as I

pytestmark = pytest.mark.gpu

GOLD = os.path.join(os.path.dirname(__file__), "golden")


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    import torch
    torch.cuda.set_device(0)


def test_fp64_run_keeps_its_order_of_additions():
    """A hundred FP64 iterations in which two vertices pass close by: short
    rows added in another order (an entry per lane) end 3e-5 away, by a CPU
    restatement of both orders; the recorded order repeats exactly."""
    import torch
    want = np.loadtxt(os.path.join(GOLD, "grid_fp64_run.txt"))
    g = I.grid(12, 12)
    x = torch.tensor(I.uniform_positions(g.n, 5), dtype=torch.float64, device="cuda")
    with G.Graph.from_inputs(g) as h:
        G.gila_layout_run_device(h.handle, G.params(k=2, iters=100, t0=0.02, precision=G.GILA_FP64), x)
    assert np.abs(x.cpu().numpy() - want).max() <= 1e-12 * np.abs(want).max()


# FP64 rows that go through the stage: empty, below and above a vector, heads
# and tails of every length, one and more chunks of 32 entries, the last with
# and without a tail; with weights and other exponents
@pytest.mark.parametrize("pq,weighted", [((2, 1), False), ((2, 1), True), ((3, 2), False)],
                         ids=["fr", "weighted", "p3q2"])
def test_staged_rows_fp64(pq, weighted):
    import torch
    p, q = pq
    rng = np.random.default_rng(3)
    sizes = list(range(1, 75)) + [96, 97, 98, 99, 127, 128, 129, 200]
    off = np.concatenate([[0], np.cumsum(sizes)])
    # cliques: rows of every length and, in turn, every alignment
    a = np.concatenate([o + np.triu_indices(s, 1)[0] for o, s in zip(off, sizes)])
    b = np.concatenate([o + np.triu_indices(s, 1)[1] for o, s in zip(off, sizes)])
    g = I.csr_from_edges(int(off[-1]) + 5, a, b)
    pos = I.uniform_positions(g.n, 9)
    w = 1.0 + rng.integers(0, 4, g.n) if weighted else None
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, 1)
    _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, 0.4, d=1.1, p=p, q=q, wt=w)
    x = torch.tensor(pos, device="cuda")
    y, disp = torch.empty_like(x), torch.empty_like(x)
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, tiled=0, small_max=256)  # every row by a group of eight
        if weighted:
            G.gila_graph_set_repulsion_weights(h.handle, w)
        G.gila_layout_step(h.handle, G.params(k=1, d=1.1, p=p, q=q, precision=G.GILA_FP64), 0.4, x, y,
                           disp)
    assert np.abs(disp.cpu().numpy() - want).max() <= 1e-12 * np.abs(want).max()


def wheel(near, ones, far):
    """Vertex 0 at the origin; vertex 1, its only neighbour, joins it to all
    the others, so that its k = 2 row is every other vertex. Along x, repulsion
    1 / distance: `near` from vertex 1, 1 from each of `ones` vertices, and,
    with `far`, -near from the last. All terms are powers of two."""
    n = 2 + ones + (1 if far else 0)
    g = I.csr_from_edges(n, [0] + [1] * (n - 2), [1] + list(range(2, n)))
    pos = np.zeros((n, 2))
    pos[1, 0] = -1.0 / near
    pos[2:2 + ones, 0] = -1.0
    if far:
        pos[n - 1, 0] = 1.0 / near
    return g, pos


# 2^24 + 1 + ... + 1 - 2^24 in the compensated mode: every one is below the
# last place of the plain sum, so that terms added plainly before the two-sum
# lose them; with a two-sum per term the result is exact but for the
# attraction (2^-48)
@pytest.mark.parametrize("ones", [5, 14, 31, 60])
def test_compensated_batch_sums_every_term(ones):
    g, pos = wheel(2.0 ** 24, ones, True)
    with G.Batch([g]) as b:
        prm = G.params(k=2, iters=1, t0=1e9, precision=G.GILA_FP32_COMPENSATED)
        out = G.gila_layout_batch_run(b.handle, prm, pos)
    assert abs(out[0, 0] - ones) <= 1e-6 * ones


# 2^24 + 1 + ... + 1 in FP32: only ones added to the large term are lost. The
# lanes of the group form (sixteen at rows of 25 to 64, eight at 9 to 24) add at
# most four entries each, so that three ones are lost, and each of at most
# seven joins of partial sums rounds a sum of at most 2^25 (unit 2) by 1
@pytest.mark.parametrize("ones", [11, 22, 40, 61])
def test_fp32_batch_keeps_partial_sums(ones):
    g, pos = wheel(2.0 ** 24, ones, False)
    with G.Batch([g]) as b:
        prm = G.params(k=2, iters=1, t0=1e9, precision=G.GILA_FP32)
        out = G.gila_layout_batch_run(b.handle, prm, pos)
    assert abs(out[0, 0] - (2.0 ** 24 + ones)) <= 3 + 7


# a whole batch drawn at a tiny scale: d and the distances scaled by 2^-e. FP32
# squares stay normal numbers down to distances of 2^-63 and FP64 ones to
# 2^-511. Scaled by a power of two a layout is the same layout, so that the
# move is held to the FP32 and FP64 bounds of a move at scale 1 (FP32: the
# approximate reciprocal and root keep their relative errors)
@pytest.mark.parametrize("prec,e", [("FP32", 30), ("FP32", 45), ("FP32", 55), ("FP32_COMPENSATED", 55),
                                    ("FP64", 300), ("FP64", 490)])
def test_batch_at_small_distances(prec, e):
    prec = getattr(G, "GILA_" + prec)
    graphs = [I.grid(9, 13), I.tri_mesh(12, 12), I.random_tree(200, 3), I.erdos_renyi(700, 4.0, 5)]
    pos = [I.uniform_positions(g.n, 80 + i).astype(np.float32).astype(np.float64)
           for i, g in enumerate(graphs)]
    s = 2.0 ** -e
    prm = G.params(k=2, iters=1, d=s, t0=s, precision=prec)
    with G.Batch(graphs) as b:
        out = G.gila_layout_batch_run(b.handle, prm, s * np.concatenate(pos)) / s
    at = 0
    for g, x in zip(graphs, pos):
        krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, 2)
        _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, x, 1.0)
        got = out[at:at + g.n] - x
        at += g.n
        slack = 4 * np.finfo(np.float32).eps * np.abs(x).max() if prec != G.GILA_FP64 else 0.0
        tol = 1e-12 if prec == G.GILA_FP64 else 1e-4
        assert np.abs(got - want).max() <= tol * np.abs(want).max() + slack, g.name


# the same for the single-graph kernels that keep to it: every FP64 form, and
# the FP32 row-per-lane form where all of a row's ids are its neighbours
@pytest.mark.parametrize("prec,e,k,tune,kernel", [
    ("FP64", 490, 2, dict(tiled=1), "row per lane"), ("FP64", 490, 2, dict(tiled=1, tile_vertices=100), "blocked"),
    ("FP64", 490, 2, dict(tiled=0), "iteration"), ("FP32", 55, 1, dict(tiled=1), "row per lane"),
    ("FP32", 55, 2, dict(tiled=0), "iteration"), ("FP32_COMPENSATED", 55, 1, dict(tiled=1), "row per lane"),
])
def test_step_at_small_distances(prec, e, k, tune, kernel):
    import torch
    prec = getattr(G, "GILA_" + prec)
    g = I.grid(40, 41)
    pos = I.uniform_positions(g.n, 90).astype(np.float32).astype(np.float64)
    s = 2.0 ** -e
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, k)
    _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, 1.0)
    x = torch.tensor(s * pos, dtype=torch.float64 if prec == G.GILA_FP64 else torch.float32, device="cuda")
    y, disp = torch.empty_like(x), torch.empty_like(x)
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, **tune)
        G.gila_profile_enable(h.handle, 2)
        G.gila_layout_step(h.handle, G.params(k=k, d=s, precision=prec), s, x, y, disp)
        torch.cuda.synchronize()
        assert kernel in G.gila_profile_read_kernel(h.handle)["name"]
    tol = 1e-12 if prec == G.GILA_FP64 else 1e-4
    assert np.abs(disp.double().cpu().numpy() / s - want).max() <= tol * np.abs(want).max()


# large weights: vertices at one place exert nothing on each other whatever
# they weigh, and with d and the distances scaled by 2^-e the layout is the
# same layout
@pytest.mark.parametrize("prec,big,e", [("FP32", 1e9, 0), ("FP32_COMPENSATED", 1e9, 0), ("FP64", 1e8, 0),
                                        ("FP32", 1e9, 50), ("FP64", 1e9, 480)])
@pytest.mark.parametrize("tiled", [0, 1])
def test_large_weights(prec, big, e, tiled):
    import torch
    prec = getattr(G, "GILA_" + prec)
    g = I.barabasi_albert(700, 2, 8)
    pos = I.uniform_positions(g.n, 95).astype(np.float32).astype(np.float64)
    pos[1::9] = pos[::9][:pos[1::9].shape[0]]  # pairs at one place
    w = np.where(np.arange(g.n) % 3 == 0, big, 1.0)
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, 2)
    _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, 1.0, wt=w)
    s = 2.0 ** -e
    x = torch.tensor(s * pos, dtype=torch.float64 if prec == G.GILA_FP64 else torch.float32, device="cuda")
    y, disp = torch.empty_like(x), torch.empty_like(x)
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, **(dict(tiled=1, tile_vertices=100) if tiled else dict(tiled=0)))
        G.gila_graph_set_repulsion_weights(h.handle, w)
        G.gila_layout_step(h.handle, G.params(k=2, d=s, precision=prec), s, x, y, disp)
    got = disp.double().cpu().numpy() / s
    tol = 1e-12 if prec == G.GILA_FP64 else 1e-4
    assert np.abs(got - want).max() <= tol * np.abs(want).max()


# the compensated wheel on weighted tiles (weights 1, all of a row in one
# tile): a two-sum per term, as in the plain kernel
@pytest.mark.parametrize("ones", [5, 14, 31, 60, 200])
@pytest.mark.parametrize("tiled", [0, 1])
def test_compensated_weighted_tiles_sum_every_term(ones, tiled):
    import torch
    g, pos = wheel(2.0 ** 24, ones, True)
    x = torch.tensor(pos, dtype=torch.float32, device="cuda")
    y, disp = torch.empty_like(x), torch.empty_like(x)
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, tiled=tiled)
        G.gila_graph_set_repulsion_weights(h.handle, np.ones(g.n))
        G.gila_layout_step(h.handle, G.params(k=2, precision=G.GILA_FP32_COMPENSATED), 1e9, x, y, disp)
    assert abs(float(disp[0, 0]) - ones) <= 1e-6 * ones


# vertices without edges feel no force wherever they are: at infinity too, in
# a slice beside longer rows
@pytest.mark.parametrize("prec", [G.GILA_FP32, G.GILA_FP32_COMPENSATED, G.GILA_FP64],
                         ids=["fp32", "fp32c", "fp64"])
def test_isolated_vertices_at_infinity(prec):
    import torch
    g = I.csr_from_edges(70, np.arange(40), np.arange(1, 41))  # a path, 29 isolated vertices
    pos = I.uniform_positions(g.n, 13)
    pos[50], pos[51], pos[69] = (np.inf, 0.0), (3e38, -np.inf), (-3e38, 3e38)
    if prec == G.GILA_FP64:
        pos[69] = (1e300, -1e300)
    dt = torch.float64 if prec == G.GILA_FP64 else torch.float32
    x = torch.tensor(pos, dtype=dt, device="cuda")
    with G.Batch([g]) as b:
        y = x.clone()
        G.gila_layout_batch_device(b.handle, G.params(k=2, iters=3, t0=0.5, precision=prec), y)
    for tiled in (0, 1):
        with G.Graph.from_inputs(g) as h:
            G.gila_graph_tune(h.handle, tiled=tiled)
            z = x.clone()
            G.gila_layout_run_device(h.handle, G.params(k=2, iters=3, t0=0.5, precision=prec), z)
        assert torch.equal(z[41:], x[41:]) and bool(torch.isfinite(z[:41]).all())
    assert torch.equal(y[41:], x[41:]) and bool(torch.isfinite(y[:41]).all())


def test_fp64_batch_far_from_the_origin():
    """Coordinates of 2^533, whose squares overflow, distances of 2^500, whose
    squares do not: the layout at the origin, to the coordinates' last place
    (2^-19 of a unit), which padding far from all vertices turned into NaN."""
    g = I.erdos_renyi(300, 4.0, 6)
    pos = np.round(I.uniform_positions(g.n, 14) * 2.0 ** 18) / 2.0 ** 18
    s, o = 2.0 ** 500, 2.0 ** 533
    with G.Batch([g]) as b:
        near = G.gila_layout_batch_run(b.handle, G.params(k=2, iters=1, t0=1.0, precision=G.GILA_FP64), pos)
        far = G.gila_layout_batch_run(b.handle, G.params(k=2, iters=1, d=s, t0=s, precision=G.GILA_FP64),
                                      o + s * pos)
    assert np.abs((far - o) / s - near).max() <= 2.0 ** -18


# a coordinate that is NaN says nothing along the other one: the pattern of
# NaN in a batch's placement after an iteration is the group kernel's, and the
# finite coordinates agree
@pytest.mark.parametrize("prec", [G.GILA_FP32, G.GILA_FP32_COMPENSATED, G.GILA_FP64],
                         ids=["fp32", "fp32c", "fp64"])
def test_nan_coordinate_in_a_batch(prec):
    g = I.grid(12, 13)
    pos = I.uniform_positions(g.n, 17)
    pos[60, 1] = np.nan
    pos[100, 0] = np.nan
    prm = G.params(k=2, iters=1, t0=1e9, precision=prec)
    out = []
    for tune in ({}, dict(group4_max=8)):
        with G.Batch([g]) as b:
            G.gila_batch_tune(b.handle, **tune)
            out.append(G.gila_layout_batch_run(b.handle, prm, pos))
    rows, groups = out
    assert np.array_equal(np.isnan(rows), np.isnan(groups)) and np.isnan(rows).sum() < 40
    fine = ~np.isnan(groups)
    tol = 1e-12 if prec == G.GILA_FP64 else 1e-5
    assert np.abs(rows - groups)[fine].max() <= tol * np.abs(groups[fine]).max()
