"""Batched layouts on clusters of CTAs: graphs of which some CTAs of a cluster
have no slice, against the oracle.

FP64 layouts of a few iterations within 1e-9 of the extent, one FP32 iteration
within 1e-4 of the largest move (as for every batch)."""
import numpy as np
import pytest

import __graft_entry__
import oracle as O
from paper_1606_02162_gb300 import gila as G
from paper_1606_02162_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    import torch
    torch.cuda.set_device(0)


def bipartite(a, b):
    """Complete bipartite: 32 long rows in the first slice, short ones behind."""
    return I.csr_from_edges(a + b, np.repeat(np.arange(a), b), np.tile(np.arange(a, a + b), a))


# few graphs, so that the largest ask for clusters of 8; four slices (97, 128
# vertices in FP64) leave four of the eight CTAs without one, five and eight
# slices three and none; the first slice of a complete bipartite graph
# outweighs several shares (32 rows of 500 ids before 16 slices of 32), in FP32
# too; graphs with another set of CTAs follow one another on a cluster
FEW = [I.grid(8, 16), I.path(97), I.cycle(128), I.grid(3, 43), I.path(160), I.tri_mesh(16, 16)]
HUBS = [bipartite(32, 500), I.grid(30, 34), bipartite(32, 700), I.path(520), bipartite(33, 480)]


def _run(graphs, k, prec, iters):
    pos = [I.uniform_positions(g.n, 70 + i).astype(np.float32).astype(np.float64)
           for i, g in enumerate(graphs)]
    off = np.concatenate([[0], np.cumsum([g.n for g in graphs])])
    with G.Batch(graphs) as b:
        prm = G.params(k=k, iters=iters, precision=prec)
        out = G.gila_layout_batch_run(b.handle, prm, np.concatenate(pos))
        again = G.gila_layout_batch_run(b.handle, prm, np.concatenate(pos))
    assert np.array_equal(out, again)
    for i, g in enumerate(graphs):
        krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, k)
        yield g, pos[i], out[off[i]:off[i + 1]], O.run(g.n, g.row_ptr, g.col_idx, krow, kcol, pos[i],
                                                       iters)


@pytest.mark.parametrize("graphs,k", [(FEW[:1], 2), (FEW[1:3], 2), (FEW, 2), (HUBS[:1], 1), (HUBS, 1),
                                      (HUBS + FEW, 1)],
                         ids=["one", "two", "few", "hub", "hubs", "mixed"])
@pytest.mark.parametrize("iters", [1, 2, 7])
def test_empty_shares_fp64(graphs, k, iters):
    for g, x, got, want in _run(graphs, k, G.GILA_FP64, iters):
        assert np.abs(got - want).max() <= 1e-9 * np.abs(want).max(), g.name


@pytest.mark.parametrize("prec", [G.GILA_FP32, G.GILA_FP32_COMPENSATED], ids=["fp32", "fp32c"])
def test_empty_shares_fp32(prec):
    for g, x, got, want in _run(HUBS, 1, prec, 1):
        slack = 4 * np.finfo(np.float32).eps * np.abs(x).max()
        assert np.abs(got - want).max() <= 1e-4 * np.abs(want - x).max() + slack, g.name
    for g, x, got, want in _run(HUBS, 1, prec, 40):  # many exchanges, another set of CTAs a graph
        assert np.isfinite(got).all()
