"""The blocked kernel's windows with several ranges. Meshes take a row per lane
since that form exists; one whose adjacency rows are not ascending keeps the
windows with shares, scans over the warps' rows and the finish in the CTA.

One step within 1e-4 (FP32 modes) and 1e-12 (FP64) of the largest move; quality
figures within 1e-11 relative."""
import numpy as np
import pytest

import __graft_entry__
import oracle as O
from paper_1606_02162_gb300 import gila as G
from paper_1606_02162_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {G.GILA_FP32: 1e-4, G.GILA_FP32_COMPENSATED: 1e-4, G.GILA_FP64: 1e-12}
NAME = "blocked_kernel (window)"


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    import torch
    torch.cuda.set_device(0)


def mesh(rows, cols, isolated):
    """A triangulated mesh, then vertices without edges; adjacency rows in
    descending order."""
    m = I.tri_mesh(rows, cols)
    g = I.csr_from_edges(m.n + isolated, *m.edge_list())
    col = g.col_idx.copy()
    for u in range(g.n):
        col[g.row_ptr[u]:g.row_ptr[u + 1]] = col[g.row_ptr[u]:g.row_ptr[u + 1]][::-1]
    return I.Graph(g.name, g.n, g.row_ptr, col)


@pytest.mark.parametrize("prec", list(TOL), ids=["fp32", "fp32c", "fp64"])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("tune", [{}, dict(ctas_per_sm=1), dict(ctas_per_sm=12)],
                         ids=["cps2", "cps1", "cps12"])
@pytest.mark.parametrize("pq", [(2, 1), (3, 2)], ids=["fr", "p3q2"])
def test_window_ranges(k, prec, tune, pq):
    import torch
    g = mesh(120, 110, 37)
    p, q = pq
    pos = I.uniform_positions(g.n, 6).astype(np.float32).astype(np.float64)
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, k)
    _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, 0.4, d=1.2, p=p, q=q)
    x = torch.tensor(pos, dtype=torch.float64 if prec == G.GILA_FP64 else torch.float32, device="cuda")
    y, disp = torch.empty_like(x), torch.empty_like(x)
    prm = G.params(k=k, d=1.2, p=p, q=q, precision=prec)
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, tiled=1, **tune)
        G.gila_profile_enable(h.handle, 2)
        G.gila_layout_step(h.handle, prm, 0.4, x, y, disp)
        torch.cuda.synchronize()
        assert G.gila_profile_read_kernel(h.handle)["name"] == NAME
        got = disp.double().cpu().numpy()
        assert np.abs(got - want).max() <= TOL[prec] * np.abs(want).max()
        assert (got[g.n - 37:] == 0).all()
        if prec != G.GILA_FP64:
            figures = G.gila_layout_metrics(h.handle, prm, x)
            for key, v in O.metrics(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, d=1.2, p=p, q=q).items():
                assert figures[key] == pytest.approx(v, rel=1e-11), key


def test_window_wait_runs_out():
    import torch
    g = mesh(60, 70, 0)
    pos = I.uniform_positions(g.n, 32).astype(np.float32).astype(np.float64)
    prm = G.params(k=2)
    krow, kcol = O.khop(g.n, g.row_ptr, g.col_idx, 2)
    _, want = O.step(g.n, g.row_ptr, g.col_idx, krow, kcol, pos, 0.4)
    x = torch.tensor(pos, dtype=torch.float32, device="cuda")
    y, disp = torch.empty_like(x), torch.empty_like(x)
    with G.Graph.from_inputs(g) as h:
        G.gila_graph_tune(h.handle, tiled=1)
        G.gila_profile_enable(h.handle, 2)
        G.gila_graph_set_wait_test(h.handle, True)
        G.gila_layout_step(h.handle, prm, 0.4, x, y, disp)
        with pytest.raises(G.GilaError) as err:
            G.gila_layout_metrics(h.handle, prm, x)
        assert err.value.status == G.GILA_ECUDA and "did not complete" in str(err.value)
        assert G.gila_profile_read_kernel(h.handle)["name"] == NAME
        G.gila_graph_set_wait_test(h.handle, False)
        G.gila_layout_step(h.handle, prm, 0.4, x, y, disp)
        got = disp.double().cpu().numpy()
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()
