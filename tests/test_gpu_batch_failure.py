"""Failure detection of batches without a fault: a test hook lets the clusters
announce positions without pushing them, so that every wait runs out after a
millisecond, the launch ends by itself, and the batch it belongs to reports
GILA_ECUDA once. Only graphs that a cluster takes wait, which also tells the
form that serves a graph."""
import numpy as np
import pytest

import __graft_entry__
from paper_1606_02162_gb300 import gila as G
from paper_1606_02162_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    import torch
    torch.cuda.set_device(0)


def _fails(call):
    with pytest.raises(G.GilaError) as err:
        call()
    assert err.value.status == G.GILA_ECUDA and "did not receive" in str(err.value)


# in a batch of one graph a cluster takes it from 16 slices of 32 rows (FP32) or
# 4 (FP64) on
@pytest.mark.parametrize("prec,n,cluster", [
    (G.GILA_FP32, 480, False), (G.GILA_FP32, 481, True), (G.GILA_FP32, 513, True),
    (G.GILA_FP32_COMPENSATED, 480, False), (G.GILA_FP32_COMPENSATED, 512, True),
    (G.GILA_FP64, 96, False), (G.GILA_FP64, 97, True), (G.GILA_FP64, 129, True),
])
def test_cluster_wait_is_reported_and_context_survives(prec, n, cluster):
    import torch
    g = I.cycle(n)
    pos = I.uniform_positions(n, 3)
    prm = G.params(k=2, iters=9, precision=prec)
    dt = torch.float64 if prec == G.GILA_FP64 else torch.float32
    with G.Batch([g]) as b, G.Batch([g]) as other:
        want = G.gila_layout_batch_run(b.handle, prm, pos)
        G.gila_batch_set_wait_test(b.handle, True)
        x = torch.tensor(pos, dtype=dt, device="cuda")
        if not cluster:
            assert np.array_equal(G.gila_layout_batch_run(b.handle, prm, pos), want)
            return
        _fails(lambda: G.gila_layout_batch_run(b.handle, prm, pos))
        # a caller that stays on the device learns of it by the next call
        G.gila_layout_batch_device(b.handle, prm, x)  # asynchronous: no error yet
        torch.cuda.synchronize()
        assert np.array_equal(G.gila_layout_batch_run(other.handle, prm, pos), want)
        G.gila_batch_set_wait_test(b.handle, False)
        _fails(lambda: G.gila_layout_batch_device(b.handle, prm, x))
        # told once; the batch and the context go on working
        assert np.array_equal(G.gila_layout_batch_run(b.handle, prm, pos), want)
        x = torch.tensor(pos, dtype=dt, device="cuda")
        G.gila_layout_batch_device(b.handle, prm, x)
        torch.cuda.synchronize()
        assert np.array_equal(x.double().cpu().numpy(), want)


def test_graphs_beside_a_failed_cluster():
    """Several graphs, some on clusters: every launch ends, whichever fail."""
    graphs = [I.grid(30, 34), I.grid(8, 16), I.path(33), I.star(200), I.tri_mesh(25, 25), I.path(5)]
    pos = np.concatenate([I.uniform_positions(g.n, 20 + i) for i, g in enumerate(graphs)])
    prm = G.params(k=2, iters=50, precision=G.GILA_FP64)
    with G.Batch(graphs) as b:
        want = G.gila_layout_batch_run(b.handle, prm, pos)
        G.gila_batch_set_wait_test(b.handle, True)
        for _ in range(2):
            _fails(lambda: G.gila_layout_batch_run(b.handle, prm, pos))
        G.gila_batch_set_wait_test(b.handle, False)
        assert np.array_equal(G.gila_layout_batch_run(b.handle, prm, pos), want)
