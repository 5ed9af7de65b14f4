"""Reading a batch's tuning back and setting it again changes nothing: the same
form of the kernel (the lane groups add in another order, so that results tell
them apart) and the same results, whatever was set and whoever chose it."""
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


@pytest.mark.parametrize("prec", [G.GILA_FP32, G.GILA_FP32_COMPENSATED, G.GILA_FP64],
                         ids=["fp32", "fp32c", "fp64"])
def test_tuning_round_trip(prec):
    import torch
    graphs = I.batch_mix(24, 40, 900, 5)
    pos = np.concatenate([I.uniform_positions(g.n, 30 + i) for i, g in enumerate(graphs)])
    prm = G.params(k=2, iters=12, precision=prec)

    def run(b):
        return G.gila_layout_batch_run(b.handle, prm, pos)

    settings = [dict(), dict(threads=256, ctas_per_sm=8), dict(ctas_per_sm=1),
                dict(group4_max=8, group8_max=24, group16_max=64), dict(group8_max=12)]
    outs = []
    for s in settings:
        with G.Batch(graphs) as b:
            G.gila_batch_tune(b.handle, **s)
            outs.append(run(b))
            for read in (G.GILA_FP32, G.GILA_FP64):
                t = G.gila_batch_get_tuning(b.handle, read)
                assert all(t[f] == v for f, v in s.items())
                G.gila_batch_tune(b.handle, **t)
                assert np.array_equal(run(b), outs[-1])
                assert G.gila_batch_get_tuning(b.handle, read) == t
    rows, groups = outs[0], outs[3]
    assert np.array_equal(outs[1], rows) and np.array_equal(outs[2], rows)
    assert not np.array_equal(rows, groups)
    # the autotuner's answer says which form it chose, and gives it on another batch
    x = torch.tensor(pos, dtype=torch.float64 if prec == G.GILA_FP64 else torch.float32, device="cuda")
    with G.Batch(graphs) as b:
        t = G.gila_batch_autotune(b.handle, prm, x, 2)
        tuned = run(b)
    with G.Batch(graphs) as b:
        G.gila_batch_tune(b.handle, **t)
        assert np.array_equal(run(b), tuned)
    if t["group4_max"] == 0:
        assert np.array_equal(tuned, rows)
