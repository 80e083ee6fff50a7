"""Batches that do not fill the persistent CTAs are cut into shorter work items,
with the same bits as a simulation alone."""
import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("sizes", [((300, 90),), ((130, 64), (40, 500)), ((512, 512),)])
def test_small_batches_use_shorter_items(sizes, precision):
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ws = [W.explosion(nr, nth, nsteps=0, seed=nr, dt=2e-6) for nr, nth in sizes]
    b = dbm.Batch(4, 4096, precision=precision)
    sims = []
    for slot, w in enumerate(ws):
        s = dbm.Simulation(dict(w.params, precision=precision))
        s.init_state(w.fields)
        b.attach(slot, s, 40)
        sims.append(s)
    b.step(40)
    info = b.launch_info()
    assert info["rows_per_item"] == 16
    width = 128 if precision == "fp32" else 64
    items = {c: sum(-(-nr // width) * -(-nth // c) for nr, nth in sizes) for c in range(1, 17)}
    cost = {c: -(-n // info["grid"]) * (c + 2) for c, n in items.items()}
    best = min(cost.values())
    # the table holds the items of a choice no worse than any other (and padding)
    assert any(items[c] <= info["items"] for c in cost if cost[c] == best)
    assert info["items"] > items[16] or cost[16] == best
    for s, w in zip(sims, ws):
        got = s.export_state()
        alone = dbm.Simulation(dict(w.params, precision=precision, variant=2))
        alone.init_state(w.fields)
        alone.step(40)
        ref = alone.export_state()
        alone.close()
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    b.close()
    for s in sims:
        s.close()
