"""The batch autotuner compares what would step the batch: kernels without work
items are timed once and keep the batch's rows, and a small FP32 batch stays on
the direct kernel."""
import numpy as np
import pytest

from debug_ring_cases import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,sizes,path", [
    ("fp64", [(130, 70), (97, 60)], "direct"), ("fp32", [(64, 64), (160, 130)], "direct"),
    ("fp32", [(640, 620), (130, 70)], "ring")])
def test_candidates_are_what_steps(precision, sizes, path):
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ws = [workload(*s) for s in sizes]
    b = dbm.Batch(4, 1 << 14, precision=precision, rows_per_item=9)
    sims = []
    for slot, w in enumerate(ws):
        sims.append(dbm.Simulation(dict(w.params, precision=precision)))
        sims[-1].init_state(w.fields)
        b.attach(slot, sims[-1], 10000)
    v, r, ms = b.autotune(steps=64)
    assert b.step_path() == path
    if path == "direct":
        assert v == (2 if precision == "fp64" else 4) and r == 9
        assert ms[0] > 0 and list(ms[1:4]) == [ms[0]] * 3
        assert b.time() == (1 if precision == "fp64" else 5) * (32 + 128)
    else:
        assert r in (16, 32, 64, -1) and b.time() == 8 * (32 + 128)
    assert (list(ms[4:8]) == [0.0] * 4) == (precision == "fp64")
    n = b.time()
    for sim, w in zip(sims, ws):
        f, lam, steps = sim.export_state()
        alone = dbm.Simulation(dict(w.params, precision=precision, variant=3))
        alone.init_state(w.fields)
        alone.step(n)
        ref = alone.export_state()
        assert steps == n and np.array_equal(f, ref[0]) and np.array_equal(lam, ref[1])
        alone.close()
        sim.close()
    b.close()
