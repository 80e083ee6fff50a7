"""An even number of steps captured into a caller's CUDA graph leaves the state in
the buffer that it came from, so the graph can be replayed: on every path, also
where a pass makes several steps."""
import numpy as np
import pytest

from debug_ring_cases import DISC_SECTOR, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 4, 16, 18, 30])
@pytest.mark.parametrize("nr,nth,shape,precision,path", [
    (300, 1, {}, "fp32", "row"), (95, 1, DISC_SECTOR, "fp32", "row"), (300, 1, {}, "fp64", "direct"),
    (64, 33, {}, "fp32", "direct"), (321, 973, {}, "fp32", "ring")])
def test_replays_advance(nr, nth, shape, precision, path, n):
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = workload(nr, nth, **shape)
    sim, ref = (dbm.Simulation(dict(w.params, precision=precision, variant=v)) for v in (0, 3))
    assert sim.step_path() == path
    for s in (sim, ref):
        s.init_state(w.fields)
    sim.step(n)                    # and what it builds on first use
    at = sim.state_device()[0]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sim.step(n, stream=torch.cuda.current_stream())
    assert sim.state_device()[0] == at
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    ref.step(4 * n)
    got, want = sim.export_state(), ref.export_state()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    for s in (sim, ref):
        s.close()
