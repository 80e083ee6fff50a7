"""A lambda that is not a number (of an imported state) at a site that does not
burn: the explicit rate, and with it f, becomes NaN there, the consistent one is
dlam / dt = 0 and f stays finite, whether or not other sites of the warp burn."""
import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nr,nth,variant", [(40, 4, 0), (200, 1, 0), (70, 50, 1), (70, 50, 4)])
@pytest.mark.parametrize("consistent", [0, 1])
@pytest.mark.parametrize("burning", [False, True])
def test_rate_of_a_nan(nr, nth, variant, precision, consistent, burning):
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = W.uniform_state(nr, nth, 1.0, 0.1, 0.0, 1.0, 0.2, dt=1e-6)
    w.params.update(omega1=2.0, omega2=3.0, reaction_energy=consistent)
    if burning:
        w.fields["T"][:, 36] = 1.3
    sim = dbm.Simulation(dict(w.params, precision=precision, variant=variant))
    sim.init_state(w.fields)
    f, lam, n = sim.export_state()
    lam[nth - 1, 33] = np.nan
    sim.import_state(f, lam, n)
    sim.step(1)
    f2, _, _ = sim.export_state()
    sim.close()
    bad = np.zeros((nth, nr), dtype=bool)
    bad[nth - 1, 33] = not consistent
    assert np.array_equal(np.isnan(f2), np.broadcast_to(bad, f2.shape))
