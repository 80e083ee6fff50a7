"""The FP64 step straight from global memory (a single simulation's default)
against the row-ring kernel (variant 4), bit for bit, at the edges of its
tasks: 32-site chunks and their 8-site quarters, whole waves of warps with a
remainder in quarters, every kind of neighbour."""
import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


def _states(w, **kw):
    from paper_1308_0653_gb300 import dbm
    got = []
    for variant in (0, 4):
        sim = dbm.Simulation(dict(w.params, precision="fp64", variant=variant, **kw))
        sim.init_state(w.fields)
        sim.step(35)
        f, lam, _ = sim.export_state()
        assert dbm.dbm_status(sim.h) == dbm.DBM_OK
        got.append((f, lam))
        sim.close()
    return got


@pytest.mark.parametrize("nr,nth,kw", [
    (1, 3, {}), (7, 2, {}), (31, 5, {}), (33, 1, {}), (40, 16, {}),            # quarters only
    (32, 620, {}), (32, 668, {}), (64, 400, {}),           # a wave, rest in quarters, 1, 2, 4 to a block
    (100, 230, {}),                                                            # rest too large for quarters
    (257, 151, dict(reaction_energy=1, m=1.5, n=0.7)),                         # more than two waves
    (45, 6, dict(sector=1)), (45, 1, dict(sector=1)), (300, 2, dict(sector=1, r_in=0.0, r_bc_inner="centre")),
    (70, 12, dict(r_in=0.0, r_bc_inner="centre")),
])
def test_same_bits_as_the_row_ring(nr, nth, kw):
    r_in = kw.pop("r_in", 0.5)
    sector = kw.pop("sector", 0)
    inner = kw.pop("r_bc_inner", "outflow")
    dth = (np.pi / 4 if sector else 2 * np.pi) / nth
    dr = 1.0 / nr
    dt = 0.35 * min(dr, (r_in + 0.5 * dr) * dth) / 12.5
    w = W.random_smooth(nr, nth, seed=nr + nth, amp=0.1, r_in=r_in, r_out=r_in + 1.0, dt=dt, tau=50 * dt,
                        omega1=3.0, omega2=5.0, sector=sector)
    w.params["r_bc_inner"] = inner
    w.fields["T"] = w.fields["T"] * 0.9  # straddle the ignition temperature
    (f, lam), (fr, lr) = _states(w, **kw)
    assert np.isfinite(f).all()
    assert np.array_equal(f, fr) and np.array_equal(lam, lr)


def test_nan_in_lambda_reaches_f():
    """A NaN lambda makes R, and with it the site's f, NaN even where nothing burns."""
    from paper_1308_0653_gb300 import dbm
    w = W.uniform_state(40, 4, 1.0, 0.1, 0.0, 1.0, 0.2, dt=1e-5)
    for variant in (0, 4):
        sim = dbm.Simulation(dict(w.params, precision="fp64", variant=variant))
        sim.init_state(w.fields)
        f, lam, n = sim.export_state()
        lam[2, 33] = np.nan
        sim.import_state(f, lam, n)
        sim.step(1)
        f2, _, _ = sim.export_state()
        sim.close()
        bad = np.zeros((4, 40), dtype=bool)
        bad[2, 33] = True
        assert np.isnan(f2[:, bad]).all() and np.isfinite(f2[:, ~bad]).all()
