"""The FP32 default's other kernels (straight from global memory on small grids,
several steps per pass on a single theta row) and the staged row stores of the
row ring against variant 2's row ring, bit for bit, at their edges: 32-site
warps, four-row blocks, one-row blocks, 96-site row blocks and their 16-step
passes, the line between the kernels, ragged widths, every kind of neighbour."""
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


def _workload(nr, nth, r_in=0.5, sector=0, r_bc_inner="outflow"):
    dth = (np.pi / 4 if sector else 2 * np.pi) / nth
    dr = 1.0 / nr
    dt = 0.35 * min(dr, (r_in + 0.5 * dr) * dth) / 12.5
    w = W.random_smooth(nr, nth, seed=nr + nth, amp=0.1, r_in=r_in, r_out=r_in + 1.0, dt=dt, tau=50 * dt,
                        omega1=3.0, omega2=5.0, sector=sector)
    w.params["r_bc_inner"] = r_bc_inner
    w.fields["T"] = w.fields["T"] * 0.9  # straddle the ignition temperature
    return w


@pytest.mark.parametrize("nr,nth,shape,options", [
    (31, 3, {}, {}), (33, 4, {}, {}), (129, 5, {}, dict(reaction_energy=1, m=1.5, n=0.7)),  # small grids
    (40, 2, dict(sector=1), {}), (70, 9, dict(sector=1, r_in=0.0, r_bc_inner="centre"), {}),
    (60, 12, dict(r_in=0.0, r_bc_inner="centre"), {}),
    (320, 972, {}, {}), (321, 973, {}, {}),                       # the last grid below the line, one above
    (129, 2500, {}, {}), (255, 1300, {}, {}), (417, 800, {}, {}),  # ring: ragged last strips of 1, 127, 33 sites
    (15, 1, {}, {}), (96, 1, {}, {}), (97, 1, {}, {}), (1000, 1, {}, {}),                    # single rows
    (193, 1, dict(sector=1), dict(reaction_energy=1, m=1.5, n=0.7)),
    (500, 1, dict(sector=1, r_in=0.0, r_bc_inner="centre"), {}),
])
def test_same_bits_as_the_row_ring(nr, nth, shape, options):
    from paper_1308_0653_gb300 import dbm
    w = _workload(nr, nth, **shape)
    got = []
    for variant in (0, 2):
        sim = dbm.Simulation(dict(w.params, precision="fp32", variant=variant, **options))
        sim.init_state(w.fields)
        for n in (1, 17, 33, 2):  # passes of 1, 16 + 1, a graph + 1, 2 steps
            sim.step(n)
        f, lam, steps = sim.export_state()
        assert steps == 53 and dbm.dbm_status(sim.h) == dbm.DBM_OK
        got.append((f, lam))
        sim.close()
    assert np.isfinite(got[0][0]).all()
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("nr,nth", [(40, 4), (200, 1), (700, 700)])
def test_nan_in_lambda_reaches_f(nr, nth):
    """A NaN lambda makes R, and with it the site's f, NaN even where nothing burns."""
    from paper_1308_0653_gb300 import dbm
    w = W.uniform_state(nr, nth, 1.0, 0.1, 0.0, 1.0, 0.2, dt=1e-6)
    sim = dbm.Simulation(dict(w.params, precision="fp32"))
    sim.init_state(w.fields)
    f, lam, n = sim.export_state()
    lam[nth - 1, 33] = np.nan
    sim.import_state(f, lam, n)
    sim.step(1)
    f2, _, _ = sim.export_state()
    sim.close()
    bad = np.zeros((nth, nr), dtype=bool)
    bad[nth - 1, 33] = True
    assert np.isnan(f2[:, bad]).all() and np.isfinite(f2[:, ~bad]).all()


@pytest.mark.parametrize("nr,nth,variant", [
    (385, 880, 5), (1001, 311, 5), (777, 501, 5),         # items short enough, ragged last strips
    (417, 800, 4), (600, 600, 4),                         # not short enough
    (2048, 512, 4),                                       # two states beyond L2
    (1000, 1, 4), (64, 64, 4),                            # the kernels without items
])
@pytest.mark.parametrize("shape", [{}, dict(sector=1, r_in=0.0, r_bc_inner="centre")])
def test_shape_of_the_row_ring(nr, nth, variant, shape):
    """Three CTAs per SM where the rule asks for them, with the other shapes' bits."""
    from paper_1308_0653_gb300 import dbm
    w = _workload(nr, nth, **shape)
    got = []
    for v in (0, 4, 5):
        sim = dbm.Simulation(dict(w.params, precision="fp32", variant=v))
        assert sim.launch_info()["variant"] == (v or variant)
        sim.init_state(w.fields)
        for n in (1, 33, 2):
            sim.step(n)
        f, lam, _ = sim.export_state()
        assert dbm.dbm_status(sim.h) == dbm.DBM_OK
        got.append((f, lam))
        sim.close()
    assert np.isfinite(got[0][0]).all()
    for f, lam in got[1:]:
        assert np.array_equal(f, got[0][0]) and np.array_equal(lam, got[0][1])
