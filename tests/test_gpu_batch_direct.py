"""Batches stepped straight from global memory (every FP64 batch, FP32 ones up to
16 tiles per SM): uneven and tiny simulations, sectors, disc centres, empty slots,
more than one group of 32 slots, simulations that end at different steps, and
FP32 batches that cross the line between the kernels, bit for bit against each
simulation alone in the row ring."""
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


def _workload(nr, nth, sector=0, centre=False, v_scale=1.0):
    r_in = 0.0 if centre else 0.5
    dth = (np.pi / 4 if sector else 2 * np.pi) / nth
    dt = 0.3 * min(1.0 / nr, (r_in + 0.5 / nr) * dth) / 12.5
    w = W.random_smooth(nr, nth, seed=nr + nth, amp=0.1, r_in=r_in, r_out=r_in + 1.0, dt=dt, tau=50 * dt,
                        omega1=3.0, omega2=5.0, sector=sector)
    if centre:
        w.params["r_bc_inner"] = "centre"
    w.params["v"] = [x * v_scale for x in (W.base_params().get("v") or (1.0, 2.92, 5.84, 8.76))]
    w.fields["T"] = w.fields["T"] * 0.9  # straddle the ignition temperature
    return w


def _alone(w, precision, nsteps):
    from paper_1308_0653_gb300 import dbm
    sim = dbm.Simulation(dict(w.params, precision=precision, variant=3))
    sim.init_state(w.fields)
    sim.step(nsteps)
    got = sim.export_state()
    sim.close()
    return got


def _check(sims, precision):
    for sim, w, n in sims:
        got, ref = sim.export_state(), _alone(w, precision, n)
        assert got[2] == n and np.isfinite(got[0]).all(), w.name
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), (w.name, w.params["nr"])


SMALL = [(1, 8), (31, 3), (33, 5), (64, 4), (97, 1)]
TURNED = [(40, 2, 1), (70, 9, 1, True), (60, 16, 0, True)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("slots,shapes", [
    (1, [(33, 7)]),
    (8, SMALL + TURNED),
    (70, SMALL + TURNED),           # three groups, the first, middle and last slots
    (32, [(160, 130), (129, 200)]),  # several waves and leftovers
])
def test_same_bits_as_alone(slots, shapes, precision):
    from paper_1308_0653_gb300 import dbm
    at = [i * (slots - 1) // max(1, len(shapes) - 1) for i in range(len(shapes))]
    b = dbm.Batch(slots, 8192, precision=precision)
    sims = []
    for k, (slot, shape) in enumerate(zip(at, shapes)):
        w = _workload(*shape, v_scale=1.0 + 0.01 * k)
        s = dbm.Simulation(dict(w.params, precision=precision))
        s.init_state(w.fields)
        b.attach(slot, s, 40 if k % 2 == 0 else 23)
        sims.append((s, w, 40 if k % 2 == 0 else 23))
    b.step(33)
    b.step(7)
    _check(sims, precision)
    b.close()
    for s, _, _ in sims:
        s.close()


def test_across_the_line_between_the_kernels():
    from paper_1308_0653_gb300 import dbm
    b = dbm.Batch(4, 8192, precision="fp32")
    ws = [_workload(96, 80), _workload(640, 620), _workload(130, 70)]
    sims = []
    for w in ws:
        sims.append(dbm.Simulation(dict(w.params, precision="fp32")))
        sims[-1].init_state(w.fields)
    b.attach(0, sims[0], 1000)
    b.step(34)             # straight from global memory
    b.attach(1, sims[1], 1000)
    b.step(34)             # the row ring
    b.detach(1)
    b.attach(3, sims[2], 1000)
    b.step(35)
    _check([(sims[0], ws[0], 103), (sims[1], ws[1], 34), (sims[2], ws[2], 35)], "fp32")
    b.close()
    for s in sims:
        s.close()


def test_constants_either_way():
    """The row ring's constants from registers (large batches) and through uniform registers."""
    from paper_1308_0653_gb300 import dbm
    b = dbm.Batch(3, 1 << 15, precision="fp32")
    ws = [_workload(700, 600, v_scale=1.01), _workload(130, 70, sector=1), _workload(2500, 2450)]
    sims = []
    for w in ws:
        sims.append(dbm.Simulation(dict(w.params, precision="fp32")))
        sims[-1].init_state(w.fields)
    b.attach(0, sims[0], 1000)
    b.attach(1, sims[1], 1000)
    b.step(34)             # 2800 sites per SM
    b.attach(2, sims[2], 1000)
    b.step(34)             # 43 000
    b.detach(2)
    b.step(35)
    _check([(sims[0], ws[0], 103), (sims[1], ws[1], 103), (sims[2], ws[2], 34)], "fp32")
    b.close()
    for s in sims:
        s.close()
