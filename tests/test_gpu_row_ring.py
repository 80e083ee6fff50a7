"""The row ring where it is what steps: its default pipelines (FP32 variants 4
and 5) on grids beyond the direct kernel's line, with full discs, disc sectors,
narrow last strips and forced rows per item, FP64's pipelines against its direct
kernel, and batches on the ring (items cut shorter, simulations that join and
leave), each with the path asserted and bit for bit."""
import numpy as np
import pytest

from debug_ring_cases import DISC, DISC_SECTOR, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


def _run(w, precision, variant, path, steps=(1, 33, 2), rows=0):
    from paper_1308_0653_gb300 import dbm
    sim = dbm.Simulation(dict(w.params, precision=precision, variant=variant, rows_per_item=rows))
    assert sim.step_path() == path
    if rows:
        assert sim.launch_info()["rows_per_item"] == min(rows, w.params["ntheta"])
    sim.init_state(w.fields)
    for n in steps:
        sim.step(n)
    f, lam, _ = sim.export_state()
    assert dbm.dbm_status(sim.h) == dbm.DBM_OK and np.isfinite(f).all()
    sim.close()
    return f, lam


@pytest.mark.parametrize("nr,nth,shape,rows", [
    (321, 974, DISC, 0), (321, 974, DISC, 5), (330, 980, DISC_SECTOR, 3),
    (130, 2500, {}, 0), (130, 2500, {}, 1), (417, 801, {}, 64), (600, 620, DISC, 0)])
def test_fp32_pipelines(nr, nth, shape, rows):
    w = workload(nr, nth, **shape)
    ref = _run(w, "fp32", 2, "ring", rows=rows)
    for variant in (4, 5):
        got = _run(w, "fp32", variant, "ring", rows=rows)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), variant


@pytest.mark.parametrize("nr,nth,shape,rows,variant", [
    (2, 20000, {}, 0, 5), (32, 17000, DISC, 16, 5), (32, 9730, {}, 16, 4), (33, 12000, {}, 0, 4)])
def test_fp32_strips_of_one_warp(nr, nth, shape, rows, variant):
    """Three CTAs per SM, which leave out warps without a site, beyond L2."""
    from paper_1308_0653_gb300 import dbm
    w = workload(nr, nth, **shape)
    sim = dbm.Simulation(dict(w.params, precision="fp32", rows_per_item=rows))
    assert sim.launch_info()["variant"] == variant
    sim.close()
    got, ref = (_run(w, "fp32", v, "ring", (1, 4), rows) for v in (0, 2))
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])


@pytest.mark.parametrize("nr,nth,shape,rows", [
    (130, 48, {}, 1), (200, 33, {}, 7), (64, 40, DISC, 0), (65, 9, DISC_SECTOR, 2), (300, 301, {}, 4),
    (700, 500, {}, 9)])  # the last two: several items per CTA
def test_fp64_pipelines(nr, nth, shape, rows):
    w = workload(nr, nth, **shape)
    ref = _run(w, "fp64", 2, "direct", (1, 4, 2))
    for variant in (1, 3, 4, 5):
        got = _run(w, "fp64", variant, "ring", (1, 4, 2), rows)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), variant


def test_the_defaults_of_small_grids_and_rows():
    from paper_1308_0653_gb300 import dbm
    for nr, nth, precision, path in ((320, 972, "fp32", "direct"), (300, 1, "fp32", "row"), (300, 1, "fp64", "direct"),
                                     (700, 700, "fp64", "direct"), (321, 973, "fp32", "ring")):
        sim = dbm.Simulation(dict(workload(nr, nth).params, precision=precision))
        assert sim.step_path() == path
        sim.close()


def _check(batch, sims):
    from paper_1308_0653_gb300 import dbm
    for sim, w, n in sims:
        f, lam, steps = sim.export_state()
        assert steps == n and dbm.dbm_status(sim.h) == dbm.DBM_OK
        alone = _run(w, "fp32", 3, "ring", (n,))
        assert np.array_equal(f, alone[0]) and np.array_equal(lam, alone[1]), w.params["nr"]
        sim.close()
    batch.close()


def _sims(ws):
    from paper_1308_0653_gb300 import dbm
    out = []
    for w in ws:
        out.append(dbm.Simulation(dict(w.params, precision="fp32")))
        out[-1].init_state(w.fields)
    return out


@pytest.mark.parametrize("rows", [0, 7, 100])
def test_batches_whose_members_join_and_leave(rows):
    from paper_1308_0653_gb300 import dbm
    ws = [workload(640, 620), workload(130, 70, **DISC), workload(97, 60, **DISC_SECTOR), workload(250, 300),
          workload(33, 5)]
    sims = _sims(ws)
    b = dbm.Batch(4, 8192, rows_per_item=rows)
    for slot in range(3):
        b.attach(slot, sims[slot], 1000)
    b.step(20)
    assert b.step_path() == "ring"
    b.detach(1)
    b.step(14)
    b.attach(1, sims[3], 33)
    b.attach(3, sims[4], 1000)
    b.step(40)
    assert b.step_path() == "ring" and b.remaining(1) == 0
    _check(b, [(s, w, n) for s, w, n in zip(sims, ws, (74, 20, 74, 33, 40))])


def test_a_batch_of_few_items_cuts_them_shorter():
    """640 x 620: 195 items of 16 rows would leave CTAs idle, 5 x 57 of 11 don't."""
    from paper_1308_0653_gb300 import dbm
    w = workload(640, 620)
    sims = _sims([w])
    b = dbm.Batch(4, 4096)
    b.attach(0, sims[0], 1000)
    b.step(37)
    info = b.launch_info()
    assert b.step_path() == "ring" and info["rows_per_item"] == 16
    cost = {c: -(-5 * -(-620 // c) // info["grid"]) * (c + 2) for c in range(1, 17)}
    best = [c for c in cost if cost[c] == min(cost.values())]
    assert 16 not in best and info["items"] in [5 * -(-620 // c) for c in best]
    _check(b, [(sims[0], w, 37)])
