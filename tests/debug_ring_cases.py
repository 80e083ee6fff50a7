"""Row-ring cases run by tests/test_gpu_debug_ring.py in a child process, once
with the release library and once with the checked one (DBM_DEBUG=1): every
ring pipeline of both precisions on ragged and degenerate grids, disc sectors
and full discs, and a batch of such simulations.  Writes every final state,
status and path to the .npz file given as argument."""
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

from paper_1308_0653_gb300 import dbm  # noqa: E402
from paper_1308_0653_gb300 import workloads as W  # noqa: E402


def workload(nr, nth, sector=0, centre=False, seed=0):
    """Smooth fields that straddle the ignition temperature, Courant number below 0.6."""
    r_in = 0.0 if centre else 0.5
    dr, dth = 1.0 / nr, (np.pi / 4 if sector else 2.0 * np.pi) / nth
    dt = 0.3 * min(dr, (r_in + 0.5 * dr) * dth) / 12.5
    w = W.random_smooth(nr, nth, seed=seed + nr + nth, amp=0.1, r_in=r_in, r_out=r_in + 1.0, dt=dt, tau=50 * dt,
                        omega1=3.0, omega2=5.0, sector=sector)
    if centre:
        w.params["r_bc_inner"] = "centre"
    w.fields["T"] = w.fields["T"] * 0.9
    return w


SECTOR, DISC, DISC_SECTOR = dict(sector=1), dict(centre=True), dict(sector=1, centre=True)
SMALL = [(5, 3, {}, 0), (130, 16, {}, 1), (257, 9, {}, 4), (150, 1, DISC_SECTOR, 0), (70, 9, SECTOR, 2),
         (40, 32, DISC, 5)]
# variant 4 of FP32 runs its ring beyond 64 warps of 32 sites per SM only
LARGE = [(321, 973, {}, 0), (321, 974, DISC, 7), (330, 980, DISC_SECTOR, 0)]
CASES = ([("fp32", v, *c) for v in (1, 2, 3, 5) for c in SMALL] + [("fp32", 4, *c) for c in LARGE] +
         [("fp32", 5, *LARGE[1])] + [("fp64", v, *c) for v in (1, 3, 4, 5) for c in SMALL])


def main(out):
    import torch
    torch.cuda.set_device(0)
    res = {"library": np.array(dbm.lib_path())}

    def record(key, sim):
        f, lam, _ = sim.export_state()
        res[key + "_f"], res[key + "_lam"] = f, lam
        res[key + "_status"] = np.array(dbm.dbm_status(sim.h))

    for prec, variant, nr, nth, shape, rows in CASES:
        w = workload(nr, nth, **shape)
        sim = dbm.Simulation(dict(w.params, precision=prec, variant=variant, rows_per_item=rows))
        sim.init_state(w.fields)
        sim.step(9)
        key = f"{prec}_v{variant}_{nr}x{nth}_{rows}"
        res[key + "_path"] = np.array(sim.step_path())
        record(key, sim)
        sim.close()
    b = dbm.Batch(5, 1 << 15, precision="fp32", rows_per_item=7)
    ws = [workload(640, 620), workload(130, 70, **DISC), workload(97, 60, **DISC_SECTOR), workload(33, 5)]
    sims = []
    for slot, w in zip((0, 1, 3, 4), ws):
        sims.append(dbm.Simulation(dict(w.params, precision="fp32")))
        sims[-1].init_state(w.fields)
        b.attach(slot, sims[-1], 10 + 5 * slot)
    b.step(40)
    res["batch_path"] = np.array(b.step_path())
    for k, sim in enumerate(sims):
        record(f"batch{k}", sim)
        sim.close()
    b.close()
    np.savez(out, **res)


if __name__ == "__main__":
    main(sys.argv[1])
