"""Cases run by tests/test_gpu_abort.py in a child process with the checked
library (DBM_DEBUG=1): steps of the row ring whose producer stops early.  Prints
one JSON line of [case, status after the step, seconds] and then the status of
an ordinary simulation."""
import json
import os
import sys
import time

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

from paper_1308_0653_gb300 import dbm  # noqa: E402
from paper_1308_0653_gb300 import workloads as W  # noqa: E402

# nr, ntheta, precision, variant, rows loaded per CTA, rows per item (which loads two
# more): within an item, or within a CTA's second one (items of 2 rows)
ALONE = [(300, 72, "fp32", 1, 3, 16), (300, 72, "fp32", 2, 3, 16), (300, 72, "fp32", 3, 5, 16),
         (321, 973, "fp32", 4, 7, 16), (300, 72, "fp32", 5, 2, 16), (300, 72, "fp64", 1, 3, 16),
         (300, 72, "fp64", 3, 3, 16), (300, 72, "fp64", 4, 4, 16), (321, 973, "fp32", 4, 6, 2),
         (150, 900, "fp64", 5, 6, 2)]


def _sim(nr, nth, precision, variant=0, stop=0, rows=0):
    w = W.random_smooth(nr, nth, seed=nr, dt=1e-6)
    sim = dbm.Simulation(dict(w.params, precision=precision, variant=variant, rows_per_item=rows))
    sim.init_state(w.fields)
    if stop:
        dbm.dbm_selftest_stop_loads(sim.h, stop)
    return sim


def main():
    import torch
    torch.cuda.set_device(0)
    out = []
    for nr, nth, precision, variant, stop, rows in ALONE:
        sim = _sim(nr, nth, precision, variant, stop, rows)
        t = time.perf_counter()
        sim.step(1)
        st = dbm.dbm_status(sim.h)
        out.append([f"{precision} variant {variant} {nr}x{nth}", st, time.perf_counter() - t])
        sim.close()
    # a batch: several items per CTA, whose warps meet at a barrier for each
    batch = dbm.Batch(3, 1 << 14, precision="fp32")
    sims = [_sim(1000, 900, "fp32", stop=25), _sim(130, 70, "fp32", stop=25), _sim(700, 640, "fp32", stop=25)]
    for slot, sim in enumerate(sims):
        batch.attach(slot, sim, 10)
    t = time.perf_counter()
    batch.step(1)
    st = [dbm.dbm_status(sim.h) for sim in sims]
    out.append(["batch", min(st), time.perf_counter() - t])
    batch.close()
    for sim in sims:
        sim.close()
    sim = _sim(300, 72, "fp32", 2)
    sim.step(3)
    out.append(["after", dbm.dbm_status(sim.h), 0.0])
    sim.close()
    print(json.dumps(out))


if __name__ == "__main__":
    main()
