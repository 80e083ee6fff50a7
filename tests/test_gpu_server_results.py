"""Arrays of a polled result are its block of host memory: writable, apart from
each other, valid after the server has gone, and freed once with the last of them."""
import gc

import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_result_arrays_outlive_the_server(monkeypatch):
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = W.explosion(70, 33, nsteps=0, seed=3, dt=2e-6)
    p = dict(w.params, precision="fp32")
    sim = dbm.Simulation(p)
    sim.init_state(w.fields)
    sim.step(5)
    ref = {k: np.empty((33, 70)) for k in dbm.FIELDS}
    dbm.dbm_moments(sim.h, *[ref[k] for k in dbm.FIELDS], totals=np.zeros(4))
    sim.close()

    lib, freed = dbm._server_lib(), []

    class Counting:
        def __getattr__(self, name):
            if name != "dbm_result_free":
                return getattr(lib, name)
            return lambda r: freed.append(lib.dbm_result_free(r))

    monkeypatch.setattr(dbm, "_server_lib", Counting)
    server = dbm.Server(64 << 20, max_slots=2, quantum=8, precision="fp32")
    status, out = server.poll(server.submit(p, w.fields, 5))
    server.close()
    assert status == dbm.DBM_OK and out["steps"] == 5
    for k in dbm.FIELDS:
        assert out[k].shape == (33, 70) and out[k].dtype == np.float64
        assert np.array_equal(out[k], ref[k])
        out[k] += 1.0
    last = out["ur"]
    del out
    gc.collect()
    assert not freed and np.array_equal(last, ref["ur"] + 1.0)
    del last
    gc.collect()
    assert freed == [dbm.DBM_OK]
