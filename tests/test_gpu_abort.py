"""Waits of the row ring that run out: with a producer that stops early every
warp of the block leaves by the abort path, the step ends within the waits'
limits with DBM_ETIMEOUT, and the GPU goes on working.  A warp's lanes, some of
which may have seen the row or the abort flag and some not, decide together
(they vote, shuffle and meet at warp barriers afterwards), and a batch's warps
all come to each item's barrier."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_steps_with_a_stopped_producer_end_with_a_timeout():
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    r = subprocess.run([sys.executable, os.path.join(HERE, "abort_cases.py")], env=dict(os.environ, DBM_DEBUG="1"),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    *cases, after = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(cases) == 11 and after[1] == dbm.DBM_OK
    for name, status, seconds in cases:
        # a wait takes 2^31 cycles; a block gives up after one or two of them
        assert status == dbm.DBM_ETIMEOUT and 0.5 < seconds < 6.0, (name, status, seconds)


def test_the_release_library_loads_everything():
    import torch
    from paper_1308_0653_gb300 import dbm
    from paper_1308_0653_gb300 import workloads as W
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = W.explosion(64, 64, nsteps=0, dt=2e-6)
    sim = dbm.Simulation(dict(w.params, precision="fp32", variant=2))
    with pytest.raises(dbm.DbmError) as e:
        dbm.dbm_selftest_stop_loads(sim.h, 3)
    assert e.value.status == dbm.DBM_EINVAL
    sim.close()
