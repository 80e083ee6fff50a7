"""What the autotuner stores for a grid on the row ring does not take smaller
grids of the same powers of two off the direct kernel."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# in a process of its own: tuned choices last as long as the process
SCRIPT = """
from debug_ring_cases import workload
from paper_1308_0653_gb300 import dbm
def sim(nr, nth):
    return dbm.Simulation(dict(workload(nr, nth).params, precision="fp32"))
big = sim(777, 501)
assert big.step_path() == "ring"
best, ms = big.autotune(steps=50)
big.close()
assert sim(777, 501).launch_info()["variant"] == best and sim(1000, 510).launch_info()["variant"] == best
small = sim(600, 300)
assert small.launch_info()["variant"] == 4 and small.step_path() == "direct", (best, ms)
print("best", best)
"""


def test_tuning_a_ring_grid_leaves_direct_ones():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    here = os.path.dirname(os.path.abspath(__file__))
    path = os.pathsep.join([os.path.dirname(here), here])
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=dict(os.environ, PYTHONPATH=path), capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    assert "best" in r.stdout
