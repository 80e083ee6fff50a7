"""The checked build's bounds and alignment checks in the row ring: no check of
a copy, a store or a neighbour read fires in any of its pipelines, and the
results equal the release build's bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _run(out, debug):
    env = dict(os.environ)
    env.pop("DBM_DEBUG", None)
    if debug:
        env["DBM_DEBUG"] = "1"
    r = subprocess.run([sys.executable, os.path.join(HERE, "debug_ring_cases.py"), str(out)], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    return dict(np.load(out))


def test_checks_of_the_row_ring_are_silent(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    rel = _run(tmp_path / "release.npz", False)
    dbg = _run(tmp_path / "debug.npz", True)
    assert "_build_debug" in str(dbg.pop("library")) and "_build_debug" not in str(rel.pop("library"))
    assert rel.keys() == dbg.keys()
    for k in rel:
        if k.endswith("_status"):
            assert int(dbg[k]) == 0 and int(rel[k]) == 0, k  # DBM_OK: no check fired
        elif k.endswith("_path"):
            assert str(dbg[k]) == str(rel[k]) == "ring", k
        else:
            assert np.isfinite(rel[k]).all() and np.array_equal(rel[k], dbg[k]), k
