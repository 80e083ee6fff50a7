"""Moments and non-equilibrium moments of one raw state against the oracle at
the edges of their kernels: 256-site blocks that span many short rows, ragged
last blocks, single rows and single sites, sectors, zero and subnormal f."""
import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ORDER = np.array([2, 2, 2, 3, 3, 3, 3, 3, 3, 4, 4, 4])  # velocity power of each Delta* component


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nr,nth,sector", [(1, 300, 0), (3, 171, 0), (255, 2, 0), (257, 1, 1), (64, 9, 0), (1, 1, 1),
                                           (513, 8, 0)])
def test_diagnostics_of_a_raw_state(orc, nr, nth, sector, precision):
    from paper_1308_0653_gb300 import dbm
    w = W.random_smooth(nr, nth, seed=nr + nth, amp=0.1, r_in=0.5, r_out=1.5, sector=sector, dt=1e-5)
    op = orc.make_params(**{k: v for k, v in w.params.items() if k != "precision"})
    f, lam = orc.init(op, w.fields)
    real = np.float64 if precision == "fp64" else np.float32
    off = 2.0 * W.uniform(3, 40, f.size).reshape(f.shape) - 1.0
    f = (f * (1.0 + 0.05 * off)).astype(real)
    f[5].flat[0], f[6].flat[0] = 0.0, 1e-40  # zero, and a subnormal of FP32
    lam = (lam if precision == "fp64" else 1.0 - lam).astype(real)
    sim = dbm.Simulation(dict(w.params, precision=precision))
    try:
        sim.import_state(f, lam, 0)
        got, mom = sim.noneq(), sim.moments(totals=True)
    finally:
        sim.close()
    f64 = f.astype(np.float64)
    # Rounding: a component of velocity power n is some 33 + 60 rounded sums and
    # products of quantities bounded by S_n = sum |f| (|v| + |u|)^n, on each side
    ref = orc.noneq(op, f64)
    macro = orc.macro(op, f64, lam.astype(np.float64))
    speed = np.concatenate([[0.0], np.repeat(np.asarray(w.params["v"]), 8)])[:, None, None]
    u = np.hypot(macro["ur"], macro["uth"])
    for c in range(12):
        S = (np.abs(f64) * (speed + u) ** ORDER[c]).sum(0)
        assert (np.abs(got[c] - ref[c]) <= 200 * 2.0 ** -53 * S).all(), f"component {c}"
    # moments: 33 sums and some 20 operations in the state's precision, T's over
    # sum f v^2 / rho + u^2
    eps = 2.0 ** (-53 if precision == "fp64" else -24)
    vmax = float(max(w.params["v"]))
    scale = {"rho": macro["rho"], "ur": 0 * u + vmax, "uth": 0 * u + vmax, "T": macro["T"] + u * u}
    for k, s in scale.items():
        assert (np.abs(mom[k] - macro[k]) <= 60 * eps * s).all(), k
    tot = orc.totals(op, f64)
    weight = 60 * eps * np.array([tot[0], tot[0] * vmax, tot[0] * vmax, tot[3]])
    assert (np.abs(mom["totals"] - tot) <= weight).all()
