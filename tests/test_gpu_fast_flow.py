"""Diagnostics of FP64 states in fast flow: their rounding errors are no larger
than those of sums over the velocities about u, in which nothing cancels."""
import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SPEEDS = np.concatenate([[0.0], np.repeat(W.PAPER_SPEEDS, 8)])[:, None, None]
H = 0.70710678118654752440
CX = np.concatenate([[0.0], np.tile([1, H, 0, -H, -1, -H, 0, H], 4)])[:, None, None]
CY = np.concatenate([[0.0], np.tile([0, H, 1, H, 0, -H, -1, -H], 4)])[:, None, None]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


def _state(u, nr=96, nth=64):
    """A state whose sites move at about u in all directions: f^eq by the oracle's
    init, each f off by up to 5 %."""
    import oracle as orc
    w = W.uniform_state(nr, nth, 1.0, 0.0, 0.0, 1.6, 0.3, dt=1e-6)
    n = (nth, nr)
    ang = 2.0 * np.pi * W.uniform(5, 1, nth * nr).reshape(n)
    size = u * (0.95 + 0.1 * W.uniform(5, 2, nth * nr).reshape(n))
    w.fields["ur"], w.fields["uth"] = size * np.cos(ang), size * np.sin(ang)
    w.fields["T"] = 1.6 + 0.16 * W.uniform(5, 3, nth * nr).reshape(n)
    op = orc.make_params(**{k: v for k, v in w.params.items() if k != "precision"})
    f, lam = orc.init(op, w.fields)
    f = f * (1.0 + 0.05 * (2.0 * W.uniform(6, 4, f.size).reshape(f.shape) - 1.0))
    return w, f, lam


def _about_u(f, real):
    """rho, v - u and its terms in `real`, velocity by velocity."""
    r2 = np.sqrt(real(2)) / 2
    unit = [x.astype(real) if real is np.float64 else np.where(np.abs(x) == H, np.sign(x).astype(real) * r2,
                                                                x.astype(real)) for x in (CX, CY)]
    vx, vy = SPEEDS.astype(real) * unit[0], SPEEDS.astype(real) * unit[1]
    f = f.astype(real)
    rho, jx, jy = f[0] * 0, f[0] * 0, f[0] * 0
    for q in range(33):
        rho, jx, jy = rho + f[q], jx + f[q] * vx[q], jy + f[q] * vy[q]
    return f, rho, vx - jx / rho, vy - jy / rho


def _temperature(f, real):
    f, rho, a, b = _about_u(f, real)
    e = f[0] * 0
    for q in range(33):
        e = e + f[q] * (a[q] * a[q] + b[q] * b[q])
    return e / (2 * rho)


@pytest.mark.parametrize("u", [0.0, 0.7, 1.4, 1.7, 2.0, 2.5])
def test_temperature_is_as_exact_as_a_second_pass(u):
    from paper_1308_0653_gb300 import dbm
    w, f, lam = _state(u)
    sim = dbm.Simulation(dict(w.params, precision="fp64"))
    sim.import_state(f, lam, 0)
    got = sim.moments()["T"]
    sim.close()
    exact = _temperature(f, np.longdouble)
    rms = [float(np.sqrt(np.mean(((T - exact) / exact).astype(np.float64) ** 2)))
           for T in (got, _temperature(f, np.float64))]
    print("RMS", u, rms)
    assert rms[0] <= rms[1], rms


def _delta(f, theta, real):
    """Delta* by sums over v - u in the polar frame."""
    f, rho, dx, dy = _about_u(f, real)
    c, s = np.cos(theta.astype(np.longdouble)).astype(real), np.sin(theta.astype(np.longdouble)).astype(real)
    a, b = dx * c[:, None] + dy * s[:, None], -dx * s[:, None] + dy * c[:, None]
    M = [rho * 0 for _ in range(12)]
    for q in range(33):
        x, y, g = a[q], b[q], f[q]
        h = g * (x * x + y * y) / 2
        for k, term in enumerate((g * x * x, g * x * y, g * y * y, g * x * x * x, g * x * x * y, g * x * y * y,
                                  g * y * y * y, h * x, h * y, h * x * x, h * x * y, h * y * y)):
            M[k] = M[k] + term
    T = (M[0] + M[2]) / (2 * rho)
    for k, e in ((0, rho * T), (2, rho * T), (9, 2 * rho * T * T), (11, 2 * rho * T * T)):
        M[k] = M[k] - e
    return np.array(M)


ORDERS = {"2": (0, 1, 2), "3": (3, 4, 5, 6), "3,1": (7, 8), "4,2": (9, 10, 11)}


@pytest.mark.parametrize("u", [0.0, 0.5, 0.7, 1.0, 1.5, 2.0, 2.5])
def test_delta_is_as_exact_as_central_sums(u):
    from paper_1308_0653_gb300 import dbm
    w, f, lam = _state(u)
    sim = dbm.Simulation(dict(w.params, precision="fp64"))
    sim.import_state(f, lam, 0)
    got = sim.noneq()
    sim.close()
    theta = 2 * np.arctan2(np.longdouble(0), np.longdouble(-1)) * np.arange(f.shape[1]) / f.shape[1]
    exact, plain = _delta(f, theta, np.longdouble), _delta(f, theta, np.float64)
    rms = {k: [float(np.sqrt(np.mean((x[list(c)] - exact[list(c)]).astype(np.float64) ** 2))) for x in (got, plain)]
           for k, c in ORDERS.items()}
    print("RMS", u, rms)
    assert all(a <= b for a, b in rms.values()), rms
