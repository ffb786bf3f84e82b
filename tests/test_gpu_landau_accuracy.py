"""FP64 fields of uniform states with |u| from 0.1 to 0.3 (GPU), against a
solve of the Landau frame with 40 digits (mpmath).

The state's moments differ from those of the populations handed over only by
roundings of the deviations (each below 0.4 in size: moments of about 20
populations, a dozen operations after them), about 10 x 0.2 x 2^-53 = 2.2e-16,
and T = 1 + dT is rounded once more: |T| error at most 3.5e-16.  u is of size
0.3 and the result of a quotient and three products: 2.5e-16.
"""
import numpy as np
import pytest

from oracle import lbm
from paper_1804_02418_gb300 import workloads as W

pytestmark = pytest.mark.gpu
mp = pytest.importorskip("mpmath")


@pytest.fixture(scope="module")
def rl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, rlbm
    build.build()
    return rlbm


def exact_fields(delta, P):
    """(ux, uy, T) of 48 deviations, 40 digits."""
    mp.mp.dps = 40
    d = [mp.mpf(float(x)) for x in delta]
    p = [[mp.mpf(float(x)) for x in row] for row in P]
    s = lambda a, b=None: sum(x * p[a][i] * (p[b][i] if b is not None else 1) for i, x in enumerate(d))
    E, Mx, My = 2 + s(0, 0), s(0, 1), s(0, 2)
    Pxx, Pxy = 1 + s(1, 1), s(1, 2)
    Pyy = E - Pxx                       # massless: T^00 = T^xx + T^yy
    e = E
    for _ in range(60):
        a, c = Pxx + e, Pyy + e
        det = a * c - Pxy * Pxy
        ux, uy = (c * Mx - Pxy * My) / det, (a * My - Pxy * Mx) / det
        step = (e - E + Mx * ux + My * uy) / (1 - ux * ux - uy * uy)
        e -= step
        if abs(step) < mp.mpf(10) ** -35:
            break
    n = ((1 + s(0)) - ux * s(1) - uy * s(2)) / mp.sqrt(1 - ux * ux - uy * uy)
    return ux, uy, e / (2 * n)


def test_fields_against_forty_digits(rl):
    rng = np.random.default_rng(9)
    t = lbm.tables()
    samples, states = [], []
    for _ in range(64):
        u, phi = rng.uniform(0.1, 0.3), rng.uniform(0, 2 * np.pi)
        d = lbm.equilibrium_deviation(*[np.array([v]) for v in (
            rng.uniform(0.95, 1.05), u * np.cos(phi), u * np.sin(phi), rng.uniform(0.95, 1.05))])[:, 0]
        d += t.w * 0.02 * rng.uniform(-1, 1, 48)
        samples.append(W.Sample(11, 11, periodic_x=True, periodic_y=True, tau=0.8))
        states.append(d)
    worst_u = worst_T = 0.0
    with rl.Solver(samples, prec="f64") as sv:
        for k, d in enumerate(states):
            sv.set_state(np.ascontiguousarray(np.broadcast_to(d[:, None, None], (48, 11, 11))), k)
        for k, d in enumerate(states):
            n, ux, uy, T = sv.moments(k)
            ex, ey, eT = exact_fields(d, t.P)
            worst_u = max(worst_u, abs(float(mp.mpf(ux[5, 5]) - ex)), abs(float(mp.mpf(uy[5, 5]) - ey)))
            worst_T = max(worst_T, abs(float(mp.mpf(T[5, 5]) - eT)))
        sv.check()
    assert worst_T <= 3.5e-16, worst_T
    assert worst_u <= 2.5e-16, worst_u
