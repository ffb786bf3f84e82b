"""Initial fields with |u| near 1 in FP32 arithmetic (GPU), against the oracle.

gamma and gamma - 1 of initial fields are formed in FP64, whose 1 - u^2 has all
its digits however close |u| is to 1, and rounded once.  What follows is FP32:
z^3 with z = W + X vx + Y vy, whose terms carry a few roundings of 2^-24 each
and are cancelled against one another only below their own size, so a site's
populations are right to about 20 x 2^-24 of its largest deviation: bound 2e-6.
BF16 storage adds its own rounding, 2^-9 of each value: bound 2^-8.
"""
import numpy as np
import pytest

from oracle import lbm
from paper_1804_02418_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ONE_MINUS_U = [0.5, 0.1, 1e-2, 1e-4, 5e-7, 1e-8, 2e-9]


@pytest.fixture(scope="module")
def rl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, rlbm
    build.build()
    return rlbm


@pytest.mark.parametrize("prec,tol", [("f32", 2e-6), ("bf16dev", 2.0 ** -8)])
def test_fast_initial_fields(rl, prec, tol):
    nx, ny = 32, len(ONE_MINUS_U) * 2
    s = W.Sample(nx, ny, periodic_x=True, periodic_y=True, tau=0.8)
    rng = np.random.default_rng(4)
    speed = 1.0 - np.repeat(ONE_MINUS_U, 2)[:, None]
    phi = rng.uniform(0, 2 * np.pi, (ny, nx))
    f = [rng.uniform(0.5, 1.5, (ny, nx)), speed * np.cos(phi), speed * np.sin(phi),
         rng.uniform(0.5, 1.5, (ny, nx))]
    assert np.all(f[1] ** 2 + f[2] ** 2 < 1.0)
    want = lbm.equilibrium_deviation(*f)
    with rl.Solver(s, prec=prec) as sv:
        sv.init(0, *f)
        sv.check()
        got = sv.get_state()
    assert np.isfinite(got).all()
    err = np.abs(got - want).max(axis=0) / np.abs(want).max(axis=0)
    assert err.max() <= tol, err.max(axis=1)
