"""The massive step at the sizes where its launch changes, against the oracle
(GPU): FP64 samples of up to 152 groups of 32 sites (one per SM) are updated
by four warps per group, up to 304 by two, larger ones by one; groups run
across row ends, so widths that are no multiple of 32 mix rows in a warp.
Bounds: the parity bars of the massive path after a few steps (FP64 1e-12,
FP32 1e-5, normwise).
"""
import numpy as np
import pytest

from oracle import massive as M

pytestmark = pytest.mark.gpu

# (nx, ny): the smallest sample; ragged rows; 152, 153, 304 and 305 groups
SIZES = [(5, 5), (33, 9), (64, 76), (61, 80), (64, 152), (61, 160)]


@pytest.fixture(scope="module")
def ms():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, massive
    build.build()
    return massive


@pytest.mark.parametrize("force", [(0.0, 0.0), (2e-5, -1e-5)])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_every_split_matches_the_oracle(ms, nx, ny, force):
    rng = np.random.default_rng(nx * 1000 + ny)
    f = [1 + 0.01 * rng.uniform(-1, 1, (ny, nx)), 0.02 * rng.uniform(-1, 1, (ny, nx)),
         0.02 * rng.uniform(-1, 1, (ny, nx)), 1 + 0.01 * rng.uniform(-1, 1, (ny, nx))]
    lat = M.Lattice(nx, ny, True, False, 0.8, *force)
    ref = M.fields(lat, M.run(lat, M.init(lat, *f), 3))
    for prec, tol in (("f64", 1e-12), ("f32", 1e-5)):
        with ms.MassiveSolver(nx, ny, True, False, 0.8, *force, prec=prec) as sv:
            sv.init(*[np.ascontiguousarray(a) for a in f])
            sv.step(3)
            got = sv.moments()
            sv.check()
        n, ux, uy, T = got
        rn, rx, ry, rT = ref
        du = np.sqrt((ux - rx) ** 2 + (uy - ry) ** 2).max() / np.sqrt(rx ** 2 + ry ** 2).max()
        assert max(np.abs(n - rn).max() / np.abs(rn).max(), du, np.abs(T - rT).max() / np.abs(rT).max()) <= tol
