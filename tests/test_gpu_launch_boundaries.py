"""FP64 samples at the sizes where the launch changes, from the device's SM
count (GPU): the step that shares a site between warps takes at most one warp
tile of 32 sites per SM (massive: two groups of 32 sites per SM), and up to two
64-thread blocks per SM a step does not place its successor's blocks early.
The massless step is compared bit for bit with the batched kernel (the same
FP64 operations in the same order), the massive one with the oracle.
"""
import numpy as np
import pytest

from oracle import massive as M
from paper_1804_02418_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, massive, rlbm
    build.build()
    return rlbm, massive, torch.cuda.get_device_properties(0).multi_processor_count


def state(rl, s, f, shape, steps=8):
    with rl.Solver(s, prec="f64") as sv:
        sv.init(0, *f)
        sv.set_launch_shape(*shape)
        sv.step(steps)
        r = sv.step(4, residual=True)
        sv.check()
        return sv.get_state(), r


# warp tiles: SMs, SMs + 1 (last split step, first whole one), 4 SMs, 4 SMs + 1
# (two blocks per SM, and one more); rows of one tile (20 sites) and ragged rows
# of two (45 sites)
@pytest.mark.parametrize("per_row", [1, 2])
@pytest.mark.parametrize("times,more", [(1, 0), (1, 1), (4, 0), (4, 1)])
def test_massless_steps_agree(lib, per_row, times, more):
    rl, _, sms = lib
    rows = -(-(times * sms) // per_row) + more
    s = W.Sample(20 if per_row == 1 else 45, rows, periodic_x=True, tau=0.7, Fx=1e-5, Fy=-2e-5)
    f = [np.ascontiguousarray(a) for a in W.random_fields(s, 3, du=0.05, dn=0.02, dT=0.02)]
    a, ra = state(rl, s, f, (0, 0, 0))
    b, rb = state(rl, s, f, (64, 0, 0))
    assert np.array_equal(a, b)
    assert abs(ra - rb) <= 1e-12 * rb


@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("times", [1, 2])
def test_massive_groups(lib, times, more):
    _, ms, sms = lib
    nx, ny = 32, times * sms + more          # one group of 32 sites per row
    rng = np.random.default_rng(ny)
    f = [1 + 0.01 * rng.uniform(-1, 1, (ny, nx)), 0.02 * rng.uniform(-1, 1, (ny, nx)),
         0.02 * rng.uniform(-1, 1, (ny, nx)), 1 + 0.01 * rng.uniform(-1, 1, (ny, nx))]
    lat = M.Lattice(nx, ny, False, True, 0.8, 1e-5, -1e-5)
    ref = M.fields(lat, M.run(lat, M.init(lat, *f), 2))
    with ms.MassiveSolver(nx, ny, False, True, 0.8, 1e-5, -1e-5, prec="f64") as sv:
        sv.init(*f)
        sv.step(2)
        got = sv.moments()
        sv.check()
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 1e-12 * max(np.abs(r).max(), 0.02)


def test_the_tuned_shape_gives_the_same_state(lib):
    rl = lib[0]
    s = W.Sample(90, 70, tau=0.8, Fx=1e-5, inv_cg=0.1, periodic_x=True)
    f = [np.ascontiguousarray(a) for a in W.random_fields(s, 8, du=0.02, dn=0.01, dT=0.01)]
    with rl.Solver(s, prec="f64") as sv:
        sv.init(0, *f)
        shape = sv.autotune()
    a, _ = state(rl, s, f, shape)
    for other in ((0, 0, 0), (256, 0, 0)):
        assert np.array_equal(a, state(rl, s, f, other)[0]), (shape, other)
