"""FP64 samples of few sites: the step that shares a site between three warps
against the batched kernel, which updates a site in one thread (GPU).

Both form the same FP64 operations in the same order (the step modules are
compiled without contraction), so states agree bit for bit; the residual's
sums run in another order (1e-12 relative).
"""
import numpy as np
import pytest

from paper_1804_02418_gb300 import workloads as W

pytestmark = pytest.mark.gpu

C = W.Contact
# at most 152 warp tiles (one per SM) take the split step: the smallest sample,
# one lane in the last tile of a row, full tiles, the largest count (2 x 76
# tiles) and one past it (which does not)
SAMPLES = {
    "smallest": lambda: W.Sample(11, 11, tau=0.6, Fy=1e-5),
    "one_lane": lambda: W.Sample(33, 40, tau=0.9, Fx=2e-5, Fy=-1e-5,
                                 contacts=[C(0, 5, 9, u_n=0.01), C(2, 8, 12, n=1.01)]),
    "periodic_no_force": lambda: W.Sample(64, 64, periodic_x=True, periodic_y=True, tau=0.8),
    "electric_force": lambda: W.Sample(50, 45, tau=0.8, Fx=1e-5, inv_cg=0.1, periodic_x=True),
    "most_tiles": lambda: W.Sample(60, 76, tau=1.2, Fx=1e-5),
    "one_more_row": lambda: W.Sample(60, 77, tau=1.2, Fx=1e-5),
}


@pytest.fixture(scope="module")
def rl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, rlbm
    build.build()
    return rlbm


@pytest.mark.parametrize("name", sorted(SAMPLES))
def test_split_step_equals_one_thread_per_site(rl, name):
    s = SAMPLES[name]()
    f = [np.ascontiguousarray(a) for a in W.random_fields(s, 5, du=0.05, dn=0.02, dT=0.02)]
    got = []
    for shape in ((0, 0, 0), (128, 0, 0)):
        with rl.Solver(s, prec="f64") as sv:
            sv.init(0, *f)
            sv.set_launch_shape(*shape)
            sv.step(7)
            r = sv.step(6, residual=True)
            sv.check()
            got.append((sv.get_state(), r))
    assert np.array_equal(got[0][0], got[1][0])
    assert abs(got[0][1] - got[1][1]) <= 1e-12 * got[1][1]


@pytest.mark.parametrize("prec,own", [("f32", True), ("f16dev", True), ("f64", False)])
def test_tuning_of_a_single_sample(rl, prec, own):
    """FP32 arithmetic and buffers within reach of the L2: the sample's own
    kernel, untimed; FP64 is timed and may take any shape."""
    s = SAMPLES["electric_force"]()
    with rl.Solver(s, prec=prec) as sv:
        sv.init(0)
        shape = sv.autotune()
        sv.step(2)
        sv.check()
    assert shape == (0, 0, 0) if own else shape[0] in (0, 64, 128, 256)
