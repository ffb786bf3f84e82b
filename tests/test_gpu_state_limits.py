"""Values at the limits through state I/O and initialisation (GPU)."""
import numpy as np
import pytest

from paper_1804_02418_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, massive, rlbm
    build.build()
    return rlbm, massive


@pytest.mark.parametrize("which", ["f64", "f32", "f16dev", "bf16dev", "massive_f64", "massive_f32"])
def test_infinite_deviations_pass_through(lib, which):
    """delta / w of an infinite delta is infinite (and NaN stays NaN)."""
    rlbm, massive = lib
    q = 45 if which.startswith("massive") else 48
    d = np.zeros((q, 11, 11))
    d[:, 3, 4] = np.inf
    d[:, 7, 2] = -np.inf
    d[:, 5, 5] = np.nan
    sv = (massive.MassiveSolver(11, 11, True, True, 0.8, prec=which[8:]) if q == 45
          else rlbm.Solver(W.Sample(11, 11, periodic_x=True, periodic_y=True), prec=which))
    with sv:
        sv.set_state(d)
        got = sv.get_state()
    assert np.array_equal(got, d, equal_nan=True)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_subnormal_density_is_positive(lib, prec):
    rlbm, _ = lib
    n = np.ones((11, 11))
    n[2, 3], n[4, 4] = 5e-324, 1e-310
    z = np.zeros((11, 11))
    with rlbm.Solver(W.Sample(11, 11), prec=prec) as sv:
        sv.init(0, n, z, z, np.ones((11, 11)))
        sv.check()
        n[2, 3] = 0.0
        sv.init(0, n, z, z, np.ones((11, 11)))
        with pytest.raises(rlbm.RlbmError):
            sv.check()
