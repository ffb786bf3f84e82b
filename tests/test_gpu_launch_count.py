"""Kernel launches that a context counts (GPU)."""
import numpy as np
import pytest

from paper_1804_02418_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, rlbm
    build.build()
    return rlbm


@pytest.mark.parametrize("prec,kernels", [("f64", 2), ("f32", 2), ("f16dev", 1)])
def test_launch_count_of_the_seed(rl, prec, kernels):
    """The Chapman-Enskog seed is two kernels with FP64 and FP32 storage."""
    one, zero = np.ones((40, 50)), np.zeros((40, 50))
    with rl.Solver(W.Sample(50, 40), prec=prec) as sv:
        before = sv.launches
        sv.init_ce(0, one, zero, zero, one)
        assert sv.launches - before == kernels
