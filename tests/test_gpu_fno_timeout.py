"""A bounded wait of the fused operator kernels that gives up (needs a GB300).

The kernels wait on mbarriers for their MMAs.  With a limit of one clock cycle
the first probe, which does not block, comes before an MMA can end (hundreds
of cycles), so blocks give up: they leave out what depends on the wait, set the
flag that rlbm_gemm_tc_error reports, wait with the default limit for the MMAs
they have committed, and return.  Nothing here faults or hangs the GPU: every
wait is bounded and every MMA completes.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, fno
    build.build()
    return torch, fno


def flag(fno):
    v = ctypes.c_int()
    assert fno._lib().rlbm_gemm_tc_error(ctypes.byref(v)) == 0
    return v.value


# one tile per canvas row and one round of the transform; two tiles and two rounds
@pytest.mark.parametrize("N,B,L", [(32, 1, 1), (136, 1, 2), (256, 2, 2)])
def test_giving_up_is_reported_and_the_operator_recovers(env, N, B, L):
    torch, fno = env
    net = fno.FNO(fno.FNOConfig(N=N, L=L), batch=B, seed=5)
    g = np.random.default_rng(3)
    rows = B * N * N
    x = torch.tensor(g.standard_normal((rows, 5)), dtype=torch.bfloat16, device="cuda")
    t = torch.tensor(g.standard_normal((rows, 4)), dtype=torch.float32, device="cuda")
    m = torch.ones(rows, dtype=torch.float32, device="cuda")

    def both():
        y = net.forward(x).clone()
        net.loss(t, m)
        return y, net.backward().clone()

    y0, g0 = both()
    assert flag(fno) == 0
    net.wait_limit = 1
    net.forward(x)
    assert flag(fno) == 1
    assert flag(fno) == 0                       # cleared by the report
    net.wait_limit = 0
    net.forward(x)
    net.loss(t, m)
    net.wait_limit = 1
    net.backward()
    assert flag(fno) == 1
    net.wait_limit = 0
    y1, g1 = both()
    assert flag(fno) == 0
    assert torch.equal(y0, y1)
    # gradients: FP32 sums whose order varies (atomics)
    assert float((g0 - g1).abs().max()) <= 2e-5 * float(g0.abs().max())
    net.wait_limit = -1
    with pytest.raises(RuntimeError):
        net.forward(x)
