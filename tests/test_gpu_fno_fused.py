"""The fused kernels of the neural operator against the same operator as a
sequence of GEMMs (GPU).

Every BF16-rounded value is formed by the same FP32 operations in the same
order on both paths, so outputs and everything the forward pass keeps are equal
bit for bit.  Weight and bias gradients are FP32 sums over all sites in another
order.  With p sites per partial sum and values of size s, reordering moves a
sum of n terms by at most about log2(n) 2^-24 times the sum of magnitudes; the
GEMM sequence adds its partial sums with atomics, whose order varies from run
to run by the same measure.  Bound: 2e-5 of each tensor's largest entry (the
gradients of these shapes cancel by less than a factor of ten).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# canvas edges: the smallest, ragged tiles (N not a multiple of 128 or 64), one
# full tile, a full tile and a remainder, two tiles, the largest; inputs 1, 5, 16
SHAPES = [(32, 1, 5, 2), (40, 3, 1, 1), (72, 2, 16, 2), (128, 2, 5, 3), (136, 1, 5, 2),
          (256, 2, 5, 4), (512, 1, 5, 2)]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, fno
    build.build()
    return torch, fno


def step(torch, fno, cfg, B, fused, monkeypatch):
    if not fused:
        monkeypatch.setattr(fno, "_fused_shape", lambda lib, cfg: False)
    net = fno.FNO(cfg, batch=B, seed=11)
    monkeypatch.undo()
    assert net.fused is fused
    g = np.random.default_rng(7)
    rows = B * cfg.N * cfg.N
    x = torch.tensor(g.standard_normal((rows, cfg.cin)), dtype=torch.bfloat16, device="cuda")
    t = torch.tensor(0.3 * g.standard_normal((rows, 4)), dtype=torch.float32, device="cuda")
    m = torch.tensor((g.uniform(0, 1, rows) < 0.7), dtype=torch.float32, device="cuda")
    y = net.forward(x).clone()
    loss = float(net.loss(t, m))
    grad = net.backward().clone()
    torch.cuda.synchronize()
    kept = [h.clone() for h in net.h16] + [z.clone() for z in net.z] + [s.clone() for s in net.S2]
    kept.append(net.x16.clone())
    grads = {k: net.get(k, "grad").double().cpu().numpy() for k in net.offsets}
    return y, loss, grads, kept, grad


@pytest.mark.parametrize("N,B,cin,L", SHAPES)
def test_fused_kernels_equal_the_gemm_sequence(env, monkeypatch, N, B, cin, L):
    import ctypes
    torch, fno = env
    cfg = fno.FNOConfig(N=N, cin=cin, L=L)
    y0, l0, g0, k0, _ = step(torch, fno, cfg, B, False, monkeypatch)
    y1, l1, g1, k1, flat = step(torch, fno, cfg, B, True, monkeypatch)
    flag = ctypes.c_int()
    assert fno._lib().rlbm_gemm_tc_error(ctypes.byref(flag)) == 0 and flag.value == 0
    for a, b in zip(k0, k1):
        assert torch.equal(a, b)
    assert torch.equal(y0, y1)
    assert abs(l0 - l1) <= 1e-6 * l0
    for k in g0:
        assert np.abs(g0[k] - g1[k]).max() <= 2e-5 * np.abs(g0[k]).max(), k
    assert torch.isfinite(flat).all()


def test_fused_forward_takes_any_input_layout(env):
    """Inputs the kernels cannot read directly (another type, strided, not
    16-byte aligned) give the same outputs."""
    torch, fno = env
    net = fno.FNO(fno.FNOConfig(N=32), batch=1, seed=3)
    rows = 32 * 32
    x = torch.randn(rows, 5, device="cuda").to(torch.bfloat16)
    ref = net.forward(x).clone()
    wide = torch.zeros(rows, 6, dtype=torch.bfloat16, device="cuda")
    wide[:, 1:] = x
    shifted = torch.zeros(rows * 5 + 1, dtype=torch.bfloat16, device="cuda")[1:].view(rows, 5)
    shifted.copy_(x)
    for other in (x.float(), x.cpu(), wide[:, 1:], shifted):
        assert torch.equal(net.forward(other), ref)
    with pytest.raises(RuntimeError):
        net.forward(x[:-1])
