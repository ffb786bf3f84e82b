"""FP64 Landau solve of fast massive states (GPU).

The FP64 Newton iteration starts from the solution of the same iteration in
FP32.  These uniform states (equilibrium moments of n, T, |u|, phi) take 13 to
15 of the 16 FP64 steps from eps = T^00, and the FP32 iteration, which sees
1 - u^2 with 1e-7 of error, does not converge on them: its last iterate must
not become the start of the FP64 iteration.  Fields: u to 1e-9 (the root is
nearly double: its error is the moments' rounding over 1 - u^2, about 1e-15 /
1e-3, with a factor of 1e3 for the 45 populations' cancellation).
"""
import numpy as np
import pytest

from oracle import massive as M

pytestmark = pytest.mark.gpu

STATES = [(2.709, 0.424, 0.999632, 4.7992), (0.88, 1.217, 0.999211, 0.9155), (1.416, 1.05, 0.99876, 3.9342),
          (1.15, 0.468, 0.99924, 5.7957), (0.755, 0.847, 0.999192, 0.196), (2.896, 1.78, 0.999539, 3.2024),
          (1.613, 0.681, 0.998125, 2.4603), (0.704, 1.865, 0.999325, 1.7916), (0.94, 0.743, 0.999499, 0.1342),
          (1.532, 0.393, 0.998715, 0.3535), (1.76, 1.687, 0.997902, 5.3541), (3.077, 2.774, 0.99926, 1.7002),
          (1.044, 1.151, 0.999244, 0.107), (2.388, 2.549, 0.99965, 3.1801), (0.503, 1.701, 0.999113, 3.9961),
          (1.586, 0.593, 0.998794, 3.4693), (0.747, 1.406, 0.997942, 2.1971), (1.426, 0.614, 0.999038, 1.7832),
          (1.671, 1.496, 0.999446, 1.849), (0.543, 2.398, 0.999719, 3.7676), (1.854, 0.659, 0.998643, 5.9166),
          (0.855, 0.809, 0.999654, 3.5995), (1.795, 0.57, 0.999109, 3.3092), (1.643, 3.071, 0.999278, 0.6396)]


@pytest.fixture(scope="module")
def ms():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02418_gb300 import build, massive
    build.build()
    return massive


def deviations(n, T, u, phi):
    """45 deviations from the rest populations (least norm) with the moments
    N^a = n U^a and T^ab of the massive equation of state."""
    m, g = 5.0, 1.0 / np.sqrt(1.0 - u * u)
    U = g * np.array([1.0, u * np.cos(phi), u * np.sin(phi)])
    h = n * (m * m + 3 * m * T + 3 * T * T) / (m + T)
    N, Tab = n * U, h * np.outer(U, U) - n * T * np.diag([1.0, -1.0, -1.0])
    p = M.quadrature()["p"]
    N0, T0 = M.moments(M.rest_populations())
    ab = [(a, b) for a in range(3) for b in range(a, 3)]
    A = np.array([p[:, a] for a in range(3)] + [p[:, a] * p[:, b] for a, b in ab])
    rhs = np.concatenate([N - N0, [Tab[a, b] - T0[a, b] for a, b in ab]])
    f0 = M.rest_populations()
    return f0 * (np.linalg.pinv(A * f0) @ rhs), U[1] / U[0], U[2] / U[0]


def test_fast_states_converge(ms):
    bad = []
    with ms.MassiveSolver(8, 8, True, True, 0.8, prec="f64") as sv:
        for s in STATES:
            d, ux, uy = deviations(*s)
            sv.set_state(np.ascontiguousarray(np.broadcast_to(d[:, None, None], (45, 8, 8))))
            got = sv.moments()
            try:
                sv.check()
            except Exception as e:
                bad.append((s, str(e)))
                continue
            assert np.hypot(got[1] - ux, got[2] - uy).max() <= 1e-9
    assert not bad, (len(bad), bad[:2])
