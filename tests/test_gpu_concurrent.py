"""Several solvers at once (GPU): each on its own stream and thread, and taking
turns on one stream.  Steps are chained launches, so a step's blocks may be
placed while other solvers' kernels run; every solver has to give the bits it
gives alone.
"""
import threading

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
    return torch, rlbm, massive


# small FP64 samples (a site shared by warps; two blocks per SM), FP32, FP16, both massive types
KINDS = [("f64", 64, 64), ("f64", 100, 100), ("f32", 200, 150), ("f16dev", 130, 70),
         ("massive_f64", 64, 64), ("massive_f64", 97, 120), ("massive_f32", 90, 50)]


def make(lib, kind, nx, ny, k, stream):
    torch, rlbm, massive = lib
    rng = np.random.default_rng(100 * k + nx)
    f = [1 + 0.01 * rng.uniform(-1, 1, (ny, nx)), 0.02 * rng.uniform(-1, 1, (ny, nx)),
         0.02 * rng.uniform(-1, 1, (ny, nx)), 1 + 0.01 * rng.uniform(-1, 1, (ny, nx))]
    if kind.startswith("massive"):
        sv = massive.MassiveSolver(nx, ny, True, False, 0.8, 1e-5, -1e-5, prec=kind[8:], stream=stream)
        sv.init(*f)
    else:
        sv = rlbm.Solver(W.Sample(nx, ny, periodic_x=True, tau=0.8, Fx=1e-5), prec=kind, stream=stream)
        sv.init(0, *f)
    return sv


def alone(lib, steps):
    torch = lib[0]
    out = []
    for k, kind in enumerate(KINDS):
        with make(lib, *kind, k, torch.cuda.Stream()) as sv:
            sv.step(steps)
            sv.check()
            out.append(sv.get_state())
    return out


def test_solvers_on_their_own_streams_and_threads(lib):
    torch = lib[0]
    want = alone(lib, 60)
    solvers = [make(lib, *kind, k, torch.cuda.Stream()) for k, kind in enumerate(KINDS)]
    start, errors = threading.Barrier(len(solvers)), []

    def work(sv):
        try:
            start.wait()
            for _ in range(6):
                sv.step(10)
        except Exception as e:        # shown by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(sv,)) for sv in solvers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for sv, w in zip(solvers, want):
        sv.check()
        assert np.array_equal(sv.get_state(), w)
        sv.close()


def test_solvers_taking_turns_on_one_stream(lib):
    torch = lib[0]
    want = alone(lib, 12)
    stream = torch.cuda.Stream()
    solvers = [make(lib, *kind, k, stream) for k, kind in enumerate(KINDS)]
    for _ in range(12):
        for sv in solvers:
            sv.step(1)
    for sv, w in zip(solvers, want):
        sv.check()
        assert np.array_equal(sv.get_state(), w)
        sv.close()
