"""The autotuner's cache and the single-sample rule (GPU)."""
import json

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


def test_entries_of_other_kernels_are_not_used(rl, tmp_path):
    """A cache written for other kernels (its keys end with the geometry hash,
    without a kernel revision) does not choose the shape; entries of this
    revision do."""
    path = str(tmp_path / "tune.json")
    s = W.Sample(200, 150, tau=0.8, Fx=1e-5)

    def tune():
        with rl.Solver(s, prec="f32", tune_cache=path) as sv:
            sv.init(0)
            return sv.autotune()

    assert tune() == (0, 0, 0)
    (key, entry), = json.load(open(path)).items()
    old = key[:key.index("|h=") + 19]
    json.dump({old: {"bx": 128, "grid": 0, "staged": 0}}, open(path, "w"))
    assert tune() == (0, 0, 0)
    now = json.load(open(path))
    assert now[old] == {"bx": 128, "grid": 0, "staged": 0} and now[key] == entry
    json.dump({key: {"bx": 64, "grid": 0, "staged": 0}}, open(path, "w"))
    assert tune() == (64, 0, 0)
