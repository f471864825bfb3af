"""st_autotune's choices are shared by handles that run the same code only: a second handle of the
shape takes them from the cache, one whose stencil or time stage is another kernel is tuned itself."""
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2201_10062_gb300 as P
    from paper_2201_10062_gb300 import build

    build.build()
    P.load_library()
    return P


def _seconds(pkg, mx, my, n, scheme="theta", theta=0.5, varying=False):
    a = 1.0 + 0.1 * np.random.default_rng(1).random((my + 2, mx + 2)) if varying else None
    s = pkg.Solver(pkg.ProblemSpec(2, mx, my, n, 1.0, scheme, theta, a, "PH", "mixed"))
    torch.cuda.synchronize()
    t = time.perf_counter()
    s.st_autotune(reps=20)
    t = time.perf_counter() - t
    s.close()
    return t


# a tuning run launches some 700 kernels of a few microseconds and waits for them, a cached one none
LIMIT = 1e-3


@pytest.mark.parametrize("n,other", [(33, dict(varying=True)), (34, dict(theta=1.0)),
                                     (35, dict(theta=0.3)), (36, dict(scheme="bdf2"))])
def test_another_stencil_is_tuned(pkg, n, other):
    assert _seconds(pkg, 63, 63, n) > LIMIT
    assert min(_seconds(pkg, 63, 63, n) for _ in range(3)) < LIMIT
    assert _seconds(pkg, 63, 63, n, **other) > LIMIT
    assert min(_seconds(pkg, 63, 63, n, **other) for _ in range(3)) < LIMIT


def test_another_time_stage_is_tuned(pkg, monkeypatch):
    """300 steps: k_dst_long, whose handle has no column tile to tune, against the CUDA-core stage."""
    assert _seconds(pkg, 15, 63, 300) > LIMIT
    assert min(_seconds(pkg, 15, 63, 300) for _ in range(3)) < LIMIT
    monkeypatch.setenv("ST_DISABLE_TENSOR_CORES", "1")
    assert _seconds(pkg, 15, 63, 300) > LIMIT
