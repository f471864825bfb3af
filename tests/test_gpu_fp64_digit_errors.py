"""The largest error of the float64 path's digit time stage against that of the CUDA-core double-float
stage (ST_DISABLE_TENSOR_CORES=1), which takes the other time axes, both against the float64 engine.
The coefficient is small, so that the symbol is the time part's alone and nothing hides the
transforms; what the digits leave out must not add up in a few nodes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_10062_gb300 as P
    from paper_2201_10062_gb300 import build

    build.build()
    P.load_library()
    return P


# no tolerance: the largest error is no larger than that of the stage it stands in for
@pytest.mark.parametrize("mx,my", [(31, 15), (127, 63), (127, 255)])
@pytest.mark.parametrize("n", [129, 191, 200, 255, 256])
@pytest.mark.parametrize("scheme,theta", [("theta", 0.5), ("bdf2", 1.0)])
def test_largest_error(pkg, monkeypatch, mx, my, n, scheme, theta):
    spec = pkg.ProblemSpec(2, mx, my, n, 1.0, scheme, theta, np.full((my + 2, mx + 2), 1e-9))
    v = torch.tensor(np.random.default_rng(n + mx).standard_normal((n, spec.m)), device="cuda")

    def apply(**env):
        for k, x in env.items():
            monkeypatch.setenv(k, x)
        s = pkg.Solver(spec)
        for k in env:
            monkeypatch.delenv(k)
        z = s.st_apply_prec(v)
        s.close()
        return z

    ref = apply(ST_FP64_ENGINE="dfma")
    digits, cores = apply(), apply(ST_DISABLE_TENSOR_CORES="1")
    assert not torch.equal(digits, cores)
    assert float((digits - ref).abs().max()) <= float((cores - ref).abs().max())
    assert float((digits - ref).norm()) <= float((cores - ref).norm())
