"""The float64 path's digit time stage over the range of its data: very small vectors (a column's scale
is a power of two that must stay finite)."""
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


# Scaling by a power of two commutes with the map but for the last place of float32's range, 2^-149, in
# the low-order parts: some hundred operations an element, each off by 2^-149 against entries of about
# 2^-112 on the way, make 2^-37 x sqrt(100) < 1e-10 of the result; 1e-9 leaves a factor of ten.
@pytest.mark.parametrize("n", [129, 200, 256])
def test_small_vectors(pkg, n):
    s = pkg.Solver(pkg.ProblemSpec(2, 31, 15, n, 1.0, "theta", 0.5))
    v = torch.tensor(np.random.default_rng(n).standard_normal((n, s.spec.m)), device="cuda")
    ref = s.st_apply_prec(v)
    z = s.st_apply_prec(v * 2.0 ** -112) * 2.0 ** 112
    s.close()
    assert float((z - ref).norm() / ref.norm()) <= 1e-9
