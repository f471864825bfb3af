"""The float64 path's tensor-core time stage (integer digits, k_time_tcd) at the time axes between the
multiples of 32: odd and even n on either side of the fold's padding to 16 rows, ragged column
tiles, several tiles a block; P^-1 v against the CUDA-core double-float stage (ST_DISABLE_TENSOR_CORES=1)
within 1e-12, as at the multiples of 32 (both carry about 2^-41 of a column's largest entry), while
a different kernel ran, and repeated calls give the same bits."""
import os

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


@pytest.mark.parametrize("dim,mx,my", [(1, 31, 1), (2, 31, 15), (2, 127, 63)])
@pytest.mark.parametrize("n", [129, 130, 143, 145, 191, 200, 241, 254, 255])
@pytest.mark.parametrize("scheme,theta", [("theta", 0.5), ("bdf2", 1.0)])
def test_digit_stage_between_multiples_of_32(pkg, dim, mx, my, n, scheme, theta):
    spec = pkg.ProblemSpec(dim, mx, my, n, 1.0, scheme, theta)
    v = torch.tensor(np.random.default_rng(n + mx).standard_normal((n, spec.m)), device="cuda")
    s = pkg.Solver(spec)
    z = s.st_apply_prec(v)
    assert torch.equal(z, s.st_apply_prec(v))
    s.close()
    os.environ["ST_DISABLE_TENSOR_CORES"] = "1"
    try:
        s = pkg.Solver(spec)
    finally:
        del os.environ["ST_DISABLE_TENSOR_CORES"]
    ref = s.st_apply_prec(v)
    s.close()
    assert not torch.equal(z, ref)
    assert float((z - ref).abs().max() / ref.abs().max()) <= 1e-12
