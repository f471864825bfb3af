"""The mixed path's tensor-core transforms of axes of 257 to 512 points (k_dst_long: time stage, y and z
passes) against the CUDA-core ones (ST_DISABLE_TENSOR_CORES=1): lengths on either side of the fold's
padding, odd and even, ragged column tiles, one and several tiles a block, long axes together with
short ones, P_theta with a varying coefficient (its y passes); repeated calls give the same bits."""
import os

import numpy as np
import pytest

from workloads import synthetic as W

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


CASES = [(1, 31, 1, 1, n, "PH") for n in (257, 258, 287, 288, 289, 365, 511, 512)]
CASES += [(1, 1023, 1, 1, 300, "PH"), (2, 127, 31, 1, 400, "PH"), (2, 31, 511, 1, 50, "PH"),
          (2, 127, 511, 1, 16, "PH"), (2, 255, 511, 1, 300, "PH"), (3, 31, 511, 63, 3, "PH"),
          (3, 31, 31, 511, 4, "PH"), (3, 31, 511, 511, 2, "PH"), (2, 31, 511, 1, 60, "Ptheta"),
          (2, 63, 511, 1, 300, "Ptheta")]


# 2e-5: float32 transforms, 22-bit operand split with float32 accumulation
@pytest.mark.parametrize("dim,mx,my,mz,n,prec", CASES)
def test_long_axes_match_cuda_cores(pkg, dim, mx, my, mz, n, prec):
    a = W.random_field(mx, my, 3) if prec == "Ptheta" else None
    spec = pkg.ProblemSpec(dim, mx, my, n, 1.0, "theta", 0.5, a, prec, "mixed", mz=mz)
    v = torch.tensor(np.random.default_rng(n + mx).standard_normal((n, spec.m)), device="cuda")
    s = pkg.Solver(spec)
    z = s.st_apply_prec_f32(v)
    for _ in range(2):
        assert torch.equal(z, s.st_apply_prec_f32(v))
    s.close()
    os.environ["ST_DISABLE_TENSOR_CORES"] = "1"
    try:
        s = pkg.Solver(spec)
    finally:
        del os.environ["ST_DISABLE_TENSOR_CORES"]
    ref = s.st_apply_prec_f32(v).double()
    s.close()
    assert float((z.double() - ref).norm() / ref.norm()) <= 2e-5
