"""P_theta with a varying coefficient: the x passes of the inner map on the tensor cores, with the diagonal
scaling as a pass of its own, against the CUDA-core passes that scale as they load
(ST_DISABLE_TENSOR_CORES=1): every tile shape of the x lines, 2D and 3D, one to three inner steps, sizes
just above the line from which the tensor cores are taken."""
import os

import numpy as np
import pytest

from workloads import synthetic as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# 2e-5: float32 transforms, 22-bit operand split with float32 accumulation
@pytest.mark.parametrize("dim,mx,my,mz,n", [(2, 63, 63, 1, 200), (2, 31, 255, 1, 100),
                                            (2, 127, 31, 1, 201), (2, 255, 127, 1, 31),
                                            (3, 31, 63, 15, 30), (3, 63, 7, 31, 61)])
@pytest.mark.parametrize("degree", [1, 2, 3])
def test_ptheta_matches_cuda_cores(dim, mx, my, mz, n, degree):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_10062_gb300 as P
    from paper_2201_10062_gb300 import build

    build.build()
    P.load_library()
    a = W.random_field(mx, my, 3) if dim == 2 else W.random_field_3d(mx, my, mz, 3)
    spec = P.ProblemSpec(dim, mx, my, n, 1.0, "theta", 0.5, a, "Ptheta", "mixed", mz=mz,
                         inner_degree=degree)
    v = torch.tensor(np.random.default_rng(n + mx).standard_normal((n, spec.m)), device="cuda")
    s = P.Solver(spec)
    z = s.st_apply_prec_f32(v)
    assert torch.equal(z, s.st_apply_prec_f32(v))
    s.close()
    os.environ["ST_DISABLE_TENSOR_CORES"] = "1"
    try:
        s = P.Solver(spec)
    finally:
        del os.environ["ST_DISABLE_TENSOR_CORES"]
    ref = s.st_apply_prec_f32(v).double()
    s.close()
    assert float((z.double() - ref).norm() / ref.norm()) <= 2e-5
