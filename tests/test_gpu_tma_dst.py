"""The tensor-core transforms of the mixed path (any axis length from 16 to 256) against the CUDA-core
ones (shared-memory FFT and FFMA kernels, ST_DISABLE_TENSOR_CORES=1), which the other tests hold
against the oracle: time axes on either side of each tile shape (h = ceil(n/2) up to 32, 64 and 128 folded rows) and of
the MMA's K step, odd lengths, column counts that leave a ragged last tile, several tiles a block, and
spatial axes of every length they take in 1D, 2D and 3D; repeated calls give the same bits."""
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


CASES = [(1, 1023, 1, 1, n) for n in (16, 17, 31, 32, 33, 47, 48, 64, 65, 96, 97, 128, 129, 160, 200,
                                      241, 255, 256)]
CASES += [(1, 31, 1, 1, 100), (2, 31, 63, 1, 65), (2, 63, 31, 1, 30), (2, 127, 127, 1, 40),
          (2, 255, 31, 1, 129), (2, 31, 255, 1, 21), (2, 255, 255, 1, 24), (2, 15, 63, 1, 50),
          (3, 31, 31, 31, 20), (3, 15, 63, 31, 18), (3, 63, 15, 127, 16)]

# sizes at which every axis takes the tensor cores by default (small vectors keep the CUDA cores along
# y, z and, for n < 64, time)
CASES += [(2, 255, 255, 1, n) for n in (16, 17, 31, 33, 48, 63)]
CASES += [(2, 127, 127, 1, 64), (2, 255, 63, 1, 65), (2, 511, 31, 1, 60), (2, 255, 127, 1, 40),
          (3, 31, 31, 31, 32), (3, 31, 63, 127, 16)]


# 2e-5: float32 transforms, 22-bit operand split with float32 accumulation.  (Against float64 the
# symbol's float32 tables add their own error on anisotropic grids, the same in both engines.)
@pytest.mark.parametrize("dim,mx,my,mz,n", CASES)
@pytest.mark.parametrize("scheme,theta", [("theta", 0.5), ("bdf2", 1.0)])
def test_float32_preconditioner_matches_cuda_cores(pkg, dim, mx, my, mz, n, scheme, theta):
    spec = pkg.ProblemSpec(dim, mx, my, n, 1.0, scheme, theta, None, "PH", "mixed", mz=mz)
    v = np.random.default_rng(n + mx).standard_normal((n, spec.m))
    d = torch.tensor(v, device="cuda")
    s = pkg.Solver(spec)
    z = s.st_apply_prec_f32(d)
    for _ in range(2):
        assert torch.equal(z, s.st_apply_prec_f32(d))
    s.close()
    os.environ["ST_DISABLE_TENSOR_CORES"] = "1"
    try:
        s = pkg.Solver(spec)
    finally:
        del os.environ["ST_DISABLE_TENSOR_CORES"]
    ref = s.st_apply_prec_f32(d).double()
    s.close()
    assert float((z.double() - ref).norm() / ref.norm()) <= 2e-5
