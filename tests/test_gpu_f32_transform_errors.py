"""Tensor-core transforms of the mixed path (fp16 operand pairs, accumulators that cut off instead of
rounding): the float32 preconditioner's error against float64, along each axis they take, is no
larger than that of the float32 CUDA-core kernels.

Both kinds round every value once a transform and add up to a few hundred products in float32; an
accumulator that takes all of an axis' K steps loses half an ulp a step, all in one direction, and was
two to five times as far off on the cases below.  Sizes where the float32 symbol tables hide the
transforms' own error (two and three space axes with large eigenvalues) are left to the time axis."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

# 1D: x lines of 1023 points stay on the CUDA cores, so only the time axis differs
CASES = [(1, 1023, 1, 1, n) for n in (127, 200, 243, 255, 256, 257, 365, 500, 512)]
CASES += [(2, 127, 63, 1, 300), (2, 127, 63, 1, 500), (2, 255, 63, 1, 256)]


@pytest.fixture(scope="module")
def pkg():
    import paper_2201_10062_gb300 as P
    from paper_2201_10062_gb300 import build

    build.build()
    P.load_library()
    return P


def _apply(pkg, case, scheme, theta, precision, v, f32):
    dim, mx, my, mz, n = case
    s = pkg.Solver(pkg.ProblemSpec(dim, mx, my, n, 1.0, scheme, theta, None, "PH", precision, mz=mz))
    z = s.st_apply_prec_f32(v).double() if f32 else s.st_apply_prec(v)
    s.close()
    return z


@pytest.mark.parametrize("dim,mx,my,mz,n", CASES)
def test_error_against_float64(pkg, monkeypatch, dim, mx, my, mz, n):
    case = (dim, mx, my, mz, n)
    g = torch.Generator(device="cuda").manual_seed(11)
    tc2 = cc2 = 0.0
    for scheme, theta in (("theta", 0.5), ("theta", 1.0), ("bdf2", 1.0)):
        for smooth in (False, True):
            v = torch.randn(n, mx * my * mz, generator=g, device="cuda", dtype=torch.float64)
            if smooth:
                x = torch.arange(1, mx + 1, device="cuda", dtype=torch.float64) / (mx + 1)
                b = torch.sin(math.pi * x)
                if dim == 2:
                    y = torch.arange(1, my + 1, device="cuda", dtype=torch.float64) / (my + 1)
                    b = (torch.sin(math.pi * y)[:, None] * b).reshape(-1)
                t = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) / n
                v = torch.exp(t)[:, None] * b + 1e-3 * v
            ref = _apply(pkg, case, scheme, theta, "fp64", v, False)
            monkeypatch.delenv("ST_DISABLE_TENSOR_CORES", raising=False)
            tc = _apply(pkg, case, scheme, theta, "mixed", v, True)
            monkeypatch.setenv("ST_DISABLE_TENSOR_CORES", "1")
            cc = _apply(pkg, case, scheme, theta, "mixed", v, True)
            monkeypatch.delenv("ST_DISABLE_TENSOR_CORES")
            assert not torch.equal(tc, cc)  # the tensor cores were used
            tc2 += float(((tc - ref).norm() / ref.norm()) ** 2)
            cc2 += float(((cc - ref).norm() / ref.norm()) ** 2)
    # no larger in the mean square; 1.25: the spread of one set of inputs (a sixth) and a margin
    assert math.sqrt(tc2) <= 1.25 * math.sqrt(cc2)
