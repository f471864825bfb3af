"""Tensor-core transforms of the mixed path one axis at a time: sizes at which only the named axis leaves
the CUDA cores, so that the results must differ from those of ST_DISABLE_TENSOR_CORES=1 by rounding, and
by no more than rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# x: few unknowns and steps; y and z: x lines too long, too few steps; time: the other axes too short
# or too long
CASES = [(2, mx, 7, 1, 20) for mx in (31, 63, 127, 255)] + [(1, 255, 1, 1, 9), (3, 63, 15, 7, 15)]
CASES += [(3, 511, 31, 7, 15), (2, 1023, 63, 1, 15), (2, 511, 127, 1, 15), (2, 511, 255, 1, 9),
          (2, 511, 511, 1, 7)]
CASES += [(3, 511, 7, mz, 15) for mz in (31, 63, 127, 255, 511)]
CASES += [(3, 1023, 7, 7, n) for n in (16, 17, 31, 32, 33, 47, 48, 63)]
CASES += [(1, 1023, 1, 1, n) for n in (64, 65, 96, 127, 129, 193, 256, 257, 288, 289, 481, 512)]


@pytest.fixture(scope="module")
def pkg():
    import paper_2201_10062_gb300 as P
    from paper_2201_10062_gb300 import build

    build.build()
    P.load_library()
    return P


# A transform on the tensor cores cuts at most four sums by half an ulp on average (2.4e-7 of the
# result) and drops a product of 2^-24; the float32 kernels round each of their sums: 6e-7 a transform
# for the two together, two transforms along each axis.
@pytest.mark.parametrize("dim,mx,my,mz,n", CASES)
def test_one_axis_on_the_tensor_cores(pkg, monkeypatch, dim, mx, my, mz, n):
    spec = pkg.ProblemSpec(dim, mx, my, n, 1.0, "theta", 0.5, None, "PH", "mixed", mz=mz)
    v = torch.tensor(np.random.default_rng(n + mx).standard_normal((n, spec.m)), device="cuda")
    z = []
    for off in ("0", "1"):
        monkeypatch.setenv("ST_DISABLE_TENSOR_CORES", off)
        s = pkg.Solver(spec)
        z.append(s.st_apply_prec_f32(v).double())
        s.close()
    assert not torch.equal(z[0], z[1])
    assert float((z[0] - z[1]).norm() / z[1].norm()) <= 6e-7 * 2 * (dim + 1)


@pytest.mark.parametrize("dim,mx,my,mz,n,precision", [(2, 63, 31, 1, 40, "mixed"), (1, 255, 1, 1, 300, "mixed"),
                                                      (2, 31, 511, 1, 60, "mixed"), (2, 63, 31, 1, 40, "fp64")])
def test_solve_host_gives_the_device_solution(pkg, dim, mx, my, mz, n, precision):
    """st_solve_host keeps the iterate in a vector of the handle (mixed: the stencil output)."""
    spec = pkg.ProblemSpec(dim, mx, my, n, 1.0, "theta", 0.5, None, "PH", precision, mz=mz)
    v = torch.tensor(np.random.default_rng(n).standard_normal((n, spec.m)), device="cuda")
    s = pkg.Solver(spec)
    u, st = s.st_solve(v, tol=1e-9)
    assert st["outer_steps"] > 1 or precision == "fp64"  # several inner runs reuse that vector
    h = np.empty((n, spec.m))
    s.st_solve_host(v.cpu().numpy(), h, tol=1e-9)
    assert np.array_equal(h, u.cpu().numpy().reshape(n, -1))
    s.close()
