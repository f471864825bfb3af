"""The double-float stencil (two x neighbours a thread) at the edges of its walk: the shortest and
longest lines, one level, the middle level of an odd n, chunks of one level, every scheme, uniform
and varying coefficients in 1D, 2D and 3D.

An inner MINRES run of a mixed solve ends at an estimate of at most 1e-7 and the float64 residual
decides, so four refinement steps reach 1e-8 when the inner operator is the true one; an
operator with a wrong node, level or coefficient leaves an error of its own size, which no number of
steps below the limit removes."""
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


GRIDS = [(1, 3, 1, 1, 5), (1, 1023, 1, 1, 65), (2, 3, 7, 1, 1), (2, 7, 3, 1, 2), (2, 15, 15, 1, 3),
         (2, 31, 63, 1, 8), (2, 127, 31, 1, 33), (3, 3, 7, 15, 4), (3, 15, 7, 3, 1),
         (3, 63, 15, 7, 7)]


@pytest.mark.parametrize("dim,mx,my,mz,n", GRIDS)
@pytest.mark.parametrize("scheme,theta", [("theta", 1.0), ("theta", 0.5), ("theta", 0.7),
                                          ("bdf2", 1.0)])
@pytest.mark.parametrize("coef", ["uniform", "general", "field"])
def test_refinement_reaches_the_float64_residual(pkg, monkeypatch, dim, mx, my, mz, n, scheme,
                                                 theta, coef):
    if coef == "general":
        monkeypatch.setenv("ST_STENCIL_GENERAL", "1")
    w = W.small_case(dim, mx, my, n, scheme, theta, coef == "field", seed=mx + n, mz=mz)
    s = pkg.Solver(pkg.ProblemSpec(dim, mx, my, n, w.T, scheme, theta, w.a_nodal, "PH", "mixed",
                                   mz=mz))
    f = torch.tensor(w.f, device="cuda")
    fH = s.st_assemble_rhs(f, torch.tensor(w.u0, device="cuda"),
                           None if w.u_prev is None else torch.tensor(w.u_prev, device="cuda"))
    u, st = s.st_solve(fH, tol=1e-8)
    y = s.st_apply_op(u.reshape(n, -1)).reshape(-1)
    r = torch.flip(fH.reshape(n, -1), (0,)).reshape(-1) - y
    s.close()
    assert float(r.norm() / fH.norm()) <= 1.01e-8
    assert st["outer_steps"] <= 4
