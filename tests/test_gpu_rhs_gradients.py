"""The right-hand-side and gradient kernels walk the time levels in chunks (16 levels a thread; the
face gradients in as many chunks as fill the chip, summed in order): levels on either side of a
chunk's edge, a single level, odd counts, 1D and 2D, with and without an extra term, against the
oracle."""
import numpy as np
import pytest

from oracle import heat as H
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


def _d(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


# every output entry is a sum of at most 2 n + 10 products: 1e-13 is 450 units of 2^-52, above
# n = 200 terms of random sign with room for the oracle's own rounding
@pytest.mark.parametrize("dim,mx,my", [(1, 63, 1), (1, 7, 1), (2, 15, 31), (2, 63, 3)])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 33, 200])
@pytest.mark.parametrize("scheme,theta", [("theta", 1.0), ("theta", 0.3), ("bdf2", 1.0)])
def test_rhs_and_gradients_match_oracle(pkg, dim, mx, my, n, scheme, theta):
    w = W.small_case(dim, mx, my, n, scheme=scheme, theta=theta, varcoef=True, seed=n + mx)
    p = H.Problem.from_workload(w)
    s = pkg.Solver(pkg.ProblemSpec(dim, mx, my, n, w.T, scheme, theta, w.a_nodal))
    r = np.random.default_rng(n)
    lam, u, extra = (r.standard_normal((n, p.m)) for _ in range(3))
    up = None if w.u_prev is None else _d(w.u_prev)
    ref = H.rhs(p, w.f, w.u0, w.u_prev)

    def rel(x, y):
        x = x.cpu().numpy().reshape(y.shape)
        return float(np.linalg.norm(x - y) / max(np.linalg.norm(y), 1e-300))

    assert rel(s.st_assemble_rhs(_d(w.f), _d(w.u0), up), ref) <= 1e-13
    assert rel(s.st_assemble_rhs(_d(w.f), _d(w.u0), up, _d(extra)), ref + extra) <= 1e-13
    gf, gu0, ga = H.adjoint_gradients(p, u, lam, w.u0)
    f_, u0_, up_ = s.st_grad_rhs(_d(lam))
    assert rel(f_, gf) <= 1e-13
    if scheme == "theta":
        assert rel(u0_, gu0) <= 1e-13
    else:  # u^(-1) is a separate input of the library
        assert rel(u0_, 2 * lam[0] - (0.5 * lam[1] if n > 1 else 0.0)) <= 1e-13
        assert rel(up_, -0.5 * lam[0]) <= 1e-13
    assert rel(s.st_grad_a(_d(lam), _d(u), _d(w.u0)), ga) <= 1e-12  # differences cancel
    s.close()
