"""A handle after a call on non-finite data.  A right-hand side with a NaN, an infinity or a value beyond
the float32 range ends a mixed solve with a breakdown; the next call on the same handle, with good data,
gives the same bits as a fresh handle.  (The float32 vectors keep a padding slot behind every x line
that has to read zero; a transform of non-finite data leaves 0 x NaN in it.)

The sizes take every kernel that writes or carries the padding: each tile shape of the x lines (31 to
255), the y pass and the time stage whose 128-column tile stacks two column sets (63 points; at most
64 levels), long axes, 3D, the CUDA-core transforms, and both P_theta maps for a varying a."""
import numpy as np
import pytest

from workloads import synthetic as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BAD = [float("nan"), float("inf"), 1e300]


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_10062_gb300 as P
    from paper_2201_10062_gb300 import build

    build.build()
    P.load_library()
    return P


CASES = [(1, 31, 1, 1, 40, "PH"), (1, 1023, 1, 1, 300, "PH"), (2, 7, 15, 1, 9, "PH"),
         (2, 31, 31, 1, 70, "PH"), (2, 63, 63, 1, 200, "PH"), (2, 127, 63, 1, 100, "PH"),
         (2, 255, 63, 1, 33, "PH"), (2, 255, 127, 1, 64, "PH"), (2, 31, 511, 1, 60, "PH"),
         (2, 127, 31, 1, 300, "PH"), (3, 15, 31, 31, 64, "PH"), (1, 255, 1, 1, 64, "Ptheta"),
         (2, 31, 31, 1, 20, "Ptheta"), (2, 127, 127, 1, 64, "Ptheta"),
         (2, 255, 63, 1, 60, "Ptheta"), (2, 511, 63, 1, 30, "Ptheta"), (3, 63, 31, 15, 30, "Ptheta")]


def _spec(pkg, dim, mx, my, mz, n, prec, precision="mixed"):
    a = None
    if prec == "Ptheta":
        a = {1: lambda: 1.0 + 0.5 * np.sin(np.linspace(0.0, 7.0, mx + 2)),
             2: lambda: W.random_field(mx, my, 3),
             3: lambda: W.random_field_3d(mx, my, mz, 3)}[dim]()
    return pkg.ProblemSpec(dim, mx, my, n, 1.0, "theta", 0.5, a, prec, precision, mz=mz)


def _data(spec, seed=5):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(spec.n, spec.m, generator=g, device="cuda", dtype=torch.float64)


def _with(v, bad):
    w = v.clone()
    w.view(-1)[(7 * w.numel()) // 11] = bad
    return w


@pytest.mark.parametrize("dim,mx,my,mz,n,prec", CASES)
def test_solve_after_breakdown(pkg, dim, mx, my, mz, n, prec):
    spec = _spec(pkg, dim, mx, my, mz, n, prec)
    v = _data(spec)
    kw = dict(tol=1e-8, maxit=40, allow_not_converged=True)
    s = pkg.Solver(spec)
    ref, st_ref = s.st_solve(v, **kw)
    s.close()
    assert torch.isfinite(ref).all()
    s = pkg.Solver(spec)
    for bad in BAD:
        with pytest.raises(pkg.SolverError) as e:
            s.st_solve(_with(v, bad), **kw)
        assert e.value.code == pkg.ST_ERR_BREAKDOWN
        u, st = s.st_solve(v, **kw)
        assert st["iterations"] == st_ref["iterations"]
        assert torch.equal(u, ref)
    s.close()


@pytest.mark.parametrize("dim,mx,my,mz,n,prec", CASES)
def test_float32_preconditioner_after_nonfinite(pkg, dim, mx, my, mz, n, prec):
    spec = _spec(pkg, dim, mx, my, mz, n, prec)
    v = _data(spec)
    s = pkg.Solver(spec)
    ref = s.st_apply_prec_f32(v)
    s.close()
    s = pkg.Solver(spec)
    for bad in BAD:
        assert not torch.isfinite(s.st_apply_prec_f32(_with(v, bad))).all()
        assert torch.equal(s.st_apply_prec_f32(v), ref)
    # the float64 pass shares scratch vectors with the float32 one, in another layout
    s.st_apply_prec(_with(v, float("nan")))
    assert torch.equal(s.st_apply_prec_f32(v), ref)
    u, _ = s.st_solve(v, tol=1e-8, maxit=40, allow_not_converged=True)
    assert torch.isfinite(u).all()
    s.close()


@pytest.mark.parametrize("prec", ["PH", "Ptheta"])
def test_float32_preconditioner_of_a_float64_handle(pkg, prec):
    """Its vectors are not padded and hold what the last float64 call left."""
    spec = _spec(pkg, 2, 63, 31, 1, 40, prec, "fp64")
    v = _data(spec)
    s = pkg.Solver(spec)
    ref = s.st_apply_prec_f32(v)
    s.st_solve(v, tol=1e-8, maxit=40, allow_not_converged=True)
    s.st_apply_prec(_with(v, float("nan")))
    assert torch.equal(s.st_apply_prec_f32(v), ref)
    s.close()


def test_batch_after_one_bad_instance(pkg):
    shapes = [(2, 63, 63, 1, 64, "PH"), (2, 127, 63, 1, 100, "PH"), (2, 255, 63, 1, 40, "PH")]
    specs = [_spec(pkg, *c) for c in shapes]
    data = [_data(sp, i) for i, sp in enumerate(specs)]
    kw = dict(tol=1e-8, maxit=60)
    b = pkg.BatchSolver(specs)
    ref, _ = b.st_solve_batch(data, **kw)
    b.close()
    b = pkg.BatchSolver(specs)
    for i in range(len(specs)):
        for bad in BAD:
            mixed = [_with(v, bad) if j == i else v for j, v in enumerate(data)]
            with pytest.raises(pkg.SolverError) as e:
                b.st_solve_batch(mixed, **kw)
            assert e.value.code == pkg.ST_ERR_BREAKDOWN
            outs, _ = b.st_solve_batch(data, **kw)
            for u, r in zip(outs, ref):
                assert torch.equal(u, r)
    b.close()


@pytest.mark.parametrize("n", [129, 200, 224, 256])
@pytest.mark.parametrize("bad", BAD[:2])
def test_float64_digit_stage_keeps_nonfinite_values(pkg, n, bad):
    """The float64 path's time stage on integer digits, which have no NaN and no infinity: as through
    the CUDA-core stages, one of them reaches the whole result, and ends a solve with a breakdown."""
    spec = _spec(pkg, 2, 63, 31, 1, n, "PH", "fp64")
    v = _data(spec)
    s = pkg.Solver(spec)
    ref = s.st_apply_prec(v)
    assert not torch.isfinite(s.st_apply_prec(_with(v, bad))).any()
    assert torch.equal(s.st_apply_prec(v), ref)
    with pytest.raises(pkg.SolverError) as e:
        s.st_solve(_with(v, bad), tol=1e-8, maxit=40)
    assert e.value.code == pkg.ST_ERR_BREAKDOWN
    s.close()
