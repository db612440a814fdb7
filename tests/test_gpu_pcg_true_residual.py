"""PCG ends on its recursive residual; the call reports the true one, b - A x.
A tolerance that the true residual can meet must be met: near the rounding level of
b - A x the two differ by more than the step between iterations leaves, and the
solve has to go on from the true residual instead of giving up.

The attainable level here is about u ||A|| ||x|| / ||b||, 3e-15 for 64^2 and 6e-15
for 128^2 (FGMRES, whose restarts use the true residual, reaches both)."""
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    return hsolve


def _rhs(n, seed):
    g = torch.Generator().manual_seed(seed)
    return (torch.rand((128, n), generator=g, dtype=torch.float64) * 2 - 1).cuda()


@pytest.mark.parametrize("side,tol,precision", [(64, 3.5e-15, "fp64"), (128, 1e-14, "fp64"),
                                                (128, 1e-14, "mixed_fp32")])
def test_attainable_tolerance_is_met(hs, side, tol, precision):
    p = I.poisson((side, side))
    s = hs.Solver.from_problem(p, leaf_size=64, symmetric=1)
    s.factor(1e-2, precision)
    for seed in range(3):
        b = _rhs(p.n, seed)
        x, info = s.solve(b, krylov="pcg", tol=tol, maxit=200)
        r = torch.linalg.vector_norm(b - s.spmv(x), dim=1) / torch.linalg.vector_norm(b, dim=1)
        assert float(r.max()) <= tol * (1 + 1e-9) and info.rel_residual <= tol
        assert info.iterations <= 12
    s.close()


def test_unattainable_tolerance_ends_early(hs):
    p = I.poisson((64, 64))
    s = hs.Solver.from_problem(p, leaf_size=64, symmetric=1)
    s.factor(1e-2, "fp64")
    _, info = s.solve(_rhs(p.n, 0), krylov="pcg", tol=1e-17, maxit=200, check=False)
    assert 1e-17 < info.rel_residual < 1e-14 and info.iterations < 40
    with pytest.raises(hs.HsolveError) as e:
        s.solve(_rhs(p.n, 0), krylov="pcg", tol=1e-17, maxit=200)
    assert e.value.code == -6
    s.close()
