"""Dense tops at sizes beside 64 and 128 times powers of two, where the inverse factor's
pairs of blocks (64, float64 Cholesky), the leaves of 128 (float32 Cholesky) and the
LU's panels end: the whole matrix is the top, so M^{-1} b is A^{-1} b.

Bars against scipy's sparse LU: 8 u kappa(A) with kappa <= 4 (s + 1)^2 / pi^2 for a
longest side of s, u = 2^-53 or 2^-24 (convection-diffusion at these sizes is no
worse conditioned than diffusion).
"""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(107, 3), (20, 16), (23, 17), (73, 7), (32, 16), (27, 19), (25, 23), (24, 24), (33, 31),
          (32, 32), (41, 25), (33, 33), (89, 23), (64, 32), (50, 41)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: str(s[0] * s[1]))
@pytest.mark.parametrize("family", ["poisson", "convdiff"])
def test_whole_matrix_as_top(family, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    spd = family == "poisson"
    p = I.poisson(shape) if spd else I.convection_diffusion(shape, 10.0)
    s = hsolve.Solver.from_problem(p, leaf_size=64, symmetric=int(spd), top_size=p.n)
    b = I.rhs(p.n, 9, seed=2)
    ref = sla.splu(p.scipy().tocsc()).solve(b.T).T
    for precision, u in (("fp64", 2.0 ** -53), ("mixed_fp32", 2.0 ** -24)):
        s.factor(1e-2, precision)
        assert s.stats()["top_size"] == p.n
        out = s.apply(torch.from_numpy(b).cuda()).cpu().numpy()
        bar = 8 * u * 4 * (max(shape) + 1) ** 2 / np.pi ** 2
        err = np.linalg.norm(out - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert err.max() < bar, (precision, err.max(), bar)
    s.close()
