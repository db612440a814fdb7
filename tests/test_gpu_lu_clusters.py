"""The general (LU, two-sided) per-cluster kernel at the edges of its register
tiles (cluster sizes from 1 to 300 unknowns, triangular inverses in registers up
to 256), against the CPU oracle.

Bars: float64 M^{-1} b within 1e-10 of the oracle's (the bar of the parity
tests); float32 GMRES solves to 1e-10 of ||b||, recomputed in float64.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402
from oracle import hsolver as H  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [1, 31, 33, 64, 97, 130, 256, 300])
@pytest.mark.parametrize("shape", [(37, 35), (11, 10, 12)])
def test_cluster_sizes(shape, leaf):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if leaf == 1:
        shape = (5, 4, 6) if len(shape) == 3 else (11, 12)
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    p, eps = I.convection_diffusion(shape, 10.0), 1e-3
    fac = H.factor(p.rowptr, p.col, p.val, p.coords, leaf, eps, symmetric=False)
    b = I.rhs(p.n, 2, seed=3)
    ref = H.solve(fac, b.T).T
    s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=0)
    bt = torch.from_numpy(b).cuda()
    s.factor(eps, "fp64")
    out = s.apply(bt).cpu().numpy()
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) < 1e-10
    s.factor(eps, "mixed_fp32")
    x, info = s.solve(bt, krylov="gmres", tol=1e-10)
    r = p.scipy() @ x.cpu().numpy().T - b.T
    assert np.linalg.norm(r) / np.linalg.norm(b) < 1e-10 * np.sqrt(2) * 1.01
    s.close()
