"""The gathered products and the Schur update at the edges of their tiles: row
tiles of 1 to 4 strips of 16 (cluster sizes and ranks around 16, 32, 48, 64 and
just above one and two tiles), inner chunks of 32, against the CPU oracle on the
general path (both one-sided products).

Bar: float64 M^{-1} b within 1e-10 of the oracle's (the bar of the parity tests).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402
from oracle import hsolver as H  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [15, 17, 32, 48, 50, 66, 80, 112, 144])
def test_strip_counts(leaf):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    p, eps = I.convection_diffusion((13, 9, 11), 10.0), 1e-3
    fac = H.factor(p.rowptr, p.col, p.val, p.coords, leaf, eps, symmetric=False)
    b = I.rhs(p.n, 1, seed=5)
    ref = H.solve(fac, b.T).T
    s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=0)
    s.factor(eps, "fp64")
    out = s.apply(torch.from_numpy(b).cuda()).cpu().numpy()
    s.close()
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) < 1e-10
