"""Float64 ranks on the Cholesky path for clusters of a few unknowns (leaf sizes 2 to
30), against the CPU oracle.

The ranks equal the oracle's wherever the matrix determines them.  It does not
everywhere: a fill block that is zero in exact arithmetic holds rounding noise, and
where conditioning lifts that noise above the noise floor its rank follows from the
last bits.  (37 x 35, clusters of 5) and (29 x 29, clusters of 3) are such inputs:
the oracle's own ranks change when entries of the matrix change by one unit in the
last place, or with the machine.  There the ranks must be the oracle's for the matrix
or for one of 40 such perturbations.  Either way M^{-1} b is within 1e-10 of that
oracle's (the bar of the parity tests; the perturbation itself moves it by 2^-52
kappa, 2e-13).
"""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402
from oracle import hsolver as H  # noqa: E402

pytestmark = pytest.mark.gpu


def _perturbed(p, seed):
    """Entries scaled by 1 + {-1, 0, 1} 2^-52, the same for (i, j) and (j, i)."""
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    key = np.minimum(rows, p.col).astype(np.int64) * p.n + np.maximum(rows, p.col)
    u, at = np.unique(key, return_inverse=True)
    step = np.random.default_rng(seed).integers(-1, 2, len(u))
    return p.val * (1 + 2.0 ** -52 * step)[at]


def _oracle(p, val, leaf, eps, b):
    fac = H.factor(p.rowptr, p.col, val, p.coords, leaf, eps, symmetric=True)
    ranks = [[lv.factors[i].k if i in lv.factors else 0 for i in range(lv.nclu)]
             for lv in fac.levels if lv.top is None]
    return ranks, H.solve(fac, b.T).T


CASES = [((24, 24), leaf, 1e-3, False) for leaf in (2, 5, 9, 18, 30)] + \
        [((30, 31), leaf, 1e-4, False) for leaf in (4, 8, 15, 30)] + \
        [((9, 10, 11), leaf, 1e-3, False) for leaf in (2, 4, 8, 16, 31)] + \
        [((37, 35), 10, 1e-3, True), ((29, 29), 4, 1e-4, True)]


@pytest.mark.parametrize("shape,leaf,eps,tie", CASES)
def test_ranks_of_small_clusters(shape, leaf, eps, tie):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    p = I.poisson(shape)
    b = I.rhs(p.n, 1, seed=3)
    want, ref = _oracle(p, p.val, leaf, eps, b)
    s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=1)
    s.factor(eps, "fp64")
    got = [s.level(li)[1].tolist() for li in range(len(want))]
    out = s.apply(torch.from_numpy(b).cuda()).cpu().numpy()
    s.close()
    for seed in range(40 if tie else 0):
        if got == want:
            break
        want, ref = _oracle(p, _perturbed(p, seed), leaf, eps, b)
    assert got == want
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) < 1e-10
