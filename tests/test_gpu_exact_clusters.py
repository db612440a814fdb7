"""The per-cluster kernels, Cholesky and LU, and the gathered products at exact
cluster sizes: around the blocks of 32, the register tiles, the row strips of 16 and
the limit of 256 unknowns, and where the operands of the general kernel leave shared
memory (float32: one of the three from 133 unknowns, the second from 163, the last
from 230), against the CPU oracle.  A grid of m 2^d unknowns bisects into clusters
of exactly m, which the test asserts.

Bars: float64 ranks equal (Cholesky) and M^{-1} b within 1e-10 of the oracle's,
the bar of the parity tests; float32 at the oracle's ranks within 8 u kappa(A) of
it, u = 2^-24, kappa <= 4 (s + 1)^2 / pi^2 for a longest side of s (first-order
rounding of a solve with A, a few such per level).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402
from oracle import hsolver as H  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [((16, 32), 16), ((17, 32), 17), ((48, 32), 48), ((49, 32), 49), ((31, 32), 31),
         ((32, 32), 32), ((33, 32), 33), ((64, 32), 64), ((65, 32), 65), ((97, 32), 97),
         ((127, 16), 127), ((64, 32), 128), ((16, 16, 8), 128), ((129, 16), 129),
         ((133, 16), 133), ((163, 16), 163), ((230, 8), 230), ((255, 8), 255), ((64, 32), 256),
         ((16, 16, 8), 256), ((257, 8), 257), ((60, 40), 300)]


@pytest.mark.parametrize("shape,m", SIZES, ids=["x".join(map(str, s)) + f"-{m}" for s, m in SIZES])
@pytest.mark.parametrize("family", ["poisson", "convdiff"])
def test_exact_sizes(family, shape, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    spd, eps = family == "poisson", 1e-3
    p = I.poisson(shape) if spd else I.convection_diffusion(shape, 10.0)
    fac = H.factor(p.rowptr, p.col, p.val, p.coords, m, eps, symmetric=spd)
    b = I.rhs(p.n, 2, seed=3)
    ref = H.solve(fac, b.T).T
    s = hsolve.Solver.from_problem(p, leaf_size=m, symmetric=int(spd))
    bt = torch.from_numpy(b).cuda()
    s.factor(eps, "fp64")
    sizes, ranks, _ = s.level(0)
    assert set(sizes.tolist()) == {m}
    want = [[lv.factors[i].k if i in lv.factors else 0 for i in range(lv.nclu)]
            for lv in fac.levels if lv.top is None]
    if spd:
        for li, w in enumerate(want):
            assert list(s.level(li)[1]) == w, li
    if m == 300:
        assert 0 < ranks.max() < 300 - 256  # fine blocks beyond 256 as well
    out = s.apply(bt).cpu().numpy()
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) < 1e-10
    s.factor_forced("mixed_fp32", want)
    out = s.apply(bt).cpu().numpy()
    s.close()
    bar = 8 * 2.0 ** -24 * 4 * (max(shape) + 1) ** 2 / np.pi ** 2
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) < bar
