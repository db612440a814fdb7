"""The substitution sweeps with many right-hand sides: on both sides of the
sizes where large clusters leave the fused kernels (160 unknowns in float64, 256
in float32, more than 64 right-hand sides), clusters whose forward step is fused
and whose backward step is not, and small dense tops whose clusters of CTAs shrink,
against the CPU oracle.

Bars: float64 within 1e-10 of the oracle's M^{-1} b, column by column; float32
against the same factorization's one-column applications, where only the order of
the sums differs: in the largest element of every column within 8 u kappa(A),
u = 2^-24, kappa <= 4 (s + 1)^2 / pi^2 for a longest side of s.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402
from oracle import hsolver as H  # noqa: E402

pytestmark = pytest.mark.gpu

# shape, leaf size, top_size: clusters of exactly 160, 162, 250, 256 and 264
CASES = {
    "m160": ((16, 20, 16), 160, 0),
    "m162": ((18, 18, 16), 162, 0),
    "m250": ((50, 40), 250, 0),
    "m256": ((16, 16, 16), 256, 0),
    "m264": ((33, 16, 8), 264, 0),
    "top272": ((17, 16), 64, 272),
    "top400": ((20, 20), 64, 400),
    "top1000": ((10, 10, 10), 64, 1000),
}


@pytest.mark.parametrize("family", ["poisson", "convdiff"])
@pytest.mark.parametrize("name", CASES)
def test_many_right_hand_sides(name, family):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    shape, leaf, top = CASES[name]
    spd, eps = family == "poisson", 1e-2
    p = I.poisson(shape) if spd else I.convection_diffusion(shape, 10.0)
    fac = H.factor(p.rowptr, p.col, p.val, p.coords, leaf, eps, symmetric=spd, top_size=top)
    s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=int(spd), top_size=top)
    b = I.rhs(p.n, 300, seed=17)
    ref = H.solve(fac, b.T).T
    bt = torch.from_numpy(b).cuda()
    s.factor(eps, "fp64")
    if top == 0:
        assert set(s.level(0)[0].tolist()) == {leaf}
    for nrhs in (8, 64, 65, 129, 300):
        out = s.apply(bt[:nrhs].contiguous()).cpu().numpy()
        err = np.linalg.norm(out - ref[:nrhs], axis=1) / np.linalg.norm(ref[:nrhs], axis=1)
        assert err.max() < 1e-10, (nrhs, int(err.argmax()), err.max())
    s.factor(eps, "mixed_fp32")
    one = torch.stack([s.apply(bt[c]) for c in range(300)])
    bar = 8 * 2.0 ** -24 * 4 * (max(shape) + 1) ** 2 / np.pi ** 2
    for nrhs in (3, 8, 31, 64, 65, 129, 300):
        out = s.apply(bt[:nrhs].contiguous())
        err = (out - one[:nrhs]).abs().amax(1) / one[:nrhs].abs().amax(1)
        assert float(err.max()) < bar, (nrhs, int(err.argmax()), float(err.max()))
    s.close()
