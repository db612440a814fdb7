"""The substitution sweeps at the edges of their tiling (group widths of the
right-hand sides, ragged cluster sizes, staging in several pieces, the dense
top, clusters beyond the fused kernels) against the CPU oracle.

Bars: float64 within 1e-10 of the oracle's M^{-1} b (both factor in float64;
the bar of the parity tests); float32 within 1e-3 of the same factorization's
one-column applications (sums of at most a few thousand terms of 6e-8 relative
rounding, times the conditioning of the blocks, up to 1 / eps = 100).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402
from oracle import hsolver as H  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    # ragged clusters, small classes
    "poisson2d": (lambda: I.poisson((41, 37)), 60, 1e-3, 0),
    # whole 16-byte columns of 64, more neighbour columns than one piece
    "poisson3d": (lambda: I.poisson((16, 16, 16)), 64, 1e-2, 0),
    # two-sided operators
    "convdiff3d": (lambda: I.convection_diffusion((11, 14, 13), 10.0), 100, 1e-2, 0),
    # dense tops of more unknowns than a tile multiple: Cholesky and LU
    "top_spd": (lambda: I.poisson((16, 16, 16)), 64, 1e-2, 1000),
    "top_lu": (lambda: I.convection_diffusion((14, 14, 14), 10.0), 64, 1e-2, 900),
    # clusters too large for the fused kernels
    "large": (lambda: I.poisson((60, 60)), 900, 1e-3, 0),
}


@pytest.mark.parametrize("name", CASES)
def test_sweep_groups(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    make, leaf, eps, top = CASES[name]
    p = make()
    fac = H.factor(p.rowptr, p.col, p.val, p.coords, leaf, eps, symmetric=p.spd, top_size=top)
    s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=1 if p.spd else 0, top_size=top)
    b = I.rhs(p.n, 41, seed=11)
    ref = H.solve(fac, b.T).T
    bt = torch.from_numpy(b).cuda()
    s.factor(eps, "fp64")
    for nrhs in (1, 2, 4, 5, 8, 9, 16, 41):
        out = s.apply(bt[:nrhs].contiguous()).cpu().numpy()
        err = np.linalg.norm(out - ref[:nrhs]) / np.linalg.norm(ref[:nrhs])
        assert err < 1e-10, (nrhs, err)
    s.factor(eps, "mixed_fp32")
    one = torch.stack([s.apply(bt[c]) for c in range(41)])
    for nrhs in (3, 7, 8, 17, 32, 33, 41):
        out = s.apply(bt[:nrhs].contiguous())
        err = float((out - one[:nrhs]).norm() / one[:nrhs].norm())
        assert err < 1e-3, (nrhs, err)
    s.close()
