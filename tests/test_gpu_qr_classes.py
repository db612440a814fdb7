"""Colour classes whose pivoted QRs do not share one launch (float32, Cholesky path),
and the widest register forms, against the one-CTA form (cluster_qr = 0): several
cluster sizes of CTAs in one class, register forms beside the shared-memory one
(clusters of 256 and 257 unknowns; fill blocks too wide for any form), 16 CTAs.

The ranks and pivot orders of the float64 path are given on every level, since a
float32 search may break near-ties its own way.  Bars: the coarse rows of level 0,
U^T A_ss^{-1}, as in test_gpu_qr_forms.py (each form within 2 u kappa r_11 / r_kk,
kappa <= 4 m^(2/dim), r_11 / r_kk <= 1 / eps); M^{-1} b, which holds every level,
within 2 x 8 u kappa(A), u = 2^-24, kappa(A) <= 4 (s + 1)^2 / pi^2 for a side of s.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
# shape, leaf, eps, level whose classes launch several groups, level with fill
# blocks of more than 1,024 columns on clusters of more than 128 unknowns
CASES = [((57, 72), 257, 1e-2, 0, None), ((40, 40, 40), 32, 1e-2, 1, None),
         ((32, 32, 32), 256, 1e-3, None, 1), ((40, 40, 40), 128, 1e-3, 1, 1)]


@pytest.mark.parametrize("shape,leaf,eps,several,wide", CASES)
def test_classes_of_several_launches(shape, leaf, eps, several, wide):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    p = I.poisson(shape)
    ref = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=1)
    ref.factor(eps, "fp64")
    lv = [ref.export_level(li, blocks=False) for li in range(ref.stats()["levels"])]
    ref.close()
    lv = [v["clusters"] for v in lv if not v["dense_top"]]
    ranks = [[c["k"] for c in v] for v in lv]
    piv = [[list(c["piv"]) for c in v] for v in lv]
    if wide is not None:
        assert any(128 < c["m"] <= 256 and max(c["piv"], default=0) >= 1024 for c in lv[wide])
    b = torch.from_numpy(I.rhs(p.n, 2, seed=9)).cuda()
    got, out = {}, {}
    for cluster_qr in (1, 0):
        s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=1, cluster_qr=cluster_qr)
        s.set_profiling(True, per_level=True)
        s.factor_forced("mixed_fp32", ranks, piv)
        if cluster_qr and several is not None:
            t = s.phase_times()
            assert t[f"qr_cluster.L{several}"][1] > t[f"count_nz.L{several}"][1]
        s.set_profiling(False)
        got[cluster_qr] = [s.export_level(0)["clusters"]] + [
            s.export_level(li, blocks=False)["clusters"] for li in range(1, len(lv))]
        out[cluster_qr] = s.apply(b)
        s.close()
    for la, lb in zip(got[1], got[0]):
        for x, y in zip(la, lb):
            assert (x["m"], x["k"], list(x["piv"])) == (y["m"], y["k"], list(y["piv"]))
    for x, y in zip(got[1][0], got[0][0]):
        if x["T"] is None or x["k"] == 0:
            continue
        k, bound = x["k"], 2 * 2 * U * 4 * x["m"] ** (2 / len(shape)) / eps
        assert np.abs(x["T"][:k] - y["T"][:k]).max() <= bound * np.abs(y["T"][:k]).max()
    bar = 2 * 8 * U * 4 * (max(shape) + 1) ** 2 / np.pi ** 2
    assert float((out[1] - out[0]).norm() / out[0].norm()) < bar
