"""The register forms of the float32 pivoted QR at the edges of their ranges
(cluster sizes of 32, 33, 64, 65, 128, 129 unknowns; classes that mix forms)
against the one-CTA form (cluster_qr = 0).

A float32 search may break near-ties of the column norms its own way, so the
ranks and pivot orders of the float64 path are given (hsolve_factor_forced)
and the stored operators compared where they do not depend on a basis choice:
the coarse rows of T' = U^T A_ss^{-1}.  Bar: both forms are within 2 u
kappa(A_ss) r_11 / r_kk of the exact rows (the perturbation bound of the
block-parity tests), with kappa <= 4 m^(2/3) for these Laplacian blocks and
r_11 / r_kk <= 1 / eps, so they differ by at most twice that.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,leaf", [((16, 16, 8), 32), ((11, 12, 8), 33), ((16, 16, 16), 64),
                                        ((13, 20, 16), 65), ((16, 16, 16), 128),
                                        ((20, 20, 20), 129), ((15, 17, 16), 260)])
def test_register_forms(shape, leaf):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    p, eps = I.poisson(shape), 1e-2
    ref = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=1)
    ref.factor(eps, "fp64")
    lv = ref.export_level(0, blocks=False)["clusters"]
    ranks, piv = [[c["k"] for c in lv]], [[list(c["piv"]) for c in lv]]
    got = {}
    for cluster_qr in (1, 0):
        s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=1, cluster_qr=cluster_qr)
        s.factor_forced("mixed_fp32", ranks, piv)
        got[cluster_qr] = s.export_level(0)["clusters"]
        s.close()
    ref.close()
    n = 0
    for a, b in zip(got[1], got[0]):
        assert (a["m"], a["k"], list(a["piv"])) == (b["m"], b["k"], list(b["piv"]))
        if a["T"] is None or a["k"] == 0:
            continue
        k, bound = a["k"], 2 * 2 * 2.0 ** -24 * 4 * a["m"] ** (2 / 3) / eps
        assert np.abs(a["T"][:k] - b["T"][:k]).max() <= bound * np.abs(b["T"][:k]).max()
        n += 1
    assert n > 4
