"""Profiling of a factorization: the per-cluster step reports its checkpoints on the
Cholesky path (its own kernel up to 256 unknowns, the general one above) as on the
LU path, and they add up to the step's time: each is the slowest cluster's of its
class at the maximum clock, so the sum lies near the launches' time, here between
half and one and a half of it for clusters whose work outweighs a launch."""
import pytest

torch = pytest.importorskip("torch")

from paper_1712_07297_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

NAMES = ("chol", "inverse", "complement", "T_C", "F_tail")


@pytest.mark.parametrize("family,shape,leaf", [("poisson", (24, 24, 24), 128),
                                               ("poisson", (60, 40), 300),
                                               ("convdiff", (24, 24, 24), 128)])
@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
def test_per_cluster_checkpoints(family, shape, leaf, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1712_07297_gb300 import build
    build.build()
    from paper_1712_07297_gb300 import hsolve
    spd = family == "poisson"
    p = I.poisson(shape) if spd else I.convection_diffusion(shape, 10.0)
    s = hsolve.Solver.from_problem(p, leaf_size=leaf, symmetric=int(spd))
    s.factor(1e-2, precision)
    s.set_profiling(True, per_level=True)
    s.factor(1e-2, precision)
    t = s.phase_times()
    s.close()
    # (the LU path has no checkpoint before its last products)
    names = NAMES if spd else ("chol", "inverse", "complement", "T_C")
    for n in names:
        assert t[f"prep.{n}.L0"][0] > 0.0, n
    total = sum(v[0] for k, v in t.items() if k.startswith("prep.") and k.endswith(".L0")
                and k != "prep.L0")
    assert 0.5 * t["prep.L0"][0] < total < 1.5 * t["prep.L0"][0]
