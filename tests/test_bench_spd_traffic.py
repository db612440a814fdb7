"""bench.py's roofline on CPU: a phase of a symmetric factorization takes the DRAM
traffic measured over the kernels that it launches, not that of the general path's
kernel of the same phase."""
import glob
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def _figure(key):
    for f in glob.glob(os.path.join(ROOT, "profiles", "*.md")):
        m = re.search(r"^traffic_bytes_per_launch\(%s, poisson3d_128\):\s*(\d+)" % key,
                      open(f).read(), re.M)
        if m:
            return int(m.group(1))
    raise AssertionError(key)


def test_symmetric_phases_have_their_own_figures():
    for phase in ("prep", "qr_cluster", "schur"):
        got = bench._traffic(phase, "poisson3d_128", 16384, 600, spd=True)
        assert got == _figure("spd_" + phase)
        assert got != bench._traffic(phase, "poisson3d_128", 16384, 600)


def test_no_figure_is_borrowed():
    # other workloads, phases without a capture
    assert bench._traffic("prep", "poisson3d_64", 2048, 149, spd=True) is None
    assert bench._traffic("gemm_fill", "poisson3d_128", 16384, 600, spd=True) is None
