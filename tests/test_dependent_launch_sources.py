"""Kernels that start before the kernel ahead of them has completed (programmatic
dependent launch) must not promise the compiler that the vectors they read are
read-only: a `const T* __restrict__` parameter may be loaded through the
non-coherent cache, which needs memory that nobody writes while the kernel runs,
and the kernel ahead writes those vectors while this one is running already.
Only what no kernel of the chain writes may carry the promise.  Read from the
sources, since no run shows a stale line reliably."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1712_07297_gb300", "csrc")

# index maps, cluster records, stored operators (sweeps); task lists, blocks,
# column runs, forced pivots and counts (the pivoted QRs of one class)
CONSTANT = {"recs", "ids", "fac", "vmap", "idx", "tasks", "order", "arena", "segs", "fpiv", "cnt"}
WAITS = re.compile(r"pdl_begin\(\)|pdl_wait\(\)|griddepcontrol\.wait")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        txt = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\(((?:[^(){}])*)\)\s*\{", txt):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(txt[i], 0)
                i += 1
            yield os.path.basename(path), m.group(1), m.group(2), txt[m.end():i]


def test_dependent_kernels_read_vectors_coherently():
    waiting = 0
    for path, name, params, body in _kernels():
        if not WAITS.search(body):
            continue
        waiting += 1
        promised = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params)
        assert set(promised) <= CONSTANT, (path, name, promised)
    assert waiting >= 7  # the two sweeps, the two of the dense top, two copies, the QR
