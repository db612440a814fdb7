"""The float32 scalars of the pivoted QRs, on the host and on the device, against
float64: the head and tau of a reflector are the float64 ones rounded once (within
0.501 ulp) wherever that is a finite float, columns of norms up to the square root of the largest float
included, and the near-tie threshold is the smallest float not below the float64
product."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1712_07297_gb300")

SOURCE = """
#include "common.h"
__global__ void kernel(long n, const float* r2, const float* x0, float* out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n;
       i += gridDim.x * (long)blockDim.x) {
    hs::householder_scalars(r2[i], x0[i], out + i, out + n + i);
    out[2 * n + i] = hs::tie_band(r2[i]);
  }
}
extern "C" int run_device(long n, const float* r2, const float* x0, float* out) {
  kernel<<<64, 256>>>(n, r2, x0, out);
  return (int)cudaDeviceSynchronize();
}
extern "C" void run(long n, const float* r2, const float* x0, float* head, float* tau,
                    float* band) {
  for (long i = 0; i < n; i++) {
    hs::householder_scalars(r2[i], x0[i], head + i, tau + i);
    band[i] = hs::tie_band(r2[i]);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("scalars")
    (d / "s.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC", "-gencode",
                    "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I" + os.path.join(PKG, "csrc"), "-I" + os.path.join(ROOT, "include"),
                    "-o", str(d / "s.so"), str(d / "s.cu")], check=True)
    return C.CDLL(str(d / "s.so"), mode=os.RTLD_LAZY)


@pytest.fixture(scope="module", params=["host", pytest.param("device", marks=pytest.mark.gpu)])
def run(request, lib):
    def host(r2, x0):
        lib.run.argtypes = [C.c_long] + [C.c_void_p] * 5
        out = [np.empty_like(r2) for _ in range(3)]
        lib.run(len(r2), r2.ctypes.data, x0.ctypes.data, *[o.ctypes.data for o in out])
        return out

    def device(r2, x0):
        import torch
        if not torch.cuda.is_available():
            pytest.skip("no CUDA device")
        lib.run_device.argtypes = [C.c_long] + [C.c_void_p] * 3
        a, b = torch.from_numpy(r2).cuda(), torch.from_numpy(x0).cuda()
        out = torch.empty(3 * len(r2), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        assert lib.run_device(len(r2), a.data_ptr(), b.data_ptr(), out.data_ptr()) == 0
        return list(out.cpu().numpy().reshape(3, -1))

    return host if request.param == "host" else device


def _columns(lo, hi, n=400_000):
    rng = np.random.default_rng(5)
    r2 = (2.0 ** rng.uniform(lo, hi, n)).astype(np.float32)
    part = np.where(rng.random(n) < 0.3, 2.0 ** rng.uniform(-40, 0, n), rng.random(n))
    x0 = (np.sqrt(r2.astype(np.float64)) * part * rng.choice([-1, 1], n)).astype(np.float32)
    x0[:100] = 0.0
    return r2, x0


@pytest.mark.parametrize("lo,hi", [(-30, 30), (-120, -60), (60, 127.99), (-148, -120)])
def test_reflector_scalars(run, lo, hi):
    r2, x0 = _columns(lo, hi)
    head, tau, _ = run(r2, x0)
    r, x = np.sqrt(r2.astype(np.float64)), x0.astype(np.float64)
    for got, want in ((head, np.where(x >= 0, x + r, x - r)), (tau, 1.0 / (r * (r + np.abs(x))))):
        with np.errstate(over="ignore"):
            w32 = want.astype(np.float32)
        fin = np.isfinite(w32)
        assert np.array_equal(np.isinf(got), ~fin)
        ulp = np.spacing(np.abs(w32[fin])).astype(np.float64)
        err = np.abs(got[fin].astype(np.float64) - want[fin]) / ulp
        # (a tau below the normal floats is rounded twice: once more when scaled)
        bar = np.where(np.abs(want[fin]) < 2.0 ** -126, 0.7505, 0.501)
        assert (err <= bar).all(), (lo, hi, (err - bar).max())
        normal = np.abs(w32[fin]) >= 2.0 ** -126
        assert (got[fin] != w32[fin])[normal].mean() < 1e-4


def test_no_column_and_overflow(run):
    # as the float64 form: no reflector
    r2 = np.array([0, 0, np.inf, np.inf], np.float32)
    x0 = np.array([0, 0, 3, -3], np.float32)
    head, tau, band = run(r2, x0)
    assert head.tolist() == [0, 0, np.inf, -np.inf] and not tau.any()
    assert band.tolist() == [0, 0, np.inf, np.inf]


@pytest.mark.parametrize("lo,hi", [(-90, 127.9)])
def test_tie_threshold(run, lo, hi):
    r2, x0 = _columns(lo, hi)
    band = run(r2, x0)[2].astype(np.float64)
    want = (1.0 - 1e-5) * r2.astype(np.float64)
    below = np.nextafter(band.astype(np.float32), np.float32(0)).astype(np.float64)
    slack = want * 2.0 ** -47
    assert (band >= want - slack).all() and (below < want + slack).all()
