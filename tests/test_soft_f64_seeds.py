"""csrc/soft_f64.cuh over the whole range of seeds it is written for, and its device form.

The header's argument needs seeds within 2^-21 of 1/x and 1/sqrt(x).  The device's are specified to 1 unit in the last
place (rcp.approx.ftz.f32) and to a relative error of 2^-22.9 (rsqrt.approx.ftz.f32: up to two units near 1); the
host form takes correctly rounded ones and moves them by up to eight units, 2^-21 and more at every significand.
The device form runs on the GPU over random operands and those at the ends of every range it distinguishes."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from test_soft_f64 import PROGRAM, ROOT

CSRC = os.path.join(ROOT, "paper_1306_6883_gb300", "csrc")
KERNEL = r"""
#include "soft_f64.cuh"
__global__ void run(const double* a, const double* b, double* q, double* r, double* h, double* t, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  q[i] = hydro::soft_div(a[i], b[i]);
  r[i] = hydro::soft_sqrt(a[i]);
  h[i] = hydro::sf_half(a[i]);
  t[i] = hydro::sf_twice(a[i]);
}
extern "C" int soft(const double* a, const double* b, double* q, double* r, double* h, double* t, int n) {
  run<<<(n + 255) / 256, 256>>>(a, b, q, r, h, t, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("ulp", [-8, -5, 5, 8])
def test_integer_pipe_operations_equal_ieee_with_the_worst_seeds(tmp_path, ulp):
    src = tmp_path / "check.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", f"-DSOFT_SEED_ULP={ulp}", f"-DSEED={ulp + 31}",
                    "-I", CSRC, "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def _operands():
    rng = np.random.default_rng(17)
    mant = np.uint64((1 << 52) - 1)
    # exponent fields at the ends of each range the routines distinguish, in every pair, both signs
    exps = np.array([0, 1, 2, 3, 511, 512, 1022, 1023, 1024, 2043, 2044, 2045, 2046, 2047], dtype=np.uint64)
    frac = np.array([0, 1, 2, (1 << 52) - 1, (1 << 52) - 2, 1 << 51, 0x5555555555555], dtype=np.uint64)
    edge = ((exps[:, None] << np.uint64(52)) | frac[None, :]).ravel()
    edge = np.concatenate([edge, edge | np.uint64(1 << 63)])
    a, b = (x.ravel() for x in np.meshgrid(edge, edge))
    # quotients at the ends of the exponent range
    m = 200000
    ea = rng.integers(1, 2047, m).astype(np.uint64)
    gap = rng.choice([-1023, -1022, -1021, -1020, -1019, 1019, 1020, 1021, 1022, 1023], m)
    eb = np.clip(ea.astype(np.int64) - gap, 0, 2047).astype(np.uint64)
    c = [(e << np.uint64(52)) | (rng.integers(0, 1 << 52, m).astype(np.uint64) & mant) for e in (ea, eb)]
    # random bits, near each other, and everyday magnitudes
    d = [rng.integers(0, 1 << 63, 1000000).astype(np.uint64) << np.uint64(1) | np.uint64(1) for _ in range(2)]
    x = rng.standard_normal(1000000) * np.exp(rng.uniform(-20, 20, 1000000))
    y = x * (1 + rng.integers(-8, 9, 1000000) * 2.0 ** -52)
    z = rng.integers(1, 1 << 26, 1000000).astype(np.float64) ** 2  # exact roots
    a = np.concatenate([a, c[0], d[0], x.view(np.uint64), z.view(np.uint64)])
    b = np.concatenate([b, c[1], d[1], y.view(np.uint64), np.abs(x).view(np.uint64)])
    return a.view(np.float64), b.view(np.float64)


@pytest.mark.gpu
def test_the_device_form_equals_ieee(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1306_6883_gb300 import build
    src, lib = tmp_path / "soft.cu", tmp_path / "libsoft.so"
    src.write_text(KERNEL)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-fmad=false", "-shared", "-Xcompiler", "-fPIC",
                    "-I", CSRC, "-o", str(lib), str(src)], check=True)
    a, b = _operands()
    A, B = (torch.from_numpy(v).cuda() for v in (a, b))
    out = [torch.empty_like(A) for _ in range(4)]
    torch.cuda.synchronize()
    fn = ctypes.CDLL(str(lib)).soft
    fn.argtypes = [ctypes.c_void_p] * 6 + [ctypes.c_int]
    assert fn(A.data_ptr(), B.data_ptr(), *[o.data_ptr() for o in out], A.numel()) == 0
    with np.errstate(all="ignore"):
        want = [a / b, np.sqrt(a), 0.5 * a, 2.0 * a]
    for name, got, ref in zip(("division", "square root", "half", "twice"), out, want):
        got = got.cpu().numpy()
        same = (got.view(np.uint64) == ref.view(np.uint64)) | (np.isnan(got) & np.isnan(ref))
        k = np.flatnonzero(~same)
        assert k.size == 0, (name, k.size, a[k[:4]], b[k[:4]], got[k[:4]], ref[k[:4]])
