"""The FP32/FP64 conversions on the integer pipes (csrc/common.cuh, wide64 and narrow32) and the
quotient by a two-part inverse (csrc/point.cuh, pt_quot) against the plain operations, bit for bit:
ties, subnormal numbers, both ends of the range, infinities and NaN. The device functions are
compiled into a small library of their own."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1302_3663_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "common.cuh"
#include "point.cuh"
__global__ void k_wide(const float* a, double* o, int n) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x)
    o[q] = bf::wide64(a[q]);
}
__global__ void k_narrow(const double* a, float* o, int n) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x)
    o[q] = bf::narrow32(a[q]);
}
__global__ void k_quot(const double* a, const double* b, double* o, int n) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const double hi = 1.0 / b[q];
    o[q] = bf::pt_quot(a[q], hi, bf::pt_low(b[q], hi));
  }
}
extern "C" void run(int which, const void* a, const void* b, void* o, int n) {
  if (which == 0) k_wide<<<152, 256>>>((const float*)a, (double*)o, n);
  else if (which == 1) k_narrow<<<152, 256>>>((const double*)a, (float*)o, n);
  else k_quot<<<152, 256>>>((const double*)a, (const double*)b, (double*)o, n);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    d = tmp_path_factory.mktemp("device_math")
    src, lib = os.path.join(d, "math.cu"), os.path.join(d, "libmath.so")
    open(src, "w").write(SOURCE)
    subprocess.run([B.nvcc()] + B.ARCH + B.NVCC_FLAGS + ["-I", B.CSRC, "-shared", "-o", lib, src],
                   check=True)
    f = ctypes.CDLL(lib).run

    def call(which, a, b=None):
        t = [torch.from_numpy(v).cuda() if v is not None else None for v in (a, b)]
        o = torch.empty(a.size, dtype=torch.float32 if which == 1 else torch.float64, device="cuda")
        torch.cuda.synchronize()
        f(which, ctypes.c_void_p(t[0].data_ptr()),
          ctypes.c_void_p(t[1].data_ptr() if b is not None else 0), ctypes.c_void_p(o.data_ptr()),
          a.size)
        torch.cuda.synchronize()
        return o.cpu().numpy()
    return call


def same(got, want):
    n = np.isnan(want)
    assert np.array_equal(np.isnan(got), n)
    i = np.int32 if got.dtype == np.float32 else np.int64
    bad = (got.view(i) != want.view(i)) & ~n
    assert not bad.any(), (got[bad][:4], want[bad][:4])


def floats():
    rng = np.random.default_rng(1)
    bits = np.concatenate([rng.integers(0, 2 ** 32, 1 << 20, dtype=np.uint64).astype(np.uint32),
                           (np.arange(512, dtype=np.uint32) << 23).repeat(3) +
                           np.tile(np.array([0, 1, 0x7fffff], np.uint32), 512)])
    return bits.view(np.float32)


def test_widening_is_exact(run):
    a = floats()
    same(run(0, a), a.astype(np.float64))


def test_narrowing_rounds_to_nearest_even(run):
    rng = np.random.default_rng(2)
    f = floats()
    f = f[np.isfinite(f)].astype(np.float64)
    up = np.nextafter(f.astype(np.float32), np.float32(np.inf)).astype(np.float64)
    tie = 0.5 * (f + np.where(np.isfinite(up), up, f))   # exact in FP64
    near = [tie, np.nextafter(tie, np.inf), np.nextafter(tie, -np.inf), f,
            f * (1 + rng.uniform(-1e-7, 1e-7, f.size))]
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -149, 2.0 ** -150, 1.5 * 2.0 ** -150,
                     2.0 ** -126, 2.0 ** -1074, 3.4028235677973366e38, 3.4028235677973362e38, 1e300])
    a = np.concatenate(near + [edge, -edge, 10.0 ** rng.uniform(-320, 308, 1 << 18)])
    with np.errstate(over="ignore", under="ignore"):
        same(run(1, a), a.astype(np.float32))


def test_quotients_round_as_a_division(run):
    rng = np.random.default_rng(3)
    n = 1 << 22
    a = rng.normal(size=n) * 10.0 ** rng.uniform(-100, 100, n)
    b = (1.0 + rng.integers(0, 2 ** 52, n) * 2.0 ** -52) * 2.0 ** rng.integers(-300, 300, n)
    same(run(2, a, b), a / b)
    # divisors without an inverse: the division's infinities, zeros and NaN
    a = np.array([1.0, -1.0, 0.0, 2.0, -3.0, 0.0])
    b = np.array([0.0, 0.0, 0.0, np.inf, np.inf, 5.0])
    with np.errstate(divide="ignore", invalid="ignore"):
        same(run(2, a, b), a / b)
