"""The stage kernel's square root and its reciprocal against exact values and
the compiler's own, over the range of FP32."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2103_10114_gb300 import agcm

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "agcm_row.cuh"
__global__ void k_roots(const float* x, float* s, float* r, float* s0, float* r0, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float p[1] = {x[i]}, q[1];
  agcm::roots<1>(p, q);
  s[i] = p[0];
  r[i] = q[0];
  s0[i] = sqrtf(x[i]);
  r0[i] = 1.f / s0[i];
}
extern "C" int roots(const float* x, float* s, float* r, float* s0, float* r0, int n) {
  k_roots<<<(n + 255) / 256, 256>>>(x, s, r, s0, r0, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(cuda_ok, tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    src, so = d / "roots.cu", d / "roots.so"
    src.write_text(PROGRAM)
    subprocess.check_call(["nvcc", *agcm.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", agcm._CSRC,
                           "-o", str(so), str(src)])
    return ctypes.CDLL(str(so))


def _run(lib, x):
    import torch

    x = torch.as_tensor(x, dtype=torch.float32, device="cuda")
    out = [torch.empty_like(x) for _ in range(4)]
    assert lib.roots(*[ctypes.c_void_p(t.data_ptr()) for t in (x, *out)], x.numel()) == 0
    return [t.cpu().numpy() for t in out]


def test_within_a_rounding_of_exact(lib):
    """Where no residual leaves the normal range (2^-100 .. 2^126): the root
    is off by its rounding, 0.5 units, and a residual's share of under 2^-20
    of one; the reciprocal is that of the root, rounded in turn."""
    rng = np.random.default_rng(1)
    x = np.concatenate([2.0 ** rng.uniform(-100, 126, 200_000), rng.uniform(0.2, 1.2, 200_000)]).astype(np.float32)
    s, r, s0, r0 = _run(lib, x)
    units = lambda got, want: (np.abs(got.astype(np.float64) - want) / np.spacing(want.astype(np.float32))).max()
    root = np.sqrt(x.astype(np.float64))
    assert units(s, root) <= 0.5001, units(s, root)
    assert units(r, 1.0 / s.astype(np.float64)) <= 0.5001, units(r, 1.0 / s.astype(np.float64))
    # the same numbers as the rounded root and quotient, but for ties within 1e-4 units
    assert (s != s0).mean() <= 1e-3 and (r != r0).mean() <= 2e-3


def test_outside_the_range(lib):
    """Zero, subnormal, negative, infinite and NaN arguments give what the root
    and the quotient give; tiny normal ones are within a unit of it."""
    tiny = np.float32(2.0) ** np.arange(-149, -126).astype(np.float32)
    odd = np.array([0.0, -0.0, -1.0, -1e-40, np.inf, -np.inf, np.nan, 1e-45, 1.1754942e-38], np.float32)
    x = np.concatenate([odd, tiny])
    s, r, s0, r0 = _run(lib, x)
    assert np.array_equal(s, s0, equal_nan=True) and np.array_equal(r, r0, equal_nan=True)
    x = (2.0 ** np.random.default_rng(2).uniform(-126, -100, 100_000)).astype(np.float32)
    s, r, s0, r0 = _run(lib, x)
    assert (np.abs(s - s0) <= np.spacing(s0)).all() and (np.abs(r - r0) <= np.spacing(r0)).all()
