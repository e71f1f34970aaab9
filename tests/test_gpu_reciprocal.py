"""The pair kernel's reciprocal (rcp_newton, csrc/lbm_step_pair.cuh) against FP64 over every
mantissa at exponents across its range: Newton's step squares the first guess' relative error
(below 2^-22, PTX's bound for rcp.approx is 2^-23) and rounds once, so 0.5 ulp + 2^-44 relative, 0.501
ulp; at most one mantissa in ten thousand away from __frcp_rn, and by one ulp; NaN at 0 and at the
infinities."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2110_05197_gb300 import build as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

SRC = """
#include "lbm_step.cuh"
#include "lbm_step_pair.cuh"
__global__ void run(const float* a, float* newton, float* ieee, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  newton[i] = lbm::rcp_newton(a[i]);
  ieee[i] = __frcp_rn(a[i]);
}
extern "C" int reciprocals(const float* a, float* newton, float* ieee, int n) {
  run<<<(n + 255) / 256, 256>>>(a, newton, ieee, n);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def reciprocals(tmp_path_factory):
    d = tmp_path_factory.mktemp("rcp")
    (d / "rcp.cu").write_text(SRC)
    subprocess.run([B.NVCC, *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I",
                    B.CSRC, "-I", os.path.join(B.ROOT, "include"), str(d / "rcp.cu"), "-o", str(d / "rcp.so")], check=True)
    fn = ctypes.CDLL(str(d / "rcp.so")).reciprocals

    def call(a):
        t = torch.from_numpy(a).cuda()
        x, y = torch.empty_like(t), torch.empty_like(t)
        torch.cuda.synchronize()
        assert fn(*[ctypes.c_void_p(v.data_ptr()) for v in (t, x, y)], t.numel()) == 0
        return x.cpu().numpy(), y.cpu().numpy()

    return call


@pytest.mark.parametrize("exponent", [-126, -100, -24, -7, -1, 0, 3, 24, 100, 125])
def test_reciprocal(reciprocals, exponent):
    bits = (np.arange(1 << 23, dtype=np.uint32) | np.uint32((exponent + 127) << 23))
    a = bits.view(np.float32).copy()
    a[::2] *= np.float32(-1)
    x, y = reciprocals(a)
    true = 1.0 / a.astype(np.float64)
    ulp = np.spacing(np.abs(true.astype(np.float32))).astype(np.float64)
    assert np.max(np.abs(x.astype(np.float64) - true) / ulp) <= 0.501
    off = np.abs(x.view(np.int32).astype(np.int64) - y.view(np.int32))
    assert off.max() <= 1 and np.mean(off > 0) <= 1e-4


def test_reciprocal_of_zero_and_infinities(reciprocals):
    x, _ = reciprocals(np.array([0.0, -0.0, np.inf, -np.inf, np.nan], np.float32))
    assert np.all(np.isnan(x))
