"""The FP32 square root of shock capturing (root in csrc/lbm_device.cuh), scalar and
packed: the same bits, the exact root but for a few values one ulp off, infinities, NaN
and zeros as sqrt gives them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "lbm_device.cuh"
__global__ void k(const float* a, float* scalar, float* packed, int n) {
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i + 1 >= n) return;
  scalar[i] = lbm::root(a[i]);
  scalar[i + 1] = lbm::root(a[i + 1]);
  const lbm::F2 v = lbm::root(lbm::F2(a[i], a[i + 1]));
  packed[i] = v.x;
  packed[i + 1] = v.y;
}
extern "C" int roots(const float* a, float* scalar, float* packed, int n) {
  k<<<(n / 2 + 255) / 256, 256>>>(a, scalar, packed, n);
  return int(cudaDeviceSynchronize());
}
"""


def test_scalar_and_packed_root(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14712_gb300 import build
    src, lib = tmp_path / "roots.cu", tmp_path / "roots.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-prec-div=false", "-I", os.path.join(ROOT, "paper_2510_14712_gb300", "csrc"),
                   "-shared", str(src), "-o", str(lib), "-lcudart"], check=True)
    fn = ctypes.CDLL(str(lib)).roots
    rng = np.random.default_rng(5)
    a = np.concatenate([2.0 ** rng.uniform(-100.5, 127.9, 1 << 20), 2.0 ** rng.uniform(-8, 8, 1 << 20), 2.0 ** rng.uniform(-148, -101, 1 << 18),
                        [0.0, -0.0, np.inf, np.nan, np.inf, 1.0, 4.0, 3.4028235e38]]).astype(np.float32)
    d = torch.from_numpy(a).cuda()
    s, p = torch.empty_like(d), torch.empty_like(d)
    assert fn(ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(s.data_ptr()), ctypes.c_void_p(p.data_ptr()), d.numel()) == 0
    s, p = s.cpu().numpy(), p.cpu().numpy()
    assert np.array_equal(s.view(np.uint32), p.view(np.uint32))
    want = np.sqrt(a.astype(np.float64)).astype(np.float32)
    assert np.array_equal(s[-8:], want[-8:], equal_nan=True)
    n = 1 << 21                                                     # exact remainder
    ulp = np.abs(s[:n].view(np.int32) - want[:n].view(np.int32))
    assert ulp.max() <= 1 and (ulp != 0).mean() <= 2e-6
    small = slice(n, n + (1 << 18))
    assert np.all(np.abs(s[small] - want[small]) <= 1e-19 + 2.0 ** -22 * want[small])
