"""The square root, its reciprocal and the reciprocal of the gate engine's reflectors
(Newton-Raphson steps in FP32, third-order steps in FP64, from the hardware's estimates)
against wider arithmetic, over the whole range that the reduction gives them."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2207_03711_gb300 import build_lib

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "gate.cuh"
using namespace mpsvqe;
template <class R>
__global__ void k(int n, const R* x, R* root, R* inv_root, R* inv) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  gate::root_and_inverse(x[i], root + i, inv_root + i);
  inv[i] = gate::inverse(x[i]);
}
extern "C" int run(int f64, int n, const void* x, void* root, void* inv_root, void* inv) {
  if (f64) k<double><<<(n + 255) / 256, 256>>>(n, (const double*)x, (double*)root, (double*)inv_root, (double*)inv);
  else k<float><<<(n + 255) / 256, 256>>>(n, (const float*)x, (float*)root, (float*)inv_root, (float*)inv);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_roots_and_reciprocals(tmp_path, dtype):
    torch = pytest.importorskip("torch")
    src, lib = tmp_path / "roots.cu", tmp_path / "roots.so"
    src.write_text(SOURCE)
    subprocess.run([build_lib._nvcc(), *build_lib.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                    build_lib.CSRC, str(src), "-o", str(lib)], check=True)
    f64 = dtype == np.float64
    info = np.finfo(dtype)
    rng = np.random.default_rng(0)
    # from 16 times the smallest normal number (below counts as zero) to a quarter of the largest
    e = rng.integers(info.minexp + 4, info.maxexp - 2, 200_000)
    x = np.ldexp(rng.uniform(1.0, 2.0, e.size), e).astype(dtype)
    edge = np.array([info.minexp + 4, info.maxexp - 3, -1, 0, 1, 2])
    x = np.concatenate([x, np.ldexp(1.0, edge).astype(dtype), np.nextafter(np.ldexp(1.0, edge).astype(dtype), dtype(0))])
    dx = torch.from_numpy(x).cuda()
    out = [torch.empty_like(dx) for _ in range(3)]
    p = [ctypes.c_void_p(t.data_ptr()) for t in [dx] + out]
    assert ctypes.CDLL(str(lib)).run(int(f64), len(x), *p) == 0
    root, inv_root, inv = (t.cpu().numpy().astype(np.longdouble) for t in out)
    w = x.astype(np.longdouble)
    s = np.sqrt(w)
    # the steps leave the square (third power) of the estimate's error, far below the last
    # place: what remains is one rounding in the reciprocal, two in the roots
    eps = np.longdouble(info.eps)
    for got, ref, ulps in ((root, s, 1.5), (inv_root, 1 / s, 1.5), (inv, 1 / w, 1.0)):
        assert np.abs(got / ref - 1).max() <= ulps * eps
