"""The one-pass overbar of 2D FP32 grids (k_gauss2_tile) against the two passes
it replaces (k_gauss along x, then y): the same values, so bit for bit, on
tiles that fit, remainders of one node, the smallest grids and every kind of
boundary (periodic, copied, mirrored)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_18042_gb300", "csrc")

KERNEL = r"""
#include "cg_lad.cuh"
using namespace cgk;
extern "C" int run(int nx, int ny, int bx, int by, const float* a, const float* b, float* t0, float* t1, float* two_a,
                   float* two_b, float* one_a, float* one_b) {
  DevGrid g{};
  g.nd = 2; g.nv = 4; g.n[0] = nx; g.n[1] = ny; g.n[2] = 1; g.N = (long long)nx * ny;
  g.bc[0][0] = g.bc[0][1] = bx; g.bc[1][0] = g.bc[1][1] = by;
  const int nb = (int)((g.N + 255) / 256);
  k_gauss<2, float><<<nb, 256>>>(g, 0, a, b, t0, t1, nullptr, 0);
  k_gauss<2, float><<<nb, 256>>>(g, 1, t0, t1, two_a, two_b, nullptr, 0);
  k_gauss2_tile<float><<<dim3((nx + GT_X - 1) / GT_X, (ny + GT_Y - 1) / GT_Y), 256>>>(g, a, b, one_a, one_b, nullptr, 0);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("overbar")
    src, out = d / "k.cu", d / "k.so"
    src.write_text(KERNEL)
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-fmad=false",
                           "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-o", str(out), str(src)])
    L = ctypes.CDLL(str(out))
    L.run.argtypes = [ctypes.c_int] * 4 + [ctypes.c_void_p] * 8
    return L


@pytest.mark.parametrize("bc", [(0, 0), (1, 2), (2, 1), (0, 4), (3, 0)])
@pytest.mark.parametrize("n", [(8, 8), (32, 16), (33, 17), (31, 15), (64, 9), (65, 130), (9, 257)])
def test_one_pass_equals_two(lib, n, bc):
    rng = np.random.default_rng(n[0] * 1000 + n[1])
    f = [torch.as_tensor(rng.uniform(0.0, 1.0, n[0] * n[1]).astype(np.float32) ** 4, device="cuda") for _ in range(2)]
    o = [torch.full_like(f[0], float("nan")) for _ in range(6)]
    assert lib.run(n[0], n[1], bc[0], bc[1], *[t.data_ptr() for t in f + o]) == 0
    for two, one in ((o[2], o[4]), (o[3], o[5])):
        assert torch.equal(two.view(torch.int32), one.view(torch.int32))
