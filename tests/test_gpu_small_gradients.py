"""FP64 interface fluxes whose derivatives are smaller than the products on the
integer pipes take (compact gradients beside a jump into gas at rest decay by
0.268 a row, through all magnitudes): the form with plain products takes them,
with the IEEE form's bits, and the sweep keeps its parity with the oracle."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2511_18042_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from tests.gpu_util import rel_err, to_dev  # noqa: E402

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_18042_gb300", "csrc")

KERNEL = r"""
#include "cg_kernels.cuh"
using namespace cgk;
constexpr int LW = 4, RW = SWEEP_TL + 9, RD = SWEEP_TL + 3, RH = SWEEP_TL + 1;
// one tile of LW lines a block, an interface a thread: the rarely taken path (x), the IEEE form (y),
// and whether the forms with plain and with integer-pipe products took the interface
__global__ void k(GbrCfg q, DevGrid g, const double* W, const double* D, const double* H, double* x, double* y, int* took) {
  const double *w = W + blockIdx.x * 4 * LW * RW, *d = D + blockIdx.x * 4 * LW * RD, *h = H + blockIdx.x * 4 * LW * RH;
  const int a = threadIdx.x % SWEEP_TL, l = threadIdx.x / SWEEP_TL, o = blockIdx.x * blockDim.x + threadIdx.x;
  const bool disc = (a & 1) != 0;
  auto ld = [&](const double* b, int r, int rows, double* v) {
    for (int m = 0; m < 4; ++m) v[m] = b[(m * LW + l) * rows + r];
  };
  auto fw = [&](int j, double* v) { ld(w, a + 2 + j, RW, v); };
  auto fd = [&](int j, double* v) { ld(d, a + 1 + j, RD, v); };
  auto fh = [&](int j, double* v) { ld(h, a + j, RH, v); };
  double xi[3] = {0.0, 0.0, 0.0}, F[4], io[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  const bool plain = gbr_flux_f64<2, true, 0, false, false>(q, g, fw, fd, fh, disc, xi, F);
  const bool fast = gbr_flux_f64<2, true, 0, false, true>(q, g, fw, fd, fh, disc, xi, F);
  took[o] = (plain ? 1 : 0) | (fast ? 2 : 0);
  gbr_flux_rare<2, true, 0, LW, 0>(q, g, w, d, h, a, l, disc, io);
  for (int v = 0; v < 4; ++v) x[4 * o + v] = io[v];
  for (int v = 0; v < 5; ++v) io[v] = 0.0;
  gbr_flux_ieee<2, true, 0, LW>(q, g, w, d, h, a, l, disc, io);
  for (int v = 0; v < 4; ++v) y[4 * o + v] = io[v];
}
extern "C" int run(int tiles, double gamma, const double* W, const double* D, const double* H, double* x, double* y, int* took) {
  DevGrid g{};
  GbrCfg q{};
  g.nd = 2;
  g.cxh[0] = g.cxh[1] = 0.25;
  g.cg2[0] = 0.0625; g.cg[0] = 0.25; g.cig2[0] = 16.0;
  g.cn[0][0] = 1.0; g.ct1[0][1] = 1.0;
  q.gamma = gamma; q.gm1 = gamma - 1.0; q.thr = 0.01; q.eps = 1e-20; q.alpha = 4.0; q.window = 4;
  q.f64_fast = 1;
  q.d_gm1 = host_divisor(q.gm1);
  k<<<tiles, SWEEP_TL * LW>>>(q, g, W, D, H, x, y, took);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("small_gradients")
    src, out = d / "k.cu", d / "k.so"
    src.write_text(KERNEL)
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-fmad=false",
                           "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-o", str(out), str(src)])
    L = ctypes.CDLL(str(out))
    L.run.argtypes = [ctypes.c_int, ctypes.c_double] + [ctypes.c_void_p] * 6
    return L


@pytest.mark.parametrize("at_rest", [True, False])
def test_plain_products_take_small_derivatives(lib, at_rest):
    tiles, rng = 1080, np.random.default_rng(17)
    W = rng.uniform(0.5, 2.0, (tiles, 4, 4, 73))
    if at_rest:  # one state a line, as ahead of a jump
        W = np.broadcast_to(W[..., :1], W.shape).copy()
        W[:, 1:3] = 0.0
    else:
        W[:, 1:3] -= 1.25
    scale = (2.0 ** -np.arange(tiles, dtype=np.float64)).reshape(tiles, 1, 1, 1)  # 1 to 2^-1079: to subnormals, to zero
    D = rng.uniform(-0.1, 0.1, (tiles, 4, 4, 67)) * scale
    H = rng.uniform(-0.1, 0.1, (tiles, 4, 4, 65)) * scale
    t = [torch.as_tensor(v, device="cuda") for v in (W, D, H)]
    x, y = (torch.empty((tiles, 256, 4), dtype=torch.float64, device="cuda") for _ in range(2))
    took = torch.empty((tiles, 256), dtype=torch.int32, device="cuda")
    assert lib.run(tiles, 1.4, *[v.data_ptr() for v in t], x.data_ptr(), y.data_ptr(), took.data_ptr()) == 0
    assert bool(torch.isfinite(y).all())
    assert torch.equal(x, y)  # (either zero: the forms' comparisons order -0 before 0)
    plain, fast = (took & 1) != 0, (took & 2) != 0
    # every interface in the linear form; limited ones reconstruct from W alone
    small = torch.arange(tiles, device="cuda") >= 480
    linear = torch.arange(256, device="cuda") % 2 == 0
    assert bool(plain[:, linear].all())
    assert not bool(fast[small][:560][:, linear].any())


@pytest.mark.parametrize("scheme", ["MIG4", "LAD_C6"])
def test_tube_with_decaying_gradients(orc, api, scheme):
    """1400 rows at rest behind a jump: gradients from O(1) through every
    magnitude to zero; one right-hand side and one step of the oracle."""
    prob = inputs.shock_tube("sod", 1600)
    prob["U"] = np.roll(prob["U"], -650, axis=1)
    prob["U"][:, -650:] = prob["U"][:, -651:-650]
    kw = dict(scheme=scheme, cfl=0.1)
    o, s = orc.Oracle(prob, **kw), api.Solver.from_problem(prob, **kw)
    assert rel_err(s.rhs(to_dev(prob["U"])), o.rhs(prob["U"])) <= 1e-13
    dt = o.cfl_dt(prob["U"])
    assert rel_err(s.rk3_step(to_dev(prob["U"]), dt), o.rk3_step(prob["U"], dt)) <= 1e-12


@pytest.mark.parametrize("n", [(700, 66), (66, 700)])
def test_2d_with_decaying_gradients(orc, api, n):
    prob = inputs.triple_point(*n)
    U = orc.Oracle(prob, scheme="MEG6").advance(prob["U"], nsteps=4)[0]
    kw = dict(scheme="MIG4")
    o, s = orc.Oracle(prob, **kw), api.Solver.from_problem(prob, **kw)
    assert rel_err(s.rhs(to_dev(U)), o.rhs(U)) <= 1e-13
    dt = o.cfl_dt(U)
    assert rel_err(s.rk3_step(to_dev(U), dt), o.rk3_step(U, dt)) <= 1e-12


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_18042_gb300 import api as a
    return a
