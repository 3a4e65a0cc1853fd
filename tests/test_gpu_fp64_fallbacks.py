"""Operands out of the range of the integer-pipe forms (csrc/cg_fp64.cuh) through
every FP64 kernel that uses them: sensor, LAD fields, coefficients and node
fluxes, overbar, divergences, interface fluxes, filter, viscous terms, line
solves, the sweep on curvilinear grids and the three Runge-Kutta updates, against
the oracle; and the products and divisions the sweep's forms are made of, bit
for bit.

Right-hand sides within 1e-13 of each variable's largest magnitude, 1e-12 for
the compact schemes (their line solves round differently by ulps); one step
within 1e-12."""
import ctypes
import math
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
#include <vector>
#include "cg_lines.cuh"
using namespace cgk;
__global__ void k(int op, const double* a, const double* b, const Divisor* D, double* x, double* y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double u = a[i], v = b[i];
    F64Range R;
    if (op == 0) { R.any(u); R.any(v); x[i] = R.ok() ? F64Products::kk(u, v) : u * v; y[i] = u * v; }
    if (op == 1) { R.any0(u); x[i] = R.ok() ? div_by(u, D[i % 4096]) : u / b[i % 4096]; y[i] = u / b[i % 4096]; }
    if (op == 2) { x[i] = coef_mul(u, v); y[i] = u * v; }
  }
}
extern "C" int run(int op, const double* a, const double* b, const double* b_host, double* x, double* y, long long n) {
  std::vector<Divisor> h(4096);
  for (int i = 0; i < 4096; ++i) h[i] = host_divisor(op == 1 ? b_host[i] : 1.0);
  Divisor* D = nullptr;
  if (cudaMalloc(&D, h.size() * sizeof(Divisor)) != cudaSuccess) return -1;
  cudaMemcpy(D, h.data(), h.size() * sizeof(Divisor), cudaMemcpyHostToDevice);
  k<<<608, 256>>>(op, a, b, D, x, y, n);
  const int rc = (int)cudaDeviceSynchronize();
  cudaFree(D);
  return rc;
}
"""


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("fp64_fallbacks")
    src, lib = d / "k.cu", d / "k.so"
    src.write_text(KERNEL)
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-fmad=false",
                           "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)])
    L = ctypes.CDLL(str(lib))
    L.run.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 5 + [ctypes.c_longlong]
    return L


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_18042_gb300 import api as a
    return a


def doubles(rng, n, lo, hi, positive=False):
    """Hard and random significands, exponents lo .. hi - 1."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    m[::5] |= np.uint64(0xFFFFFFFFFFFE0)
    m[1::7] &= np.uint64(0x1F)
    s = np.zeros(n, np.uint64) if positive else rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)
    return (s | (rng.integers(1023 + lo, 1023 + hi, n).astype(np.uint64) << np.uint64(52)) | m).view(np.float64)


@pytest.mark.parametrize("op", [0, 1, 2], ids=["kk", "host_divisor", "coef_mul"])
def test_products_and_divisions_equal_ieee(forms, op):
    n, rng = 1 << 21, np.random.default_rng(30 + op)
    a, b = doubles(rng, n, -410, 410), doubles(rng, n, -410, 410)
    a[::3], b[::3] = doubles(rng, a[::3].size, -2, 2), doubles(rng, a[::3].size, -2, 2)
    if op == 1:  # parameters as the host prepares them; numerators also zero, out of range and without a value
        b = doubles(rng, n, -100, 100, positive=True)
        b[:8] = [1.0, 2.0, 0.4, 60.0, 1.0 / 3.0, 0.1, np.nextafter(1.0, 2.0), np.nextafter(2.0, 0.0)]
    elif op == 2:  # line coefficients with any value
        a = doubles(rng, n, -40, 40)
        b = doubles(rng, n, -1023, 1025)
    if op:
        (a if op == 1 else b)[:8] = [0.0, -0.0, 5e-324, -1e-310, np.inf, -np.inf, np.nan, 2.0 ** -400]
    ta, tb = torch.as_tensor(a, device="cuda"), torch.as_tensor(b, device="cuda")
    x, y = torch.empty_like(ta), torch.empty_like(ta)
    assert forms.run(op, ta.data_ptr(), tb.data_ptr(), b.ctypes.data, x.data_ptr(), y.data_ptr(), n) == 0
    bad = torch.nonzero((x.view(torch.int64) != y.view(torch.int64)) & ~(torch.isnan(x) & torch.isnan(y))).flatten()
    assert bad.numel() == 0, [(float(ta[i]).hex(), float(tb[i]).hex()) for i in bad[:4].tolist()]


HYB = dict(scheme="HYBRID", hybrid_mode=1, hybrid_sensor=1)
SCHEMES = [dict(scheme="MEG6"), dict(scheme="MIG4"), dict(scheme="LAD_E4"), dict(scheme="LAD_C6"), HYB]
IDS = ["meg6", "mig4", "lad_e4", "lad_c6", "hybrid"]


def tol(kw):
    return 1e-12 if kw["scheme"] in ("MIG4", "LAD_C6") else 1e-13


def box_2d(orc):
    prob = inputs.triple_point(83, 70)
    prob["U"] = orc.Oracle(prob, scheme="MEG6").advance(prob["U"], nsteps=6)[0]
    return prob


def box_3d(viscous):
    """A wavy periodic grid, a smooth flow without critical points of its fields."""
    xyz, per = inputs.wavy_grid_3d((18, 14, 12), amp=0.05)
    x, y, z = xyz
    t = 2 * math.pi
    W = np.stack([1.0 + 0.1 * np.sin(t * (x + y)) + 0.05 * np.sin(t * (x + 2 * y + 3 * z) + 0.7),
                  0.1 * np.sin(t * x) + 0.05 * np.sin(t * (x + 0.3 * y - z) + 0.4),
                  0.08 * np.sin(t * y) + 0.04 * np.cos(t * z), 0.06 * np.sin(t * z) + 0.03 * np.sin(t * x),
                  8.0 + 0.3 * np.cos(t * z) + 0.2 * np.cos(t * (2 * x - y + z) + 1.3)])
    prob = inputs.field_on_curvilinear(xyz, per, W)
    return inputs._viscous(prob, 30.0, 0.3, 0.5, 1.0) if viscous else prob


def scaled(prob, kw, state):
    """(parameters, state): every value out of the forms' range, or a spot of them."""
    U, kw = prob["U"].copy(), dict(kw)
    f = {"tiny": 2.0 ** -420, "huge": 2.0 ** 420, "spot": 1.0}[state]
    if kw["scheme"] == "HYBRID":
        kw["hyb_rho"] = f * float(np.quantile(U[0], 0.3))  # both fluxes in use
    U *= f
    if state == "spot":
        U[..., 5:7, 5:8] *= 1e-125
    return kw, U


@pytest.mark.parametrize("state", ["tiny", "huge", "spot"])
@pytest.mark.parametrize("kw", SCHEMES, ids=IDS)
@pytest.mark.parametrize("box", ["2d", "3d", "3d_viscous"])
def test_out_of_range_states(orc, api, box, kw, state):
    prob = box_2d(orc) if box == "2d" else box_3d(box == "3d_viscous")
    kw, U = scaled(prob, kw, state)
    o, s = orc.Oracle(prob, **kw), api.Solver.from_problem(prob, **kw)
    Ro = o.rhs(U)
    assert np.isfinite(Ro).all()
    assert rel_err(s.rhs(to_dev(U)), Ro) <= tol(kw)
    if box == "3d_viscous" or state == "spot":  # (a spot does not survive a step; viscosity is not scaled with the state)
        return
    dt = o.cfl_dt(U)
    assert abs(s.cfl_dt(to_dev(U)) - dt) <= 1e-14 * dt
    assert rel_err(s.rk3_step(to_dev(U), dt), o.rk3_step(U, dt)) <= 1e-12


@pytest.mark.parametrize("path", ["table", "persistent"])
@pytest.mark.parametrize("f", [2.0 ** -420, 2.0 ** 420], ids=["tiny", "huge"])
def test_out_of_range_batch(api, path, f):
    """Members of a work table as alone, bit for bit."""
    probs = inputs.batched_riemann(count=4, seed=9, n_lo=24, n_hi=70)
    kw = dict(HYB, hyb_rho=0.3 * f)
    U0 = [to_dev(p["U"] * f) for p in probs]
    alone, members = ([u.clone() for u in U0] for _ in range(2))
    batch = api.Batch([api.Solver.from_problem(p, **kw) for p in probs], members)
    batch.set_path(path)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for _ in range(3):
            batch.step(stream)
    batch.sync(stream)
    dt = torch.zeros(2, dtype=torch.float64, device="cuda")
    for p, u, v in zip(probs, alone, members):
        s = api.Solver.from_problem(p, **kw)
        for _ in range(3):
            s.step(u, dt)
        assert torch.isfinite(u).all() and torch.equal(u, v)
