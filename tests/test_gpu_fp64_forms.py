"""The FP64 forms of the interface sweep on the integer and FP32 pipes
(csrc/cg_fp64.cuh) and the cases in which the sweep leaves them.

Division, square root, product and the comparisons must equal the IEEE operations bit
for bit (they claim correct rounding, so there is no tolerance); the sweep must
keep the parity of one RHS evaluation with the oracle (1e-13 of each
variable's largest magnitude) where operands are out of the forms' range."""
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
#include "cg_fp64.cuh"
using namespace cgk;
__global__ void k(int op, const double* a, const double* b, double* x, double* y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double u = a[i], v = b[i];
    if (op == 0) { x[i] = div_f64(u, v); y[i] = u / v; }
    if (op == 1) { x[i] = sqrt_f64(u); y[i] = sqrt(u); }
    if (op == 2) { F64Range R; R.any(v); x[i] = R.ok() ? rcp_by(divisor(v)) : 1.0 / v; y[i] = 1.0 / v; }
    if (op == 3) { F64Range R; R.any0(u); x[i] = R.ok() ? div_by(u, host_divisor_sixty()) : u / 60.0; y[i] = u / 60.0; }
    if (op == 4) { x[i] = min_f64(u, v) + max_f64(u, v); y[i] = (u < v ? u : v) + (u > v ? u : v); }
    if (op == 5) { x[i] = minmod_f64(u, v); y[i] = (u > 0 && v > 0) ? (u < v ? u : v) : ((u < 0 && v < 0) ? (u > v ? u : v) : 0.0); }
    if (op == 7) {
      F64Range R; R.any(u);
      const double p = F64Products{R}.kz(u, v);
      x[i] = R.ok() ? p : u * v; y[i] = u * v;
    }
    if (op == 6) { x[i] = nonneg(u) ? 1.0 : 0.0; y[i] = 0.0 <= u ? 1.0 : 0.0; }
  }
}
extern "C" int run(int op, const double* a, const double* b, double* x, double* y, long long n) {
  k<<<608, 256>>>(op, a, b, x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("fp64_forms")
    src, lib = d / "k.cu", d / "k.so"
    src.write_text(KERNEL.replace("host_divisor_sixty()", "Divisor{0x001e000000000000ull, 0x0011111111111111ull, "
                                  "0.53333333333f, 0x40400000u}"))
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-fmad=false",
                           "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)])
    L = ctypes.CDLL(str(lib))
    L.run.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 4 + [ctypes.c_longlong]
    return L


def operands(seed, n=1 << 22):
    """Doubles with hard significands (few bits, all ones, near a power of two,
    random), exponents near 0, over the forms' range and over all of binary64,
    both signs, and the special values."""
    rng = np.random.default_rng(seed)
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    kind = rng.integers(0, 8, n)
    m = np.where(kind == 0, m & np.uint64(0xFFFFFF0000000), m)
    m = np.where(kind == 1, m | np.uint64(0xFFFFFF0000000), m)
    m = np.where(kind == 2, m & np.uint64(0x1F), m)
    m = np.where(kind == 3, m | np.uint64(0xFFFFFFFFFFFE0), m)
    span = np.where(rng.integers(0, 4, n) == 0, 402, 3)
    e = 1023 + np.rint(rng.uniform(-1.0, 1.0, n) * span).astype(np.int64)
    e = np.where(rng.integers(0, 32, n) == 0, rng.integers(0, 2048, n), e).astype(np.uint64)
    bits = (rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) | (e << np.uint64(52)) | m
    x = bits.view(np.float64).copy()
    x[:8] = [0.0, -0.0, 1.0, 2.0, 5e-324, -np.inf, np.inf, np.nan]
    return x


@pytest.mark.parametrize("op", range(8), ids=["div", "sqrt", "rcp", "sixty", "minmax", "minmod", "nonneg", "mul"])
def test_forms_equal_ieee(forms, op):
    a, b = operands(op), operands(100 + op)
    rng = np.random.default_rng(200 + op)
    q = rng.integers(0, a.size, a.size // 4)  # near-exact quotients, near-squares and equal operands
    with np.errstate(all="ignore"):
        if op == 1:
            s = np.abs(a[q])
            a[: q.size] = ((s * s).view(np.int64) + rng.integers(-2, 3, q.size)).view(np.float64)
        elif op == 0:
            a[8: 8 + q.size - 8] = (b[8: q.size] * rng.integers(1, 1 << 20, q.size - 8)).astype(np.float64)
        else:
            a[8: q.size] = b[8: q.size]
    if op in (4, 5):  # comparisons are of finite values
        a, b = np.where(np.isfinite(a), a, 1.0), np.where(np.isfinite(b), b, -1.0)
    ta, tb = torch.as_tensor(a, device="cuda"), torch.as_tensor(b, device="cuda")
    x, y = torch.empty_like(ta), torch.empty_like(ta)
    assert forms.run(op, ta.data_ptr(), tb.data_ptr(), x.data_ptr(), y.data_ptr(), ta.numel()) == 0
    same = x.view(torch.int64) == y.view(torch.int64)
    if op == 5:
        same |= (x == 0) & (y == 0)  # either zero
    same |= torch.isnan(x) & torch.isnan(y)
    bad = torch.nonzero(~same).flatten()
    assert bad.numel() == 0, [(float(ta[i]).hex(), float(tb[i]).hex()) for i in bad[:4].tolist()]


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_18042_gb300 import api as a
    return a


def rhs_parity(orc, api, prob, U, **kw):
    o, s = orc.Oracle(prob, **kw), api.Solver.from_problem(prob, **kw)
    assert rel_err(s.rhs(to_dev(U)), o.rhs(U)) <= 1e-13


@pytest.mark.parametrize("scheme", ["MEG6", "MIG4"])
@pytest.mark.parametrize("scale", [2.0 ** -420, 2.0 ** 420], ids=["tiny", "huge"])
def test_rhs_out_of_range_states(orc, api, scheme, scale):
    """Every interface leaves the forms: Sod with density and pressure scaled."""
    prob = inputs.shock_tube("sod", 130)
    U, _, _ = orc.Oracle(prob, scheme=scheme, cfl=0.3).advance(prob["U"], nsteps=3)
    prob["inflow"] = {k: (v[0] * scale, v[1], v[2] * scale) for k, v in prob["inflow"].items()}
    rhs_parity(orc, api, prob, U * scale, scheme=scheme)


@pytest.mark.parametrize("n", [(70, 66), (63, 64)])
def test_rhs_partly_out_of_range_2d(orc, api, n):
    """Some interfaces of a tile leave the forms: a spot of density and pressure 1e-125."""
    prob = inputs.triple_point(*n)
    U = orc.Oracle(prob, scheme="MEG6").advance(prob["U"], nsteps=3)[0]
    U[:, 20:23, 31:34] *= 1e-125
    rhs_parity(orc, api, prob, U, scheme="MEG6")


@pytest.mark.parametrize("kw", [dict(omega_window=w) for w in (1, 2, 3, 4)] + [dict(mp_eps=-1.0), dict(mp_alpha=2.5)])
def test_rhs_windows_and_mp_parameters(orc, api, kw):
    """The sensor window as node bits, MP5 with another alpha, and a negative
    tolerance (which the forms do not take); shocked data, grid spacings whose
    unit normals are not exactly 1."""
    prob = inputs.triple_point(131, 67)
    U = orc.Oracle(prob, scheme="MEG6").advance(prob["U"], nsteps=6)[0]
    rhs_parity(orc, api, prob, U, scheme="MEG6", **kw)
