"""The choices of the FP64 interface sweep (HLLC state, sensor window) in the
corners where a shortened test could choose differently, against the oracle
(1e-13 of each variable's largest magnitude for one RHS evaluation)."""
import numpy as np
import pytest

from paper_2511_18042_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from tests.gpu_util import rel_err, to_dev  # noqa: E402


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_18042_gb300 import api as a
    return a


@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("gamma", [1.001, 1.000001])
def test_contact_right_of_the_right_wave(orc, api, gamma, fma):
    """gamma near 1 and a strong jump: the estimated contact speed can exceed
    the right wave's, SR < 0 <= S*.  The flux there is the left star state's
    (the first test of Eq. (10) that holds decides)."""
    rL, pL, rR = 95.6224235889941, 6034.428430832117, 0.014406564806903267
    c = np.sqrt(gamma * pL / rL)
    jumps = []
    for pR in (4e-3, 1e-3, 1e-4):
        for d in np.linspace(-2e-3, 6e-3, 33):
            jumps.append((pR, -c * (1.0 + d)))
    N = 16 * len(jumps)
    W = np.empty((3, N))
    for k, (pR, u) in enumerate(jumps):
        W[:, 16 * k:16 * k + 8] = np.array([rL, u, pL])[:, None]
        W[:, 16 * k + 8:16 * k + 16] = np.array([rR, u, pR])[:, None]
    prob = inputs._problem("jumps", 1, [N], [1.0], [[inputs.EXTRAP, inputs.EXTRAP]], W, gamma)
    # the waves of the cell states at every jump from the dense to the thin gas
    gm1 = gamma - 1.0
    pR, u = np.array(jumps).T
    H = [(p / gm1 + 0.5 * r * u * u + p) / r for r, p in ((rL, pL), (rR, pR))]
    sL, sR = np.sqrt(rL), np.sqrt(rR)
    ch = np.sqrt(gm1 * ((sL * H[0] + sR * H[1]) / (sL + sR) - 0.5 * u * u))
    SL = np.minimum(u - c, u - ch)
    SR = np.maximum(u + np.sqrt(gamma * pR / rR), u + ch)
    S = (rR * u * (SR - u) - rL * u * (SL - u) + (pL - pR)) / (rR * (SR - u) - rL * (SL - u))
    assert ((SR < 0) & (S >= 0)).sum() >= 3
    kw = dict(scheme="MEG6")
    o, s = orc.Oracle(prob, **kw), api.Solver.from_problem(prob, fma_sweep=fma, **kw)
    # (fused multiply-adds: rounding only)
    assert rel_err(s.rhs(to_dev(prob["U"])), o.rhs(prob["U"])) <= (1e-9 if fma else 1e-13)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("at", [(16, 32), (16, 44), (16, 56)])
def test_sensor_window_with_a_nan(orc, api, at, precision):
    """A node without a value: the nodes whose stencil does not hold it keep
    theirs.  The window's maximum is taken in order and a comparison with NaN
    is false, so a NaN discards what came before it."""
    prob = inputs.triple_point(96, 64)
    U = orc.Oracle(prob, scheme="MEG6").advance(prob["U"], nsteps=12)[0]
    U[:, at[1], at[0]] = np.nan
    kw = dict(scheme="MEG6")
    Ro = orc.Oracle(prob, **kw).rhs(U)
    Rg = api.Solver.from_problem(prob, precision=precision, **kw).rhs(to_dev(U)).cpu().numpy()
    assert np.array_equal(np.isfinite(Rg), np.isfinite(Ro))
    ok = np.isfinite(Ro).all(axis=0)
    assert 0 < (~ok).sum() < ok.size // 4
    assert rel_err(Rg[:, ok], Ro[:, ok]) <= (1e-3 if precision else 1e-13)


@pytest.mark.parametrize("thresh", [float("nan"), float("inf"), -1.0])
def test_sensor_thresholds_out_of_the_ordinary(orc, api, thresh):
    """No node is above NaN or infinity (the linear reconstruction everywhere);
    every node is above a negative threshold."""
    prob = inputs.triple_point(96, 64)
    U = orc.Oracle(prob, scheme="MEG6").advance(prob["U"], nsteps=12)[0]
    kw = dict(scheme="MEG6", sensor_thresh=thresh)
    Ro = orc.Oracle(prob, **kw).rhs(U)
    assert rel_err(api.Solver.from_problem(prob, **kw).rhs(to_dev(U)), Ro) <= 1e-13


@pytest.mark.parametrize("eps", [0.0, -0.0])
def test_mp_tolerance_of_either_zero(orc, api, eps):
    prob = inputs.triple_point(96, 64)
    U = orc.Oracle(prob, scheme="MEG6").advance(prob["U"], nsteps=12)[0]
    kw = dict(scheme="MEG6", mp_eps=eps)
    Ro = orc.Oracle(prob, **kw).rhs(U)
    assert rel_err(api.Solver.from_problem(prob, **kw).rhs(to_dev(U)), Ro) <= 1e-13
