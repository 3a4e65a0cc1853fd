"""2D grids with more rows than a launch's y dimension holds tiles."""
import numpy as np
import pytest

from paper_2511_18042_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("rows", [65535 * 16, 65535 * 16 + 8, 65535 * 16 + 40])
def test_mixed_lad_on_a_tall_grid(rows):
    """The mixed form's LAD on 8 x 1,048,560 (the most tiles of 16 rows that
    fit a launch's y dimension) and a few rows more: data of period 8 along y
    gives every row the values of a short grid, bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_18042_gb300 import api
    rng = np.random.default_rng(5)
    W = np.empty((4, 8, 8))
    W[0], W[3] = rng.uniform(0.5, 2.0, (2, 8, 8))
    W[1], W[2] = rng.uniform(-1.0, 1.0, (2, 8, 8))

    def rhs(n):
        prob = inputs._problem("rows", 2, [8, n], [0.1, 0.1], [[0, 0], [0, 0]], W, 1.4)
        U = torch.as_tensor(prob["U"], device="cuda").repeat(1, n // 8, 1)
        return api.Solver.from_problem(prob, scheme="LAD_E4", precision=1).rhs(U)

    assert torch.equal(rhs(rows), rhs(64)[:, :8].repeat(1, rows // 8, 1))
