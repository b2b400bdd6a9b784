"""The cost of a residual, a sum over baselines and timeslot chunks by one block.

With zero coherencies the residual is V itself, so the cost is sum |V|^2.  The
float32 values are added to about twice float32's precision; sizes below one
value per thread, ragged, and many per thread, magnitudes from where the sum
is beyond float32's range to tiny ones.  Tolerance: the values themselves are
float32 sums of at most 8 T F squares (T F <= 40) in the kernel's chunks,
(8 T F + 2) 2^-24 relative since all terms are positive.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402


@pytest.mark.parametrize("scale", [1.0, 1e18, 1e-12])
@pytest.mark.parametrize("N,T,F", [(2, 1, 1), (45, 1, 1), (46, 3, 1), (64, 10, 4), (150, 10, 1)])
def test_cost_is_the_sum_of_squares(N, T, F, scale):
    B = N * (N - 1) // 2
    rng = np.random.default_rng(N)
    V = (scale * (rng.standard_normal((T, B, F, 2, 2)) + 1j * rng.standard_normal((T, B, F, 2, 2)))).astype(np.complex64)
    shp = sc.Shape(N, T, F, 1, 1)
    ws = sc.workspace(shp, sc.SC_MIXED)
    C = torch.zeros((T, B, F), dtype=torch.complex64, device="cuda")
    J = torch.eye(2, dtype=torch.complex128, device="cuda").repeat(N, 1, 1).contiguous()
    _, cost = sc.residual(shp, torch.as_tensor(V).cuda(), C, J, sc.SC_MIXED, ws)
    want = np.sum(np.abs(V.astype(np.complex128)) ** 2)
    assert abs(cost.item() - want) <= (8 * T * F + 2) * 2.0 ** -24 * want
    assert sc.device_status(ws) == 0
