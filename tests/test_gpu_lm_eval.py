"""The LM evaluation's two forms: the short one, for launches of up to two
blocks per SM, and the general one above, on either side of the line (tile
pairs of 16 stations: 23 tiles are 276 blocks, 25 are 325).

A solve's cost at its last step comes from the evaluation, in pair arithmetic
over the statistics of the float32 data; the residual call forms the same cost
from the visibilities in float32.  Over T F <= 12 terms per baseline these
agree to 1e-5 relative (the residual call's roundings; sums of positive terms).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402


@pytest.mark.parametrize("N,T,F", [(2, 5, 1), (17, 12, 1), (64, 5, 1), (368, 2, 1), (390, 2, 2)])
def test_solve_cost_equals_the_residual_cost(N, T, F):
    g = torch.Generator(device="cuda").manual_seed(N)
    B = N * (N - 1) // 2
    X = torch.view_as_complex(torch.randn((T, B, F, 2, 2, 2), generator=g, device="cuda"))
    C = torch.view_as_complex(torch.randn((T, B, F, 2), generator=g, device="cuda"))
    J0 = torch.eye(2, dtype=torch.complex128, device="cuda").repeat(N, 1, 1).contiguous()
    shp = sc.Shape(N, T, F, 1, 1)
    ws = sc.workspace(shp, sc.SC_MIXED)
    out = sc.solve_cluster(shp, X, C, J0, sc.SC_MIXED, ws, n_lm=3)
    J, cost = out[0], out[1]
    _, want = sc.residual(shp, X, C, J, sc.SC_MIXED, ws)
    assert sc.device_status(ws) == 0
    assert np.isfinite(cost.item())
    assert abs(cost.item() - want.item()) <= 1e-5 * want.item()
