"""The float32 triangular solves at the edges of the cluster kernel's ranges.

Orders of 2 tile rows (fewer rows than CTAs), 8 and 9 (clusters of 8 and of
16), 16 and 17 (one row per CTA, then two for the first), 24 and 25 (the
largest order of the cluster, the smallest of the general kernel), with full
and ragged last tiles.  The solve is backward stable: |b - A x| is at most
8 sqrt(n) u of |A| |x|, u = 2^-24 (the bound of the factorisation's tests), and
the same bits come back from every launch, whichever CTA is first.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402


@pytest.mark.parametrize("n", [65, 128, 449, 512, 513, 1024, 1025, 1536, 1537])
def test_float32_solve_at_cluster_edges(n):
    rng = np.random.default_rng(n)
    M = rng.standard_normal((n, n))
    Ad = torch.as_tensor(M @ M.T / n + 0.05 * np.eye(n)).to("cuda", torch.float32).contiguous()
    A = Ad.double().cpu().numpy()
    b = torch.as_tensor(rng.standard_normal(n)).cuda()
    ws = sc.cholesky_workspace(n, sc.SC_MIXED)
    first = None
    for _ in range(20):
        x = sc.cholesky_solve(Ad.clone(), b, sc.SC_MIXED, ws)[1].cpu().numpy()
        assert sc.device_status(ws) == 0
        first = x if first is None else first
        assert np.array_equal(x, first)
    res = np.abs(b.cpu().numpy() - A @ first) / (np.abs(A) @ np.abs(first))
    assert res.max() <= 8.0 * np.sqrt(n) * 2.0 ** -24, res.max()
