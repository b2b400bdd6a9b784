"""The float64 factorisation and solve (16x16 tiles, 32-row solve blocks) at the
orders where they can go wrong: one tile and less, the edges of the 16-, 32-
and 64-wide tiles, the first orders with tasks of either kind, several block
counts; alone through sc_cholesky_solve.  (A batch gives the same bits as a
job alone: test_gpu_batch.py.)

Bounds: |A - L L^T|_ij <= 8 sqrt(n) u sqrt(A_ii A_jj) and |b - A x| <= 8
sqrt(n) u (|A| |x|), u = 2^-53, the backward errors of the method (Higham,
Accuracy and Stability of Numerical Algorithms, Thms. 10.3, 10.4) with the
sqrt(n) growth of random rounding, as in test_gpu_cholesky.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402

U = 2.0 ** -53


@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 48, 64, 65, 80, 129, 193, 255, 330, 700])
def test_float64_factor_and_solve_at_tile_edges(n):
    rng = np.random.default_rng(n)
    M = rng.standard_normal((n, n))
    A = M @ M.T / n + 0.05 * np.eye(n)
    # rows and columns of very different size: the bound is per entry
    s = 10.0 ** rng.uniform(-3, 3, n)
    A = A * np.outer(s, s)
    b = rng.standard_normal(n) * s
    Ad = torch.as_tensor(A).cuda()
    ws = sc.cholesky_workspace(n, sc.SC_FP64)
    L, x = sc.cholesky_solve(Ad.clone(), torch.as_tensor(b).cuda(), sc.SC_FP64, ws)
    assert sc.device_status(ws) == 0
    L, x = np.tril(L.cpu().numpy()), x.cpu().numpy()
    assert np.all(np.diag(L) > 0)
    d = np.sqrt(np.diag(A))
    assert (np.abs(L @ L.T - A) / np.outer(d, d)).max() <= 8 * np.sqrt(n) * U
    assert (np.abs(b - A @ x) / (np.abs(A) @ np.abs(x))).max() <= 8 * np.sqrt(n) * U


@pytest.mark.parametrize("n,bad", [(16, 0), (40, 17), (200, 199)])
def test_float64_negative_pivot_is_reported(n, bad):
    A = np.eye(n) * 2.0
    A[bad, bad] = -1.0
    ws = sc.cholesky_workspace(n, sc.SC_FP64)
    sc.cholesky_solve(torch.as_tensor(A).cuda(), None, sc.SC_FP64, ws)
    assert sc.device_status(ws) == sc.SC_STATUS_NOTPD
