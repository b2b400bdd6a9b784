"""The float64 factorisation at both ends of the float64 range: pivots whose
reciprocal is subnormal (2^1022 and above), subnormal pivots whose reciprocal
is finite (0.75 x 2^-1022) and subnormal pivots whose reciprocal is not
(2^-1030).

A is B times a power of two s, B near a multiple of the identity, so that L /
sqrt(s) and x are those of B.  Bounds, in units of s: the method's, 8 sqrt(n) u
sqrt(B_ii B_jj) and 8 sqrt(n) u |B| |x| (u = 2^-53, as in
test_gpu_cholesky_f64.py), and where numbers of A's size are subnormal one
quantum q = 2^-1074 / s for every rounding of an entry: at most 2 n + 32 in
the factor (16 steps in its tile, 17 terms for each of n / 16 panels), 4 n + 64
with the right-hand side's, each of which moves the residual by at most
q (1 + sum |x|)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402

U = 2.0 ** -53


@pytest.mark.parametrize("diag,e", [(1.5, 1022), (0.75, -1022), (1.5, -1030)])
@pytest.mark.parametrize("n", [1, 2, 20, 70])
def test_float64_factor_at_the_ends_of_the_range(n, diag, e):
    q = 2.0 ** (-1074 - e) if e < 0 else 0.0
    unit = max(q, 2.0 ** -50)
    rng = np.random.default_rng(n)
    M = rng.uniform(-1, 1, (n, n))
    B = np.round((0.25 / n * (M + M.T)) / unit) * unit  # exact in float64 times 2^e
    np.fill_diagonal(B, diag)
    b = np.round(rng.uniform(-0.5, 0.5, n) / unit) * unit
    A, rhs = np.ldexp(B, e), np.ldexp(b, e)
    assert np.array_equal(np.ldexp(A, -e), B) and np.array_equal(np.ldexp(rhs, -e), b)
    ws = sc.cholesky_workspace(n, sc.SC_FP64)
    L, x = sc.cholesky_solve(torch.as_tensor(A).cuda(), torch.as_tensor(rhs).cuda(), sc.SC_FP64, ws)
    assert sc.device_status(ws) == 0
    L, x = np.ldexp(np.tril(L.cpu().numpy()), -e // 2), x.cpu().numpy()
    assert np.abs(L @ L.T - B).max() <= 8 * np.sqrt(n) * U * diag + (2 * n + 32) * q
    bound = 8 * np.sqrt(n) * U * (np.abs(B) @ np.abs(x)) + (4 * n + 64) * q * (1 + np.abs(x).sum())
    assert np.all(np.abs(b - B @ x) <= bound)
