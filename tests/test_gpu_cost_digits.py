"""The cost of a float32 residual is summed with no fewer digits than float64
additions keep.

Zero coherencies leave V as the residual, and one component per visibility
with 12 significant bits has a square that float32 holds, so the values that the
block sums are known exactly.  130816 of them (512 stations, one timeslot), in
rows of 1024: the first row large, the others 2^-22 to 2^-26 of it
and odd, which a sum of two float32 words loses.  Bound: a thread's sum is
rounded twice to float64, its block adds ten times and the blocks' sums take at
most seven additions more, all values are positive: 19 x 2^-53 relative, and one
more for the words below."""
from fractions import Fraction

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402


@pytest.mark.parametrize("small", [2.0 ** -11, 2.0 ** -12, 2.0 ** -13])
def test_cost_keeps_float64_digits(small):
    N = 512
    B = N * (N - 1) // 2
    rows = [4095.0] + [((4095 - 2 * k) if k % 2 else (4093 - 6 * k)) * small for k in range(1, 128)]
    v = torch.tensor(rows, dtype=torch.float32).repeat_interleave(1024)[:B]
    exact = sum(Fraction(float(r)) ** 2 * min(1024, B - 1024 * i) for i, r in enumerate(rows))
    assert all(float(torch.tensor(r) ** 2) == r * r for r in rows)
    V = torch.zeros((1, B, 1, 2, 2), dtype=torch.complex64)
    V[0, :, 0, 0, 1] = v
    shp = sc.Shape(N, 1, 1, 1, 1)
    C = torch.zeros((1, B, 1), dtype=torch.complex64, device="cuda")
    J = torch.eye(2, dtype=torch.complex128, device="cuda").repeat(N, 1, 1).contiguous()
    R, cost = sc.residual(shp, V.cuda(), C, J, sc.SC_MIXED, sc.workspace(shp, sc.SC_MIXED))
    assert torch.equal(R.cpu(), V)
    assert abs(Fraction(cost.item()) - exact) <= 20 * Fraction(2) ** -53 * exact


@pytest.mark.parametrize("N,T,prec", [(2, 1, "mixed"), (256, 1, "mixed"), (257, 1, "mixed"), (300, 3, "mixed"),
                                      (900, 2, "mixed"), (257, 1, "fp64")])
def test_cost_of_ones_counts_them(N, T, prec):
    """One block up to 32768 values (256 stations), segments of 8192 above."""
    prec, cdt = (sc.SC_MIXED, torch.complex64) if prec == "mixed" else (sc.SC_FP64, torch.complex128)
    B = N * (N - 1) // 2
    V = torch.zeros((T, B, 1, 2, 2), dtype=cdt, device="cuda")
    V[..., 1, 1] = 1j
    shp = sc.Shape(N, T, 1, 1, 1)
    J = torch.eye(2, dtype=torch.complex128, device="cuda").repeat(N, 1, 1).contiguous()
    ws = sc.workspace(shp, prec)
    for _ in range(2):  # the sums replace values of the first call
        _, cost = sc.residual(shp, V, torch.zeros((T, B, 1), dtype=cdt, device="cuda"), J, prec, ws)
        assert cost.item() == T * B
