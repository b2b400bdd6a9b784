"""Every split of the complex64 residual pass into items, against the float64
arithmetic of the same rounded inputs.

An item is up to five timeslots, or up to four timeslots x channels, of a
baseline; (T, F) below reach each item size, uneven last slabs of timeslots,
uneven last groups of channels and both at once, and K the ring's four stages
and more.  Tolerance: each residual sums K + 1 float32 terms c G bounded by
s = max|V| + sum_k max|c_k| max|J_k|^2, so (K + 8) 2^-23 s, without a
correction; the cost sums squares of residuals each off by that much.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc, synth  # noqa: E402


@pytest.mark.parametrize("T,F,K", [(1, 1, 4), (2, 1, 5), (3, 1, 4), (4, 1, 4), (5, 1, 9), (6, 1, 4), (11, 1, 4),
                                   (3, 2, 4), (1, 5, 4), (1, 7, 8), (2, 3, 4), (3, 3, 4), (10, 4, 6), (7, 5, 4)])
def test_every_item_split(T, F, K):
    N = 23
    rng = np.random.default_rng(100 * T + 10 * F + K)
    cplx = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    p, q = synth.baseline_pairs(N)
    V = cplx(T, len(p), F, 2, 2).astype(np.complex64)
    C = cplx(K, T, len(p), F).astype(np.complex64)
    J = cplx(K, N, 2, 2)
    J = J.astype(np.complex64).astype(np.complex128)
    ref = V.astype(np.complex128)
    for k in range(K):
        G = J[k, p] @ J[k, q].conj().transpose(0, 2, 1)
        ref = ref - C[k].astype(np.complex128)[..., None, None] * G[None, :, None]
    shp = sc.Shape(N, T, F, K, 1)
    ws = sc.workspace(shp, sc.SC_MIXED)
    dev = lambda a: torch.as_tensor(a).cuda()
    out, cost = sc.residual_all(shp, dev(V), dev(C), dev(J), sc.SC_MIXED, ws, corr=-1)
    s = np.abs(V).max() + sum(np.abs(C[k]).max() * np.linalg.norm(J[k], axis=(1, 2)).max() ** 2 for k in range(K))
    tol = (K + 8) * 2.0 ** -23 * s
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= tol
    want, e = np.sum(np.abs(ref) ** 2), tol * np.sqrt(ref.size)
    assert abs(cost.item() - want) <= 2 * np.sqrt(want) * e + e * e
    assert sc.device_status(ws) == 0
